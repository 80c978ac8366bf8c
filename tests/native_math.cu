// The reciprocals and square roots of the stage kernels over an array.
#include "cpr_common.cuh"

template <class T>
__global__ void eval(const T* x, T* r, T* s, T* r0, T* s0, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = cpr::frcp_ftz(x[i]);
    s[i] = cpr::fsqrt_ftz(x[i]);
    r0[i] = T(1) / x[i];
    s0[i] = sqrt(x[i]);
}

template <class T>
static int run(const void* x, void* r, void* s, void* r0, void* s0, int n)
{
    eval<T><<<(n + 255) / 256, 256>>>((const T*)x, (T*)r, (T*)s, (T*)r0, (T*)s0, n);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}

extern "C" int native_math_f32(const void* x, void* r, void* s, void* r0, void* s0, int n)
{
    return run<float>(x, r, s, r0, s0, n);
}
extern "C" int native_math_f64(const void* x, void* r, void* s, void* r0, void* s0, int n)
{
    return run<double>(x, r, s, r0, s0, n);
}
