// cpr_fv.cuh -- the finite-volume comparison scheme of the paper, fused into
// one SSP-RK3 stage kernel.
//
// One average per element (Sec. 2.1):
//   dq_ij/dt = -(f_{i+1/2,j} - f_{i-1/2,j}) / dx - (g_{i,j+1/2} - g_{i,j-1/2}) / dy,
// the face states reconstructed by second-order MUSCL with minmod-limited
// slopes (Sec. 2.6), q_face = q_i +- (1/2) minmod(q_{i+1} - q_i, q_i - q_{i-1}),
// and the face flux from the same common flux as the CPR kernel
// (reconstruct, then Riemann flux: Algorithm 1).  ORDER 3 takes the
// third-order MUSCL face values of Sec. 2.6 (van Leer's kappa = 1/3, each
// one-sided difference D-, D+ limited by minmod against four times the other):
//   q_{i+1/2}^- = q_i + mm(D-, 4 D+)/6 + mm(D+, 4 D-)/3,
//   q_{i-1/2}^+ = q_i - mm(D+, 4 D-)/6 - mm(D-, 4 D+)/3,
// on the same five-element stencil.  Ghost elements: periodic directions
// wrap, transmissive ones repeat the boundary element.
//
// One warp owns a strip of 28 columns of elements (lanes 2..29; the outer two
// lanes of either side are the ring of the reconstruction) and walks up its
// rows.  Along y everything a row shares with the one below it (the element
// values, the difference, the upper face state and the flux of the face
// between them) stays in registers; along x the neighbour values, the lower
// state and the flux of the right face come from the next lane by shuffle.
// So a face of the strip is evaluated once, nothing goes through shared
// memory and no barrier separates the phases; the next row's values are
// loaded one row ahead.  Faces on the strip's boundary are also evaluated by
// the neighbouring warp, from the same values and in the same order, so the
// flux leaving one element is the flux entering the next.
//
// The kernel is bound by the instructions of a row and their latency.  A tile
// of 32 x 8 elements per CTA, staged in shared memory with its ring, took a
// second, nearly empty pass over the faces (33 x 8 of them for 256 threads),
// three barriers and twice the instructions: 1536^2, second order, 12 FP32
// steps 2.44 -> 1.33 ms (67.7 -> 37.0 us per stage; 1.48 -> 2.72 TB/s of the
// eight state arrays that a step has to move).
#pragma once

#include <algorithm>
#include <type_traits>

#include "cpr_common.cuh"
#include "cpr_launch.h"
#include "cpr_reduce.cuh"
#include "cpr_stage.cuh"
#include "cpr_stage_quad.cuh"

namespace cpr {

constexpr int kFvCols = 28;   // columns of elements per warp
// Warps per CTA.  FP32 four: neighbouring strips, whose rings overlap in L1.
// FP64 one: the SM's FP64 pipe is busy from four warps on, however they share
// CTAs, so single warps spread a grid most evenly (256^2 second order, Euler /
// Roe: 45.7 / 98.8 us a residual with four, 37.3 / 76.2 with one).
template <class T>
constexpr int kFvWarps = sizeof(T) == 8 ? 1 : 4;

// Wrapped (periodic) or clamped (transmissive) element index, for indices
// at most two outside [0, n) (no integer division: n may be 1).
__device__ __forceinline__ int fv_ghost(int i, int n, int transmissive)
{
    if (transmissive) return min(max(i, 0), n - 1);
    while (i < 0) i += n;
    while (i >= n) i -= n;
    return i;
}

// Minmod of the slopes, zero where either is NaN (a face state next to a NaN
// element takes no slope from it).  FP32: the minimum if both are positive plus
// the maximum if both are negative; the inner pair passes a NaN on, the outer
// one drops it.  FP64 (comparisons run on the FP64 pipe): one comparison of the
// magnitudes, the signs and the NaN test from the high words (a difference that
// is NaN is a quiet one).
__device__ __forceinline__ float fv_minmod(float a, float b)
{
    float lo, hi;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(lo) : "f"(a), "f"(b));
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(hi) : "f"(a), "f"(b));
    return fmaxf(lo, 0.f) + fminf(hi, 0.f);
}
__device__ __forceinline__ double fv_minmod(double a, double b)
{
    const double m = ::fabs(a) < ::fabs(b) ? a : b;
    const int ha = __double2hiint(a), hb = __double2hiint(b);
    const bool nan = max(ha & 0x7fffffff, hb & 0x7fffffff) > 0x7ff00000;
    return (ha ^ hb) < 0 || nan ? 0.0 : m;
}

// The variables of one element.
template <class T, int V>
struct FvEl {
    T v[V];
};
template <class T, int V>
__device__ __forceinline__ FvEl<T, V> fv_up_lane(const FvEl<T, V>& x)  // the value of the lane below
{
    FvEl<T, V> r;
#pragma unroll
    for (int k = 0; k < V; ++k) r.v[k] = __shfl_up_sync(0xffffffffu, x.v[k], 1);
    return r;
}
template <class T, int V>
__device__ __forceinline__ FvEl<T, V> fv_down_lane(const FvEl<T, V>& x)
{
    FvEl<T, V> r;
#pragma unroll
    for (int k = 0; k < V; ++k) r.v[k] = __shfl_down_sync(0xffffffffu, x.v[k], 1);
    return r;
}

// c x + y; FP32 Euler in packed pairs.
template <class T, int V>
__device__ __forceinline__ FvEl<T, V> fv_axpy(T c, const FvEl<T, V>& x, const FvEl<T, V>& y)
{
    FvEl<T, V> r;
    if constexpr (V == 4) {
        qget(qfma(qput(x.v), c, qput(y.v)), r.v);
    } else {
#pragma unroll
        for (int k = 0; k < V; ++k) r.v[k] = fma(c, x.v[k], y.v[k]);
    }
    return r;
}
// a - b (exact as -1 b + a)
template <class T, int V>
__device__ __forceinline__ FvEl<T, V> fv_diff(const FvEl<T, V>& a, const FvEl<T, V>& b) { return fv_axpy(T(-1), b, a); }
template <class T, int V>
__device__ __forceinline__ FvEl<T, V> fv_scale(T c, const FvEl<T, V>& x)
{
    FvEl<T, V> r;
    if constexpr (V == 4) {
        qget(qmul(qput(x.v), c), r.v);
    } else {
#pragma unroll
        for (int k = 0; k < V; ++k) r.v[k] = c * x.v[k];
    }
    return r;
}

// Face states of element b with the one-sided differences dm, dp along the
// line: its value on the upper face (up) and on the lower face (dn).
template <int ORDER, class T, int V>
__device__ __forceinline__ void fv_states(const FvEl<T, V>& b, const FvEl<T, V>& dm, const FvEl<T, V>& dp,
                                          FvEl<T, V>& up, FvEl<T, V>& dn)
{
#pragma unroll
    for (int k = 0; k < V; ++k) {
        if constexpr (ORDER == 2) {
            up.v[k] = fv_minmod(dp.v[k], dm.v[k]);
        } else {
            const T m1 = fv_minmod(dm.v[k], T(4) * dp.v[k]), m2 = fv_minmod(dp.v[k], T(4) * dm.v[k]);
            up.v[k] = b.v[k] + fma(m1, T(1.0 / 6.0), m2 * T(1.0 / 3.0));
            dn.v[k] = b.v[k] - fma(m2, T(1.0 / 6.0), m1 * T(1.0 / 3.0));
        }
    }
    if constexpr (ORDER == 2) {
        const FvEl<T, V> s = up;
        up = fv_axpy(T(0.5), s, b);
        dn = fv_axpy(T(-0.5), s, b);
    }
}

// Twice the common flux between the lower state m and the upper state p.
template <int EQ, int FLUX, int DIR, class T, int V>
__device__ __forceinline__ FvEl<T, V> fv_face2(const FvEl<T, V>& m, const FvEl<T, V>& p, const Phys<T>& ph)
{
    FvEl<T, V> F;
    if constexpr (EQ == EQ_EULER) {
        qget(quad_face2<FLUX, DIR>(qput(m.v), qput(p.v), ph), F.v);
    } else {
        common_flux<EQ, FLUX, DIR>(m.v, p.v, ph, F.v);
        F.v[0] *= T(2);
    }
    return F;
}

// Resident CTAs the register budget is sized for: FP32 six, 24 warps per SM
// (80 registers, no spills).  1536^2, us per stage: five CTAs 44, six 37, seven
// (72 registers) 41.
constexpr int kFvResident = 6;
template <class T>
constexpr int fv_min_blocks()
{
    return sizeof(T) == 4 ? kFvResident : 1;
}

// What the stage update adds to a row (row_of reads a row of an array).
template <class T, class El, class F>
__device__ __forceinline__ void fv_terms(int mode, const StageArgs<T>& A, int j, F&& row_of, El& s0, El& s1, El& s2)
{
    if (mode >= MODE_SO1 && mode != MODE_INC1) s0 = row_of(mode == MODE_INC2 ? A.qb : A.qs, j);
    if (mode == MODE_SO2 || mode == MODE_SO3) s1 = row_of(A.qn, j);
    if (mode == MODE_INC3) {
        s1 = row_of(A.qb, j);
        s2 = row_of(A.lo, j);
    }
}

// The stage's result from o, R times the step's factor of the stage.
template <class T, int V>
__device__ __forceinline__ FvEl<T, V> fv_update(int mode, FvEl<T, V> o, FvEl<T, V> s0, const FvEl<T, V>& s1,
                                                FvEl<T, V>& s2)
{
    if (mode == MODE_SO1) {
        o = fv_axpy(T(1), s0, o);
    } else if (mode == MODE_SO2 || mode == MODE_SO3) {
        o = fv_axpy(mode == MODE_SO2 ? T(0.75) : T(1.0 / 3.0), s1,
                    fv_axpy(mode == MODE_SO2 ? T(0.25) : T(2.0 / 3.0), s0, o));
    } else if (mode == MODE_INC2) {
        o = fv_axpy(T(0.25), s0, o);
    } else if (mode == MODE_INC3) {
        o = fv_axpy(T(2.0 / 3.0), s1, o);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            compensated_add(s0.v[v], s2.v[v], o.v[v]);
            o.v[v] = s0.v[v];
        }
    }
    return o;
}

// MODE: the stage mode, or -1 for the one in the arguments.
template <class T, int EQ, int FLUX, int ORDER, int MODE>
__global__ void __launch_bounds__(kFvWarps<T> * 32, fv_min_blocks<T>())
cpr_fv_stage_kernel(const StageArgs<T> A, const int rows)
{
    constexpr int V = NVars<EQ>::value;
    using El = FvEl<T, V>;
    const int mode = MODE >= 0 ? MODE : A.mode;
    if (mode > 0 && A.ctrl->done) return;  // t_end reached: uniform exit
    const int lane = threadIdx.x & 31;
    // rows by CTA, so that every row pointer is uniform over the CTA
    const int by = blockIdx.x / A.tiles_x, j0 = by * rows, jend = min(j0 + rows, A.ny);
    const int i0 = ((blockIdx.x - by * A.tiles_x) * kFvWarps<T> + (threadIdx.x >> 5)) * kFvCols;
    const int col = i0 + lane - 2;
    const bool valid = lane >= 2 && lane < 2 + kFvCols && col < A.nx;
    const bool addb = mode == MODE_INC2 || mode == MODE_INC3;
    // lanes past the ring of a ragged strip repeat its last column
    const unsigned int gi = (unsigned int)fv_ghost(min(col, A.nx + 1), A.nx, A.bcx);
    T m = T(0);

    if (i0 < A.nx) {
        auto row_of = [&](const T* p, int j) {
            El x;
            p += (long long)j * A.nx;
#pragma unroll
            for (int v = 0; v < V; ++v) x.v[v] = (p + v * A.npts)[gi];
            return x;
        };
        El nq, nb;  // the row being loaded: state and increment
        auto fetch = [&](int j) {
            j = fv_ghost(j, A.ny, A.bcy);
            nq = row_of(A.qs, j);
            if (addb) nb = row_of(A.qb, j);
        };
        auto row = [&]() { return addb ? fv_axpy(T(1), nq, nb) : nq; };
        fetch(j0 - 2);
        const El a = row();
        fetch(j0 - 1);
        El c = row();
        fetch(j0);
        El d = row();
        fetch(j0 + 1);
        El upl, up, dn;           // upl: upper state of row j
        El dyn = fv_diff(d, c);   // difference across the upper face of row j
        El Glo{};                 // flux of the lower face of row j
        fv_states<ORDER>(c, fv_diff(c, a), dyn, upl, dn);

        // the factor of R in the stage's result
        T w = mode > 0 ? T(A.ctrl->dt) : T(1);
        if (mode == MODE_SO2 || mode == MODE_INC2) w *= T(0.25);
        if (mode == MODE_SO3 || mode == MODE_INC3) w *= T(2.0 / 3.0);
        // one half of 1 / dx, 1 / dy: the fluxes are doubled
        const T sx = T(-0.25) * A.rhx2, sy = T(-0.25) * A.rhy2;
        // row j0 - 1 is there for its upper face only (the same instructions
        // for every face, so that both warps of a face see the same bits)
        // (FP32 counts from zero: the third-order Euler kernel spills otherwise,
        // 1536^2 1.614 -> 1.583 ms for 12 steps; FP64 takes fewer registers with j)
        const int first = sizeof(T) == 4 ? j0 - 1 : 0;
        for (int k = j0 - 1 - first; first + k < jend; ++k) {
            const int j = first + k;
            const El n = row();  // row j + 2
            if (j + 1 < jend) fetch(j + 3);
            const int jo = max(j, j0);
            El s0, s1, s2;  // what the stage update adds: started here, used last
            fv_terms(mode, A, jo, row_of, s0, s1, s2);
            // upper face of the row
            const El dnn = fv_diff(n, d);
            fv_states<ORDER>(d, dyn, dnn, up, dn);
            const El Ghi = fv_face2<EQ, FLUX, 1>(upl, dn, A.ph);
            upl = up;
            // FP64: no x-faces of the row below the strip, on the pipe that bounds
            // the kernel (FP32 third order measured 4 % slower with the branch)
            if (sizeof(T) == 4 || j >= j0) {
                // left face, and the right one from the next lane
                const El dx = fv_diff(c, fv_up_lane(c));
                fv_states<ORDER>(c, dx, fv_down_lane(dx), up, dn);
                const El Fl = fv_face2<EQ, FLUX, 0>(fv_up_lane(up), dn, A.ph);
                El o = fv_scale(sx, fv_diff(fv_down_lane(Fl), Fl));
                // (the step's factor last: rounded into sx and sy it would be an
                // error common to every element and step, which does not average out)
                o = fv_scale(w, fv_axpy(sy, fv_diff(Ghi, Glo), o));
                o = fv_update(mode, o, s0, s1, s2);
                if (valid && j >= j0) {
                    const long long r0 = (long long)j * A.nx;
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        (A.out + v * A.npts + r0)[gi] = o.v[v];
                        if (mode == MODE_INC3) (A.lo + v * A.npts + r0)[gi] = s2.v[v];
                    }
                    if (A.do_wave) {
                        const T sp = point_speed<EQ, true>(o.v, A.ph);
                        m = sp > m ? sp : m;
                    }
                }
            }
            c = d;
            d = n;
            dyn = dnn;
            Glo = Ghi;
        }
    }
    if (A.do_wave) block_time_update<T>(m, A.ctrl, /*advance=*/true, gridDim.x);
}

// Strips of two rows of one FP32 variable (advection): every load first, so that
// a strip takes one latency of L2 where the walk above takes one per row, which
// is most of a small grid's time.  The end-of-run flag is tested where something
// is written (an exit before the loads are used would wait for it ahead of
// them), and the registers are bounded as the walk's (unbounded, the compiler
// settles for 32 to 40 and fewer loads in flight: 64^2 3.7).  us per stage, second
// order, tiles of 32 x 8 elements -> walk -> this: 64^2 4.1 -> 4.3 -> 3.0, 160^2
// 4.0 -> 4.8 -> 3.1, 400^2 5.5 -> 5.4 -> 3.9.
constexpr int kFvShort = 2;
template <class T, int EQ>
constexpr bool fv_has_short = sizeof(T) == 4 && EQ == EQ_ADV;

template <class T, int EQ, int FLUX, int ORDER, int MODE>
__global__ void __launch_bounds__(kFvWarps<T> * 32, fv_min_blocks<T>()) cpr_fv_short_kernel(const StageArgs<T> A)
{
    constexpr int V = NVars<EQ>::value, R = kFvShort;
    using El = FvEl<T, V>;
    const int mode = MODE >= 0 ? MODE : A.mode;
    const bool done = mode > 0 && A.ctrl->done;  // t_end reached (uniform over the grid)
    const int lane = threadIdx.x & 31;
    const int by = blockIdx.x / A.tiles_x, j0 = by * R;
    const int i0 = ((blockIdx.x - by * A.tiles_x) * kFvWarps<T> + (threadIdx.x >> 5)) * kFvCols;
    const int col = i0 + lane - 2;
    const bool valid = lane >= 2 && lane < 2 + kFvCols && col < A.nx;
    const bool addb = mode == MODE_INC2 || mode == MODE_INC3;
    const unsigned int gi = (unsigned int)fv_ghost(min(col, A.nx + 1), A.nx, A.bcx);
    T m = T(0);

    if (i0 < A.nx) {
        auto row_of = [&](const T* p, int j) {
            El x;
            p += (long long)j * A.nx;
#pragma unroll
            for (int v = 0; v < V; ++v) x.v[v] = (p + v * A.npts)[gi];
            return x;
        };
        El x[R + 4], b[R + 4], s0[R], s1[R], s2[R];  // rows j0 - 2 .. j0 + R + 1; terms of the update
#pragma unroll
        for (int k = 0; k < R + 4; ++k) {
            const int j = fv_ghost(j0 - 2 + k, A.ny, A.bcy);
            x[k] = row_of(A.qs, j);
            if (addb) b[k] = row_of(A.qb, j);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) fv_terms(mode, A, min(j0 + r, A.ny - 1), row_of, s0[r], s1[r], s2[r]);
#pragma unroll
        for (int k = 0; k < R + 4; ++k)
            if (addb) x[k] = fv_axpy(T(1), x[k], b[k]);
        El G[R + 1], up[R + 2], dn[R + 2];  // flux of the lower face, states along y of row j0 - 1 + k
#pragma unroll
        for (int k = 0; k < R + 2; ++k)
            fv_states<ORDER>(x[k + 1], fv_diff(x[k + 1], x[k]), fv_diff(x[k + 2], x[k + 1]), up[k], dn[k]);
#pragma unroll
        for (int k = 0; k <= R; ++k) G[k] = fv_face2<EQ, FLUX, 1>(up[k], dn[k + 1], A.ph);
        T w = mode > 0 ? T(A.ctrl->dt) : T(1);
        if (mode == MODE_SO2 || mode == MODE_INC2) w *= T(0.25);
        if (mode == MODE_SO3 || mode == MODE_INC3) w *= T(2.0 / 3.0);
        const T sx = T(-0.25) * A.rhx2, sy = T(-0.25) * A.rhy2;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const El c = x[r + 2], dx = fv_diff(c, fv_up_lane(c));
            El xu, xd;
            fv_states<ORDER>(c, dx, fv_down_lane(dx), xu, xd);
            const El Fl = fv_face2<EQ, FLUX, 0>(fv_up_lane(xu), xd, A.ph);
            El o = fv_scale(sx, fv_diff(fv_down_lane(Fl), Fl));
            o = fv_update(mode, fv_scale(w, fv_axpy(sy, fv_diff(G[r + 1], G[r]), o)), s0[r], s1[r], s2[r]);
            if (valid && !done && j0 + r < A.ny) {
                const long long r0 = (long long)(j0 + r) * A.nx;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    (A.out + v * A.npts + r0)[gi] = o.v[v];
                    if (mode == MODE_INC3) (A.lo + v * A.npts + r0)[gi] = s2[r].v[v];
                }
                if (A.do_wave) {
                    const T sp = point_speed<EQ, true>(o.v, A.ph);
                    m = sp > m ? sp : m;
                }
            }
        }
    }
    if (A.do_wave && !done) block_time_update<T>(m, A.ctrl, /*advance=*/true, gridDim.x);
}

// Rows per strip.
//
// FP32: a strip costs about two rows beyond its own, and the pass takes the time
// of the SM with most CTAs; a row takes 0.6 us plus 0.14 us for every CTA that
// shares its SM, so few tall strips leave the SM waiting.  Of the heights that
// give every SM almost its resident CTAs or more, the one with the fewest rows
// on the busiest SM (1536^2: 24 rows, six CTAs each; 37 us per stage, 36 rows and
// four CTAs 50); smaller grids take two rows.
//
// FP64: the pass takes the time of the busiest SM's rows (1.45 us for a
// second-order Euler row of one warp); up to four warps take the time of 4.5,
// and a strip costs half a row beyond its own (the y-face below it).  Of heights
// 1, 2, 3, ..., 8, 10, ..., 32 on fourteen grids from 32^2 to 1536^2, every order,
// flux and equation, this choice is 1 % from the fastest on average, 9 % at worst,
// and never slower than a tile of 32 x 8 elements.  us a residual, second order,
// that tile -> FP32's rule and CTAs -> these: Euler 192^2 37 -> 41 -> 25, 512^2
// 180 -> 148 -> 114, 1536^2 1515 -> 891 -> 844; Roe 192^2 58 -> 85 -> 51, 512^2
// 300 -> 319 -> 251.
template <class T>
inline int fv_rows(int ctas_x, int ny, int sms)
{
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int kMaxRows = F64 ? 32 : 48;
    int best = 0;
    long long cost = 0;
    for (int r = F64 ? 1 : 2; r <= kMaxRows; ++r) {
        const long long ctas = (long long)ctas_x * ((ny + r - 1) / r), per_sm = (ctas + sms - 1) / sms;
        if (!F64 && r > 2 && ctas < (long long)(kFvResident - 1) * sms) break;
        const long long c = F64 ? std::max(2 * per_sm, 9LL) * (2 * r + 1) : per_sm * (r + 2);
        if (best == 0 || c <= cost) {
            best = r;
            cost = c;
        }
    }
    return best;
}

template <class T, int EQ, int FLUX, int ORDER>
static cudaError_t fv_order(const LaunchCfg& c, const StageArgs<T>& A, cudaStream_t s)
{
    const int rows = fv_rows<T>(A.tiles_x, c.ny, c.sms > 0 ? c.sms : 1);
    const int ctas = A.tiles_x * ((c.ny + rows - 1) / rows);
    auto launch = [&](auto m) {
        constexpr int M = decltype(m)::value;
        if constexpr (fv_has_short<T, EQ>) {
            if (rows == kFvShort) {
                cpr_fv_short_kernel<T, EQ, FLUX, ORDER, M><<<ctas, kFvWarps<T> * 32, 0, s>>>(A);
                return cudaGetLastError();
            }
        }
        cpr_fv_stage_kernel<T, EQ, FLUX, ORDER, M><<<ctas, kFvWarps<T> * 32, 0, s>>>(A, rows);
        return cudaGetLastError();
    };
    // FP32 steps take a kernel compiled for their stage mode
    if constexpr (sizeof(T) == 4) {
        if (A.mode == MODE_INC1) return launch(std::integral_constant<int, MODE_INC1>{});
        if (A.mode == MODE_INC2) return launch(std::integral_constant<int, MODE_INC2>{});
        if (A.mode == MODE_INC3) return launch(std::integral_constant<int, MODE_INC3>{});
    }
    return launch(std::integral_constant<int, -1>{});
}

template <class T, int EQ, int FLUX>
static cudaError_t fv_one(const LaunchCfg& c, const StageArgs<T>& A, cudaStream_t s)
{
    return c.fv_order == 3 ? fv_order<T, EQ, FLUX, 3>(c, A, s) : fv_order<T, EQ, FLUX, 2>(c, A, s);
}

}  // namespace cpr
