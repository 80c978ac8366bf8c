// cpr_stage.cuh -- the CPR residual and SSP-RK3 stages: the scheme, the stage
// modes, what all stage kernels share, and the kernel of the stand-alone FP32
// Euler residual.
//
// A CTA owns a tile of TX x TY elements and computes, for every solution point
// of the tile, the CPR right-hand side of Sec. 2.2 (Eq. 16-17)
//   R_ab = -(2/hx) [ sum_l D_al f_lb + (F*_L,b - f_L,b) g_L'(xi_a) + (F*_R,b - f_R,b) g_R'(xi_a) ]
//          -(2/hy) [ sum_l D_bl g_al + (G*_B,a - g_B,a) g_L'(eta_b) + (G*_T,a - g_T,a) g_R'(eta_b) ]
// and then one stage of the three-stage SSP Runge-Kutta scheme of Sec. 4, in
// one pass over HBM.  Two forms of the stage update:
//   Shu-Osher (modes 1-3): q1 = q + dt R(q); q2 = 3/4 q + 1/4 (q1 + dt R(q1));
//     q' = 1/3 q + 2/3 (q2 + dt R(q2)) -- the stage states are stored.
//   increments (modes 4-6, FP32): the same scheme written as
//     B1 = dt R(q); B2 = (B1 + dt R(q + B1)) / 4; q' = q + 2/3 (B2 + dt R(q + B2)),
//     with q' accumulated in two floats (hi + lo, error-free transformation),
//     so that the O(1e-3) update of an O(1) state does not lose its low bits
//     every stage.  hi' goes to a second buffer (neighbour CTAs still read hi).
//
// Kernels: FP32 Euler stages cpr_stage_quad.cuh, FP64 Euler cpr_stage_f64.cuh,
// advection cpr_stage_adv.cuh.  The tile below runs the stand-alone FP32 Euler
// residual (mode 0); built with -DCPR_FP32_DELTA=1, in the delta form, every FP32
// Euler stage.
//
// Thread roles (N = p+1 points per direction, NT = TX*TY*N threads): thread
// (el, k) is the x-line "row k of element el" and the y-line "column k of
// element el".  Its row comes from HBM into registers; its column is read
// from the shared-memory copy of the tile.
//
// Delta form: every flux is evaluated as an exact algebraic difference
// f(q_ref + d) - f(q_ref) from the state q_ref at point (0, 0) of its element.
// The divergence and the edge terms only need flux differences (the rows of
// D sum to zero, the edge weights sum to one), so the rounding error of the
// O(1) flux values drops out.  The common flux on a face inside the tile is
// formed relative to the upper (right/top) element's reference and shifted by
// f(ref_upper) - f(ref_lower) for the lower element's jump; on the tile's
// right/top edge it is formed relative to the lower element's reference.
//
// Phases (one barrier after each of 1-3):
//   1 own row: into the tile copy, x-line (flux differences, d/dxi, edge
//     states and fluxes; the right edge values go to shared memory); halo
//     lines (the edge states of the neighbour elements facing the tile)
//     straight from L2
//   2 y-line of column k from the tile copy: d/deta, edge states and fluxes
//   3 d/deta into the dead tile copy; common flux on the element's left and
//     lower face points, one evaluation per face point, giving the jumps
//     F* - f of both elements; the tile's right / upper edge faces go to
//     dedicated threads (no divergent tail in every warp)
//   4 row k: x- and y-parts of R, stage update, store; optional fused element
//     averages (Algorithm 9) and max signal speed of the result.
#pragma once

#include "cpr_common.cuh"
#include "cpr_reduce.cuh"

namespace cpr {

// What only the quad forms (Euler) need: their tables and the division of a
// tile index by tiles_x (div_invariant).
template <class T>
struct QuadArgs {
    QuadTab<T> tab;
    unsigned int tx_magic;
    int tx_shift;
};

template <class T>
struct StageArgs {
    const T* qs;      // stage input state (increment modes: hi of q^n)
    const T* qb;      // increment modes 5, 6: B1 / B2, added to qs on load
    const T* qn;      // Shu-Osher modes 2, 3: q^n
    T* out;           // residual, stage state, increment, or hi of q^{n+1}
    T* lo;            // mode 6: low part of q^n, updated in place
    T* avg;           // element averages of out (do_avg)
    Ctrl* ctrl;       // time control (mode >= 1)
    long long npts;   // points per variable, ne * N * N
    int nx, ny;
    int bcx, bcy;     // 1: transmissive
    int tiles_x;
    int mode;
    int do_avg, do_wave;
    int pf_lo;        // mode 6 on states larger than L2: launch the instantiation that prefetches the low part
    T rhx2, rhy2;     // 2/hx, 2/hy (CPR advection: times the velocity)
    Phys<T> ph;
    Tab<T> tab;
    TabPr<T> tp;      // the tables in pairs over points (two-lane path)
    QuadArgs<T> qx;   // the quad forms' own arguments (Euler)
};

template <int N, int V, int TX, int TY, bool DELTA>
struct StageLayout {
    static constexpr int NN = N * N;
    // N = 4: rows of 16 bytes, element stride 16 words, row b of element el
    // stored at slot b ^ ((el >> 1) & 3).  A quarter warp's row accesses
    // (two elements) and a warp's column reads (eight elements, one word
    // each) then both hit distinct banks.  N = 3, 5: unpadded elements (the
    // row reads of a warp are conflict-free, column reads at most two-way);
    // N = 2: stride 6 (rows of 8 bytes stay aligned).
    static constexpr bool SWZ = N == 4;
    static constexpr int ES = SWZ ? 16 : (N == 2 ? 6 : NN);
    static constexpr int E = TX * TY;
    static constexpr int PE = (TX + 2) * (TY + 2);     // tile with its halo ring
    // The y-derivatives go over the dead tile copy in phase 3 (a buffer of
    // their own, written in phase 2, holds fewer registers across the
    // barrier but leaves too little of the SM's shared memory / L1 to L1).
    static constexpr int SQ = V * E * ES;              // tile copy, then the y-derivatives
    static constexpr int XR = V * TY * (TX + 1) * N;   // right edge states, elements -1..TX-1
    static constexpr int XH = V * TY * N;              // left edge states of the right halo
    static constexpr int XF = V * E * N;               // right edge fluxes, then the right jumps
    static constexpr int YT = V * (TY + 1) * TX * N;   // top edge states, elements -1..TY-1
    static constexpr int YH = V * TX * N;              // bottom edge states of the upper halo
    static constexpr int YF = V * E * N;               // top edge fluxes, then the top jumps
    static constexpr int JB = V * E * N;               // bottom jumps
    static constexpr int RF = DELTA ? V * PE : 0;      // element reference states
    static constexpr int TOTAL = SQ + XR + XH + XF + YT + YH + YF + JB + RF;
    // point (b, a) (row b, column a) of element el in a tile array
    __device__ static int sq(int v, int el, int b, int a)
    {
        return (v * E + el) * ES + (SWZ ? 4 * (b ^ ((el >> 1) & 3)) : b * N) + a;
    }
    __device__ static int xr(int v, int ty, int f, int k) { return ((v * TY + ty) * (TX + 1) + f) * N + k; }
    __device__ static int xh(int v, int ty, int k) { return (v * TY + ty) * N + k; }
    __device__ static int yt(int v, int g, int tx, int k) { return ((v * (TY + 1) + g) * TX + tx) * N + k; }
    __device__ static int yh(int v, int tx, int k) { return (v * TX + tx) * N + k; }
    // per-element line values (XF, YF, JB): line k of element el
    __device__ static int ef(int v, int el, int k) { return (v * E + el) * N + k; }
    // reference of the element at tile coordinates (lx, ly), -1 <= lx <= TX
    __device__ static int rf(int v, int lx, int ly) { return v * PE + (ly + 1) * (TX + 2) + (lx + 1); }
};

// Edge value of a line of N values: sum_l c_l x_l, in one fixed fma order so
// that every CTA computing the same edge state gets the same bits.
template <int N, class T>
__device__ __forceinline__ T line_dot(const T* c, const T* x)
{
    T s = c[0] * x[0];
#pragma unroll
    for (int l = 1; l < N; ++l) s = fma(c[l], x[l], s);
    return s;
}

template <int N, class T>
__device__ __forceinline__ void gload_row(const T* __restrict__ s, T* x)
{
    if constexpr (sizeof(T) == 4 && N == 4) {
        float4 t = *reinterpret_cast<const float4*>(s);
        x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else if constexpr (sizeof(T) == 4 && N == 2) {
        float2 t = *reinterpret_cast<const float2*>(s);
        x[0] = t.x; x[1] = t.y;
    } else if constexpr (sizeof(T) == 8 && N % 2 == 0) {
#pragma unroll
        for (int a = 0; a < N; a += 2) {
            double2 t = *reinterpret_cast<const double2*>(s + a);
            x[a] = t.x; x[a + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = s[a];
    }
}

template <int N, class T>
__device__ __forceinline__ void gstore_row(T* __restrict__ d, const T* x)
{
    if constexpr (sizeof(T) == 4 && N == 4) {
        *reinterpret_cast<float4*>(d) = make_float4(x[0], x[1], x[2], x[3]);
    } else if constexpr (sizeof(T) == 4 && N == 2) {
        *reinterpret_cast<float2*>(d) = make_float2(x[0], x[1]);
    } else if constexpr (sizeof(T) == 8 && N % 2 == 0) {
#pragma unroll
        for (int a = 0; a < N; a += 2) *reinterpret_cast<double2*>(d + a) = make_double2(x[a], x[a + 1]);
    } else {
#pragma unroll
        for (int a = 0; a < N; ++a) d[a] = x[a];
    }
}

// Row of N values of one variable in shared memory (16-byte aligned when N = 4).
template <int N, class T>
__device__ __forceinline__ void sm_store_row(T* d, const T* x)
{
    if constexpr (sizeof(T) == 4 && N == 4) {
        *reinterpret_cast<float4*>(d) = make_float4(x[0], x[1], x[2], x[3]);
    } else {
#pragma unroll
        for (int a = 0; a < N; ++a) d[a] = x[a];
    }
}

template <int N, class T>
__device__ __forceinline__ void sm_load_row(const T* s, T* x)
{
    if constexpr (sizeof(T) == 4 && N == 4) {
        float4 t = *reinterpret_cast<const float4*>(s);
        x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else {
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = s[a];
    }
}

// Flux difference f_DIR(ref + d) - f_DIR(ref) (delta form) or f_DIR(d) (plain).
template <int EQ, int DIR, bool DELTA, class T>
__device__ __forceinline__ void line_flux(const Ref<T>& r, const T* d, const Phys<T>& ph, T* out)
{
    if constexpr (DELTA) dflux<EQ, DIR>(r, d, ph, out);
    else if constexpr (DIR == 0) flux_x<EQ>(d, ph, out);
    else flux_y<EQ>(d, ph, out);
}

// Common flux through an x-face (DIR 0) or y-face (DIR 1) between the lower
// state dm and the upper state dp: relative to the reference in the delta
// form (F* - f(ref)), the flux itself otherwise.
template <int EQ, int FLUX, int DIR, bool DELTA, class T>
__device__ __forceinline__ void face_flux(const Ref<T>& r, const T* dm, const T* dp, const Phys<T>& ph, T* G)
{
    if constexpr (DELTA) common_flux_delta<EQ, FLUX, DIR>(r, dm, dp, ph, G);
    else common_flux<EQ, FLUX, DIR>(dm, dp, ph, G);
}

// The line operators of the two-lane path on one line of V variables.
// em/ep: edge states (l(-1), l(+1)) of q; gm/gp: the same of the flux f; r:
// the flux derivative at the N points.  Per variable the operations are
// those of pdot and of the derivative sum, in the same order, whichever the
// loop nesting: variable by variable (N < 5), or each table pair loaded once
// and applied to all variables (N = 5, where it measured faster; for N = 4
// it was 0.3-0.5 % slower).
template <int N, int NP, int V, class T>
__device__ __forceinline__ void pair_line_ops(const TabPr<T>& tp, const Pr<T> (&q)[NP][V], const Pr<T> (&f)[NP][V],
                                              T* em, T* ep, T* gm, T* gp, T (&r)[N][V])
{
    if constexpr (N < 5) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            Pr<T> cq[NP], cf[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                cq[j] = q[j][v];
                cf[j] = f[j][v];
            }
            em[v] = pdot<NP>(tp.lm2, cq);
            ep[v] = pdot<NP>(tp.lp2, cq);
            gm[v] = pdot<NP>(tp.lm2, cf);
            gp[v] = pdot<NP>(tp.lp2, cf);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                Pr<T> a = pmul(tp.D2[i][0], pbc(cf[0].v.x));
#pragma unroll
                for (int l = 1; l < N; ++l) a = pfma(tp.D2[i][l], pbc(l % 2 ? cf[l / 2].v.y : cf[l / 2].v.x), a);
                r[2 * i][v] = a.v.x;
                if (2 * i + 1 < N) r[2 * i + 1][v] = a.v.y;
            }
        }
    } else {
        // edge states of q, then of f: the pair sums of pdot, all variables
        Pr<T> sm[V], sp[V];
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
            const Pr<T>(&x)[NP][V] = pass == 0 ? q : f;
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const Pr<T> cm = tp.lm2[j], cp = tp.lp2[j];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    sm[v] = j == 0 ? pmul(cm, x[0][v]) : pfma(cm, x[j][v], sm[v]);
                    sp[v] = j == 0 ? pmul(cp, x[0][v]) : pfma(cp, x[j][v], sp[v]);
                }
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                (pass == 0 ? em : gm)[v] = sm[v].v.x + sm[v].v.y;
                (pass == 0 ? ep : gp)[v] = sp[v].v.x + sp[v].v.y;
            }
        }
        // derivative: sum_l D2[i][l] f_l, the same accumulation order as above
        Pr<T> acc[NP][V];
#pragma unroll
        for (int l = 0; l < N; ++l) {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const Pr<T> c = tp.D2[i][l];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const Pr<T> fl = pbc(l % 2 ? f[l / 2][v].v.y : f[l / 2][v].v.x);
                    acc[i][v] = l == 0 ? pmul(c, fl) : pfma(c, fl, acc[i][v]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                r[2 * i][v] = acc[i][v].v.x;
                if (2 * i + 1 < N) r[2 * i + 1][v] = acc[i][v].v.y;
            }
    }
}

// q' = hi + lo + D as hi' + lo' (Knuth's two-sum of hi and D, then the old
// and new low parts folded back); the pair keeps about 48 bits.
__device__ __forceinline__ void compensated_add(float& hi, float& lo, float D)
{
    const float s = __fadd_rn(hi, D);
    const float bv = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bv)), __fsub_rn(D, bv));
    const float e = __fadd_rn(err, lo);
    const float h2 = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(h2, s));
    hi = h2;
}
__device__ __forceinline__ void compensated_add(double& hi, double& lo, double D)
{
    hi += D + lo;
    lo = 0.0;
}

// FP32 fluxes in the delta form (1) or directly (0).
#ifndef CPR_FP32_DELTA
#define CPR_FP32_DELTA 0
#endif
template <class T>
constexpr bool stage_delta()
{
    return sizeof(T) == 4 && CPR_FP32_DELTA != 0;
}

// Resident CTAs per SM the register budget is sized for (FP32: as many as the
// shared memory allows; FP64, in the grouped batch kernels: as the registers
// allow).
#ifndef CPR_STAGE_MINB_FP32
#define CPR_STAGE_MINB_FP32 4
#endif
#ifndef CPR_STAGE_MINB_FP32_N3
#define CPR_STAGE_MINB_FP32_N3 6
#endif
#ifndef CPR_STAGE_MINB_FP32_N2
#define CPR_STAGE_MINB_FP32_N2 4
#endif
#ifndef CPR_STAGE_MINB_FP32_N5
#define CPR_STAGE_MINB_FP32_N5 3
#endif
// Launches of at most two CTAs per SM (grids that fit the device at once,
// e.g. 128 x 128 elements of p = 3 on 152 SMs) take an instantiation
// compiled for two resident CTAs: twice the registers let the compiler keep
// more loads in flight, which is what bounds a CTA when the SM holds only
// one or two of them.
#ifndef CPR_STAGE_MINB_WIDE
#define CPR_STAGE_MINB_WIDE 2
#endif
// The counts are for tiles of 64 elements; a smaller tile (ELEMS elements)
// takes proportionally more CTAs, so that the threads per SM and the
// registers per thread stay the same.
template <class T, int N, bool WIDE = false, int ELEMS = 64>
constexpr int stage_min_blocks()
{
    static_assert(64 % ELEMS == 0, "tiles of 64 elements or a divisor of it");
    return (64 / ELEMS) *
           (sizeof(T) == 8 ? 1
            : WIDE         ? CPR_STAGE_MINB_WIDE
                           : (N == 2 ? CPR_STAGE_MINB_FP32_N2
                                     : (N == 3 ? CPR_STAGE_MINB_FP32_N3
                                               : (N == 4 ? CPR_STAGE_MINB_FP32 : CPR_STAGE_MINB_FP32_N5))));
}

// Threads of a CTA: whole warps (the warp-level reductions use every lane).
constexpr int stage_threads(int n) { return (n + 31) / 32 * 32; }

}  // namespace cpr

#include "cpr_stage_adv.cuh"
#include "cpr_stage_f64.cuh"
#include "cpr_stage_quad.cuh"

namespace cpr {

// The FP32 Euler stage updates take the quad form (the stand-alone residual
// the one below).
template <class T, int EQ, bool DELTA>
constexpr bool stage_quad = sizeof(T) == 4 && EQ == EQ_EULER && !DELTA;

// Dynamic shared memory of a stage-update CTA.
template <class T, int P, int EQ, int TX, int TY, bool DELTA>
constexpr size_t stage_smem()
{
    if constexpr (EQ == EQ_ADV) return sizeof(T) * AdvLayout<P + 1, TX, TY>::TOTAL;
    else if constexpr (sizeof(T) == 8) return sizeof(Quad<double>) * F64Layout<P + 1, TX, TY>::TOTAL;
    else if constexpr (stage_quad<T, EQ, DELTA>) return sizeof(Quad<float>) * QuadLayout<P + 1, TX, TY>::TOTAL;
    else return sizeof(T) * StageLayout<P + 1, NVars<EQ>::value, TX, TY, DELTA>::TOTAL;
}

// Threads of a stage-update CTA.
template <class T, int P, int EQ, int TX, int TY>
constexpr int stage_block = sizeof(T) == 8 && EQ == EQ_EULER ? 2 * f64_role_threads(P, TX, TY) : TX * TY * (P + 1);

// One tile of the stage: the work of one CTA.  tile indexes the instance's
// TX x TY tiles (row-major); threads tid >= NT of a wider CTA only take part
// in the barriers.  nslots: the tiles of the instance that report a maximum
// speed (the last one to finish closes the step).
template <class T, int P, int EQ, int DIV, int FLUX, int TX, int TY, bool DELTA, bool PF = false>
__device__ __forceinline__ void stage_tile(const StageArgs<T>& A, const Tab<T>& tb, const TabPr<T>& tp, int tile,
                                           int tid, unsigned char* smem_raw, int nslots)
{
    constexpr int N = P + 1, NN = N * N, V = NVars<EQ>::value;
    constexpr int NT = TX * TY * N;
    // Two-lane path (pairs of points of a line; packed FP32 instructions):
    // LP divergence, fluxes evaluated directly; even N, and N = 5 (for N = 3
    // it measured 1 % faster on the batch and 1 % slower on the limited run).
    // An odd line's last pair repeats its last point (PH): the table pairs
    // carry zero for it, and its derivative and residual lanes are not stored.
    static_assert(EQ == EQ_EULER && sizeof(T) == 4, "FP64 and advection have tiles of their own");
    constexpr bool PAIRED = DIV == DIV_LP && !DELTA && (N % 2 == 0 || N == 5);
    constexpr int NP = (N + 1) / 2;
    auto PH = [](int i) { return i < N ? i : N - 1; };
    static_assert(TX * TY >= TX + TY, "every tile-edge face point needs a thread of its own");
    using L = StageLayout<N, V, TX, TY, DELTA>;
    T* sq = reinterpret_cast<T*>(smem_raw);
    T* ryS = sq;  // y-derivatives, over the dead tile copy
    T* xR = sq + L::SQ;
    T* xH = xR + L::XR;
    T* xF = xH + L::XH;
    T* yT = xF + L::XF;
    T* yH = yT + L::YT;
    T* yF = yH + L::YH;
    T* jB = yF + L::YF;
    T* rfS = jB + L::JB;
    T* avS = xR;         // row partial sums of the averages, reuses xR after phase 3

    if (A.mode > 0 && A.ctrl->done) return;  // t_end reached: uniform exit
    // a limited run: clear the marked-element count of the limiter pass
    // that follows this stage (stream order keeps it apart from the last one)
    if (A.mode > 0 && A.do_avg && tile == 0 && tid == 0) A.ctrl->marked = 0;

    const bool active = tid < NT;
    const int i0 = (tile % A.tiles_x) * TX;
    const int j0 = (tile / A.tiles_x) * TY;
    const int TXe = min(TX, A.nx - i0), TYe = min(TY, A.ny - j0);
    const int el = tid / N, k = tid % N;
    const int tx = el % TX, ty = el / TX;
    const bool valid = active && tx < TXe && ty < TYe;
    const long long e = (long long)(j0 + ty) * A.nx + (i0 + tx);
    const bool addb = A.mode == MODE_INC2 || A.mode == MODE_INC3;
    const bool lwall = A.bcx && i0 + tx == 0;

    // ---- phase 1: own row -> tile copy and x-line; halo lines --------------
    T rx[N][V];           // d/dxi of the flux differences along row k
    T eL[V], fL[V];       // own left edge state and flux
    Ref<T> rf;            // own reference (delta form)
    if (PF && valid && k == 0 && (tx & 1) == 0) {
        // the low part is first read in phase 4, from HBM when the state
        // does not fit in L2: start it towards L2 now, one prefetch per
        // 128-byte line (two elements' rows of one variable)
#pragma unroll
        for (int v = 0; v < V; ++v) asm volatile("prefetch.global.L2 [%0];" ::"l"(A.lo + v * A.npts + e * NN));
    }
    if (valid) {
        T d[N][V], q0[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const T* src = A.qs + v * A.npts + e * NN;
            const T* srb = A.qb + v * A.npts + e * NN;
            T row[N];
            gload_row<N>(src + k * N, row);
            if (addb) {
                T b[N];
                gload_row<N>(srb + k * N, b);
#pragma unroll
                for (int a = 0; a < N; ++a) row[a] += b[a];
            }
            sm_store_row<N>(sq + L::sq(v, el, k, 0), row);
            q0[v] = T(0);
            if (DELTA) {
                // point (0, 0) of the element, formed exactly as the halo
                // loaders form it
                q0[v] = k == 0 ? row[0] : (addb ? src[0] + srb[0] : src[0]);
                if (k == 0) rfS[L::rf(v, tx, ty)] = q0[v];
            }
#pragma unroll
            for (int a = 0; a < N; ++a) d[a][v] = DELTA ? row[a] - q0[v] : row[a];
        }
        if constexpr (DELTA) rf = make_ref<EQ>(q0, A.ph);
        T f[N][V], col[N], eR[V], fR[V];
        if constexpr (PAIRED) {
            Pr<T> qp[NP][V], fp[NP][V];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
#pragma unroll
                for (int v = 0; v < V; ++v) qp[j][v] = pmk(d[2 * j][v], d[PH(2 * j + 1)][v]);
                flux_pair<EQ, 0>(qp[j], A.ph, fp[j]);
            }
            pair_line_ops<N, NP, V>(tp, qp, fp, eL, eR, fL, fR, rx);
        } else {
#pragma unroll
        for (int a = 0; a < N; ++a) line_flux<EQ, 0, DELTA>(rf, d[a], A.ph, f[a]);
#pragma unroll
        for (int v = 0; v < V; ++v) {
#pragma unroll
            for (int l = 0; l < N; ++l) col[l] = d[l][v];
            eL[v] = line_dot<N>(tb.lm, col);
            eR[v] = line_dot<N>(tb.lp, col);
        }
        if constexpr (DIV == DIV_LP) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
#pragma unroll
                for (int l = 0; l < N; ++l) col[l] = f[l][v];
#pragma unroll
                for (int a = 0; a < N; ++a) rx[a][v] = line_dot<N>(tb.D[a], col);
                fL[v] = line_dot<N>(tb.lm, col);
                fR[v] = line_dot<N>(tb.lp, col);
            }
        } else {
#pragma unroll
            for (int a = 0; a < N; ++a) {
                T dq[V], qa[V];
#pragma unroll
                for (int v = 0; v < V; ++v) {
#pragma unroll
                    for (int l = 0; l < N; ++l) col[l] = d[l][v];
                    dq[v] = line_dot<N>(tb.D[a], col);
                    qa[v] = DELTA ? q0[v] + d[a][v] : d[a][v];
                }
                flux_jvp<EQ, 0>(qa, dq, A.ph, rx[a]);
            }
            line_flux<EQ, 0, DELTA>(rf, eL, A.ph, fL);
            line_flux<EQ, 0, DELTA>(rf, eR, A.ph, fR);
        }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            xR[L::xr(v, ty, tx + 1, k)] = eR[v];
            xF[L::ef(v, el, k)] = fR[v];
        }
    }
    {
        constexpr int NXH = 2 * TY * N, NYH = 2 * TX * N;
        // Halo line t for the variables v0, v0 + vstep, ... < V.  Every warp
        // takes part: with NT a multiple of the line count each thread keeps
        // one line (its index arithmetic done once) for NT / lines variables;
        // otherwise one (line, variable) per thread and pass.
        auto halo_line = [&](int t, int v0, int vstep) {
            const bool xdir = t < NXH;
            const int r0 = xdir ? t : t - NXH;
            const int side = xdir ? r0 / (TY * N) : r0 / (TX * N);
            const int r = xdir ? r0 % (TY * N) : r0 % (TX * N);
            const int pos = r / N, kk = r % N;  // pos: tile row (x) or tile column (y)
            if (pos >= (xdir ? TYe : TXe)) return;
            int gi, gj;
            if (xdir) {
                gi = side ? i0 + TXe : i0 - 1;
                gj = j0 + pos;
                if (gi < 0 || gi >= A.nx) {
                    if (A.bcx) return;
                    gi = gi < 0 ? gi + A.nx : gi - A.nx;
                }
            } else {
                gi = i0 + pos;
                gj = side ? j0 + TYe : j0 - 1;
                if (gj < 0 || gj >= A.ny) {
                    if (A.bcy) return;
                    gj = gj < 0 ? gj + A.ny : gj - A.ny;
                }
            }
            const long long eh = (long long)gj * A.nx + gi;
            const int lx = xdir ? (side ? TXe : -1) : pos;
            const int ly = xdir ? pos : (side ? TYe : -1);
            const T* coef = side ? tb.lm : tb.lp;  // the edge facing the tile
            for (int v = v0; v < V; v += vstep) {
                const T* src = A.qs + v * A.npts + eh * NN;
                const T* srb = addb ? A.qb + v * A.npts + eh * NN : src;
                T ref = T(0);
                if (DELTA) ref = addb ? src[0] + srb[0] : src[0];
                T line[N];
                if (xdir) {
                    gload_row<N>(src + kk * N, line);
                    if (addb) {
                        T b[N];
                        gload_row<N>(srb + kk * N, b);
#pragma unroll
                        for (int l = 0; l < N; ++l) line[l] += b[l];
                    }
                } else {
#pragma unroll
                    for (int l = 0; l < N; ++l) line[l] = addb ? src[l * N + kk] + srb[l * N + kk] : src[l * N + kk];
                }
#pragma unroll
                for (int l = 0; l < N; ++l) line[l] -= ref;
                T dv;
                if constexpr (PAIRED) {
                    Pr<T> lp2[NP];
#pragma unroll
                    for (int j = 0; j < NP; ++j) lp2[j] = pmk(line[2 * j], line[PH(2 * j + 1)]);
                    dv = pdot<NP>(side ? tp.lm2 : tp.lp2, lp2);
                } else {
                    dv = line_dot<N>(coef, line);
                }
                if (xdir) {
                    if (side) xH[L::xh(v, pos, kk)] = dv;
                    else xR[L::xr(v, pos, 0, kk)] = dv;
                } else {
                    if (side) yH[L::yh(v, pos, kk)] = dv;
                    else yT[L::yt(v, 0, pos, kk)] = dv;
                }
                if (DELTA && kk == 0) rfS[L::rf(v, lx, ly)] = ref;
            }
        };
        constexpr int LINES = NXH + NYH;
        if constexpr (NT % LINES == 0) {
            if (active) halo_line(tid % LINES, tid / LINES, NT / LINES);
        } else {
            for (int tv = tid; active && tv < V * LINES; tv += NT) halo_line(tv % LINES, tv / LINES, V);
        }
    }
    // Phase 2 reads only the rows of its own element from the tile copy.  For
    // even N the column identity is the row identity and a warp holds whole
    // elements (32 % N == 0), so the rows it reads were written by its own
    // warp: a warp barrier orders them.  Everything else phase 1 writes
    // (edge states, halo lines) is read after the next CTA barrier.
    if constexpr (N % 2 == 0 && 32 % N == 0 && !DELTA) __syncwarp();
    else __syncthreads();

    // ---- phase 2: y-line (column kc of element elc) --------------------------
    // Column identity of the thread.  Odd N: k-major (a warp holds one column
    // of 32 consecutive elements), so that the column accesses of the tile
    // copy (odd element stride) and of the y-derivatives meet no bank
    // conflict; the element-major identity would put two elements' columns
    // in one bank.  Even N: the row identity (the N = 4 swizzle makes both
    // access patterns conflict-free for it).
    constexpr bool KMAJ = (N % 2 == 1) && !DELTA;
    const int elc = KMAJ ? tid % (TX * TY) : el, kc = KMAJ ? tid / (TX * TY) : k;
    const int txc = elc % TX, tyc = elc / TX;
    const bool validc = active && txc < TXe && tyc < TYe;
    const bool bwallc = A.bcy && j0 + tyc == 0;
    T ry[N][V];           // d/deta of the flux differences along column kc
    T eB[V], gB[V];       // own bottom edge state and flux
    if (validc) {
        T d[N][V], g[N][V], col[N], eT[V], gT[V];
#pragma unroll
        for (int b = 0; b < N; ++b)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const T x = sq[L::sq(v, elc, b, kc)];
                d[b][v] = DELTA ? x - rf.q[v] : x;
            }
        if constexpr (PAIRED) {
            Pr<T> qp[NP][V], gp[NP][V];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
#pragma unroll
                for (int v = 0; v < V; ++v) qp[j][v] = pmk(d[2 * j][v], d[PH(2 * j + 1)][v]);
                flux_pair<EQ, 1>(qp[j], A.ph, gp[j]);
            }
            pair_line_ops<N, NP, V>(tp, qp, gp, eB, eT, gB, gT, ry);
        } else {
#pragma unroll
        for (int b = 0; b < N; ++b) line_flux<EQ, 1, DELTA>(rf, d[b], A.ph, g[b]);
#pragma unroll
        for (int v = 0; v < V; ++v) {
#pragma unroll
            for (int l = 0; l < N; ++l) col[l] = d[l][v];
            eB[v] = line_dot<N>(tb.lm, col);
            eT[v] = line_dot<N>(tb.lp, col);
        }
        if constexpr (DIV == DIV_LP) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
#pragma unroll
                for (int l = 0; l < N; ++l) col[l] = g[l][v];
#pragma unroll
                for (int b = 0; b < N; ++b) ry[b][v] = line_dot<N>(tb.D[b], col);
                gB[v] = line_dot<N>(tb.lm, col);
                gT[v] = line_dot<N>(tb.lp, col);
            }
        } else {
#pragma unroll
            for (int b = 0; b < N; ++b) {
                T dq[V], qb[V];
#pragma unroll
                for (int v = 0; v < V; ++v) {
#pragma unroll
                    for (int l = 0; l < N; ++l) col[l] = d[l][v];
                    dq[v] = line_dot<N>(tb.D[b], col);
                    qb[v] = DELTA ? rf.q[v] + d[b][v] : d[b][v];
                }
                flux_jvp<EQ, 1>(qb, dq, A.ph, ry[b]);
            }
            line_flux<EQ, 1, DELTA>(rf, eB, A.ph, gB);
            line_flux<EQ, 1, DELTA>(rf, eT, A.ph, gT);
        }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            yT[L::yt(v, tyc + 1, txc, kc)] = eT[v];
            yF[L::ef(v, elc, kc)] = gT[v];
        }
    }
    __syncthreads();

    // ---- phase 3: common fluxes and jumps ----------------------------------
    // Each element takes the face points of its left and lower faces (the
    // tile's right and upper edges go to dedicated threads), evaluates the
    // common flux once relative to its own reference, and forms the jumps
    // F* - f of both elements of the face: its own (kept) and the
    // neighbour's (over the neighbour's edge flux in shared memory, shifted to
    // the neighbour's reference).
    T JL[V];
    if (validc) {
#pragma unroll
        for (int b = 0; b < N; ++b)
#pragma unroll
            for (int v = 0; v < V; ++v) ryS[L::sq(v, elc, b, kc)] = ry[b][v];
    }
    // lower face of column kc of element elc (column identity); in the delta
    // form (row identity = column identity) relative to the element's
    // reference rf0 with state q0
    auto lower_face = [&](const Ref<T>& rf0, const T (&q0)[V]) {
        T o[V], dm[V], G[V], sh[V];
#pragma unroll
        for (int v = 0; v < V; ++v) o[v] = (DELTA && !bwallc) ? rfS[L::rf(v, txc, tyc - 1)] - q0[v] : T(0);
#pragma unroll
        for (int v = 0; v < V; ++v) dm[v] = bwallc ? eB[v] : yT[L::yt(v, tyc, txc, kc)] + o[v];
        face_flux<EQ, FLUX, 1, DELTA>(rf0, dm, eB, A.ph, G);
#pragma unroll
        for (int v = 0; v < V; ++v) jB[L::ef(v, elc, kc)] = G[v] - gB[v];
        if (tyc > 0) {
            if constexpr (DELTA) dflux<EQ, 1>(rf0, o, A.ph, sh);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                T* pj = yF + L::ef(v, elc - TX, kc);
                *pj = (DELTA ? G[v] - sh[v] : G[v]) - *pj;
            }
        }
    };
    if (valid) {
        T q0[V];
#pragma unroll
        for (int v = 0; v < V; ++v) q0[v] = DELTA ? rfS[L::rf(v, tx, ty)] : T(0);
        if constexpr (DELTA) rf = make_ref<EQ>(q0, A.ph);
        T o[V], dm[V], G[V], sh[V];
        // left face
#pragma unroll
        for (int v = 0; v < V; ++v) o[v] = (DELTA && !lwall) ? rfS[L::rf(v, tx - 1, ty)] - q0[v] : T(0);
#pragma unroll
        for (int v = 0; v < V; ++v) dm[v] = lwall ? eL[v] : xR[L::xr(v, ty, tx, k)] + o[v];
        face_flux<EQ, FLUX, 0, DELTA>(rf, dm, eL, A.ph, G);
#pragma unroll
        for (int v = 0; v < V; ++v) JL[v] = G[v] - fL[v];
        if (tx > 0) {
            // f(ref_own) - f(ref_left) = -(f(ref_own + (ref_left - ref_own)) - f(ref_own))
            if constexpr (DELTA) dflux<EQ, 0>(rf, o, A.ph, sh);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                T* pj = xF + L::ef(v, el - 1, k);
                *pj = (DELTA ? G[v] - sh[v] : G[v]) - *pj;
            }
        }
        if constexpr (!KMAJ) lower_face(rf, q0);
    }
    if constexpr (KMAJ) {
        if (validc) {
            const T q0[V] = {};
            lower_face(rf, q0);
        }
    }
    if (tid < (TX + TY) * N) {
        // right face of the tile's last column (x) / upper face of its last row
        const bool xe = tid < TY * N;
        const int r = xe ? tid : tid - TY * N;
        const int pos = r / N, kk = r % N;
        if (pos < (xe ? TYe : TXe)) {
            const int ex = xe ? TXe - 1 : pos, ey = xe ? pos : TYe - 1;
            const bool wall = xe ? (A.bcx && i0 + TXe == A.nx) : (A.bcy && j0 + TYe == A.ny);
            T qe[V], Em[V], dp[V], G[V];
            Ref<T> re;
#pragma unroll
            for (int v = 0; v < V; ++v) qe[v] = DELTA ? rfS[L::rf(v, ex, ey)] : T(0);
            if constexpr (DELTA) re = make_ref<EQ>(qe, A.ph);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                Em[v] = xe ? xR[L::xr(v, ey, ex + 1, kk)] : yT[L::yt(v, ey + 1, ex, kk)];
                if (wall) {
                    dp[v] = Em[v];
                } else {
                    const T h = xe ? xH[L::xh(v, ey, kk)] : yH[L::yh(v, ex, kk)];
                    const T on = DELTA ? (xe ? rfS[L::rf(v, ex + 1, ey)] : rfS[L::rf(v, ex, ey + 1)]) - qe[v] : T(0);
                    dp[v] = h + on;
                }
            }
            if (xe) face_flux<EQ, FLUX, 0, DELTA>(re, Em, dp, A.ph, G);
            else face_flux<EQ, FLUX, 1, DELTA>(re, Em, dp, A.ph, G);
            T* J = xe ? xF : yF;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                T* pj = J + L::ef(v, ey * TX + ex, kk);
                *pj = G[v] - *pj;
            }
        }
    }
    __syncthreads();

    // ---- phase 4: R on row k, stage update, store ----------------------------
    T o[N][V];
    if (valid) {
        // g_L'(eta_k), g_R'(eta_k): one select chain instead of an indexed
        // parameter load
        T glk = tb.dgl[0], grk = tb.dgr[0];
#pragma unroll
        for (int b = 1; b < N; ++b) {
            if (k == b) {
                glk = tb.dgl[b];
                grk = tb.dgr[b];
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            T acc[N], jb[N], jt[N];
            sm_load_row<N>(ryS + L::sq(v, el, k, 0), acc);
            sm_load_row<N>(jB + L::ef(v, el, 0), jb);
            sm_load_row<N>(yF + L::ef(v, el, 0), jt);
            const T JR = xF[L::ef(v, el, k)];
            if constexpr (PAIRED) {
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    const int i1 = PH(2 * i + 1);
                    Pr<T> ys = pfma(pmk(jb[2 * i], jb[i1]), pbc(glk), pmk(acc[2 * i], acc[i1]));
                    ys = pfma(pmk(jt[2 * i], jt[i1]), pbc(grk), ys);
                    Pr<T> xs = pfma(pbc(JL[v]), tp.dgl2[i], pmk(rx[2 * i][v], rx[i1][v]));
                    xs = pfma(pbc(JR), tp.dgr2[i], xs);
                    const Pr<T> r = pfma(pbc(-A.rhx2), xs, pmul(pbc(-A.rhy2), ys));
                    o[2 * i][v] = r.v.x;
                    if (2 * i + 1 < N) o[2 * i + 1][v] = r.v.y;
                }
            } else {
#pragma unroll
            for (int a = 0; a < N; ++a) {
                T ys = acc[a] + jb[a] * glk;
                ys = ys + jt[a] * grk;
                T xs = rx[a][v] + JL[v] * tb.dgl[a];
                xs = xs + JR * tb.dgr[a];
                o[a][v] = -A.rhy2 * ys - A.rhx2 * xs;
            }
            }
        }
        const long long off = e * NN + k * N;
        if (A.mode == MODE_RESIDUAL) {
        } else if (A.mode <= MODE_SO3) {
            const T dt = T(A.ctrl->dt);
            const T cA = A.mode == MODE_SO2 ? T(0.75) : T(1.0 / 3.0);
            const T cB = A.mode == MODE_SO1 ? T(1) : (A.mode == MODE_SO2 ? T(0.25) : T(2.0 / 3.0));
#pragma unroll
            for (int v = 0; v < V; ++v) {
                T qs[N], qn[N];
                gload_row<N>(A.qs + v * A.npts + off, qs);
                if (A.mode == MODE_SO1) {
#pragma unroll
                    for (int a = 0; a < N; ++a) o[a][v] = qs[a] + dt * o[a][v];
                } else {
                    gload_row<N>(A.qn + v * A.npts + off, qn);
#pragma unroll
                    for (int a = 0; a < N; ++a) o[a][v] = cA * qn[a] + cB * (qs[a] + dt * o[a][v]);
                }
            }
        } else {
            const T dt = T(A.ctrl->dt);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if (A.mode == MODE_INC1) {
#pragma unroll
                    for (int a = 0; a < N; ++a) o[a][v] = dt * o[a][v];
                } else {
                    T b[N];
                    gload_row<N>(A.qb + v * A.npts + off, b);
                    if (A.mode == MODE_INC2) {
#pragma unroll
                        for (int a = 0; a < N; ++a) o[a][v] = T(0.25) * (b[a] + dt * o[a][v]);
                    } else {
                        T hi[N], lo[N];
                        gload_row<N>(A.qs + v * A.npts + off, hi);
                        gload_row<N>(A.lo + v * A.npts + off, lo);
#pragma unroll
                        for (int a = 0; a < N; ++a) {
                            compensated_add(hi[a], lo[a], T(2.0 / 3.0) * (b[a] + dt * o[a][v]));
                            o[a][v] = hi[a];
                        }
                        gstore_row<N>(A.lo + v * A.npts + off, lo);
                    }
                }
            }
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            T row[N];
#pragma unroll
            for (int a = 0; a < N; ++a) row[a] = o[a][v];
            gstore_row<N>(A.out + v * A.npts + off, row);
        }
    }

    // ---- fused element averages (Algorithm 9) -----------------------------
    if (A.do_avg) {
        if (valid) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                T col[N];
#pragma unroll
                for (int a = 0; a < N; ++a) col[a] = o[a][v];
                avS[(v * TX * TY + el) * N + k] = line_dot<N>(tb.cavg[k], col);
            }
        }
        __syncthreads();
        if (valid && k == 0) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                T s = avS[(v * TX * TY + el) * N];
#pragma unroll
                for (int b = 1; b < N; ++b) s = s + avS[(v * TX * TY + el) * N + b];
                A.avg[(long long)v * (A.npts / NN) + e] = s;
            }
        }
    }

    // ---- fused max signal speed for the next CFL step ---------------------
    // (only CFL runs need the speed; a run of fixed steps only closes the
    // step; the branch is uniform over the grid)
    if (A.do_wave) {
        const bool cfl = !(A.ctrl->dt_fixed > 0.0);
        T m = T(0);
        if (cfl && valid) {
#pragma unroll
            for (int a = 0; a < N; ++a) {
                T s = point_speed<EQ>(o[a], A.ph);
                m = s > m ? s : m;
            }
        }
        block_time_update<T>(m, A.ctrl, /*advance=*/true, nslots, cfl);
    }
}

// PF: the instantiation for compensated stages whose states exceed L2 (it
// prefetches the low part; launched only when StageArgs::pf_lo is set).
template <class T, int P, int EQ, int DIV, int FLUX, int TX, int TY, bool DELTA, bool PF = false, bool WIDE = false>
__global__ void __launch_bounds__(TX * TY * (P + 1),
                                  (PF && stage_quad<T, EQ, DELTA> ? quad_min_blocks<P, WIDE, TX * TY>()
                                                                  : stage_min_blocks<T, P + 1, WIDE, TX * TY>()))
cpr_stage_kernel(const StageArgs<T> A)
{
    static_assert((TX * TY * (P + 1)) % 32 == 0, "whole warps: the warp-level reductions use every lane");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if constexpr (PF && stage_quad<T, EQ, DELTA>)
        stage_tile_quad<P, DIV, FLUX, TX, TY, true, MODE_INC3>(A, A.tab, A.qx, blockIdx.x, threadIdx.x, smem_raw,
                                                              gridDim.x);
    else
        stage_tile<T, P, EQ, DIV, FLUX, TX, TY, DELTA, PF>(A, A.tab, A.tp, blockIdx.x, threadIdx.x, smem_raw,
                                                           gridDim.x);
}

}  // namespace cpr
