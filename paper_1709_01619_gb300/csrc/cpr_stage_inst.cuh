// cpr_stage_inst.cuh -- launcher of the stage kernel for one (dtype, order);
// included by one translation unit per (dtype, order) so that they compile
// in parallel.
#pragma once

#include <type_traits>

#include "cpr_launch.h"
#include "cpr_tabconv.cuh"
#include "cpr_stage.cuh"
#include "cpr_adjoint_quad.cuh"

namespace cpr {


// The FP32 Euler stage updates (quad form).  A single problem with the LP
// divergence and Rusanov's flux takes a kernel compiled for the stage mode
// (1-6; the arrays it reads and its update are then fixed at compile time:
// 1024^2 p = 3 4.63 -> 4.51 ms for 8 steps, 128^2 1.178 -> 1.105 ms for 64);
// other divergences and fluxes one kernel for every mode.  So does an instance
// of a batch: its SMs run CTAs of every order and stage at once, and the
// kernels of three orders and three modes evict one another's instructions
// (64 instances, 24 steps: 32.5 ms with one kernel per order, 35.0 with three).
template <int P, int DIV, int FLUX, int TX, int TY, class F>
static cudaError_t with_quad_kernel(int mode, bool wide, bool shared, F&& f)
{
    constexpr int E = TX * TY, MB = quad_min_blocks<P, false, E>(), MW = quad_min_blocks<P, true, E>();
    constexpr int MS = stage_min_blocks<float, P + 1, false, E>();
    if (shared) return f(cpr_stage_quad_kernel<P, DIV, FLUX, TX, TY, MS, 0>);
    if constexpr (DIV == DIV_LP && FLUX == FLUX_RUSANOV) {
        auto pick = [&](auto m) {
            constexpr int M = decltype(m)::value;
            return wide ? f(cpr_stage_quad_kernel<P, DIV, FLUX, TX, TY, MW, M>)
                        : f(cpr_stage_quad_kernel<P, DIV, FLUX, TX, TY, MB, M>);
        };
        switch (mode) {
        case MODE_SO1: return pick(std::integral_constant<int, MODE_SO1>{});
        case MODE_SO2: return pick(std::integral_constant<int, MODE_SO2>{});
        case MODE_SO3: return pick(std::integral_constant<int, MODE_SO3>{});
        case MODE_INC1: return pick(std::integral_constant<int, MODE_INC1>{});
        case MODE_INC2: return pick(std::integral_constant<int, MODE_INC2>{});
        default: return pick(std::integral_constant<int, MODE_INC3>{});
        }
    } else {
        return wide ? f(cpr_stage_quad_kernel<P, DIV, FLUX, TX, TY, MW, 0>)
                    : f(cpr_stage_quad_kernel<P, DIV, FLUX, TX, TY, MB, 0>);
    }
}

// The tile of a single FP64 problem.  A stage takes the time of the scheduler
// with most warps (cpr_stage_f64.cuh): of n tiles (size(k, tx, ty) gives their
// elements and returns their warps), the one with the fewest warps on the
// busiest scheduler, each step down counted 10 % dearer for its longer
// boundary.  An instance of a batch (sms 0) takes the largest.
// us per Euler stage, p = 3: 16^2 elements 16.7 (4 x 4), 64^2 26.4, 96^2 45.9
// (8 x 8 tiles, one thread for a row and a column: 36 at every size below 64^2).
template <class F>
inline int f64_tile(const LaunchCfg& c, int n, F&& size)
{
    int best = 0;
    double cost = 0.0, dearer = 1.0;
    for (int k = 0; c.sms > 0 && k < n; ++k, dearer *= 1.1) {
        int tx, ty;
        const int tile_warps = size(k, &tx, &ty);
        const long long ctas = (long long)((c.nx + tx - 1) / tx) * ((c.ny + ty - 1) / ty);
        const long long warps = (ctas + c.sms - 1) / c.sms * tile_warps;
        const double w = (double)((warps + 3) / 4) * dearer;
        if (k == 0 || w < cost) {
            best = k;
            cost = w;
        }
    }
    return best;
}

template <int P, int DIV, int FLUX, int K>
static cudaError_t stage_f64_tile(const LaunchCfg& c, StageArgs<double> A, cudaStream_t s, bool prep)
{
    constexpr int TX = f64_tile_x(K), TY = f64_tile_y(K);
    const size_t smem = stage_smem<double, P, EQ_EULER, TX, TY, false>();
    auto kern = cpr_stage_f64_kernel<P, DIV, FLUX, TX, TY, f64_min_blocks(P, K)>;
    if (prep) return allow_smem(kern, smem);
    A.tiles_x = (c.nx + TX - 1) / TX;
    div_magic((unsigned)A.tiles_x, &A.qx.tx_magic, &A.qx.tx_shift);
    return launch_ordered(c, kern, A.tiles_x * ((c.ny + TY - 1) / TY), 2 * f64_role_threads(P, TX, TY), smem, s, A);
}

template <int P, int DIV, int FLUX>
static cudaError_t stage_f64(const LaunchCfg& c, const StageArgs<double>& A, cudaStream_t s, bool prep)
{
    const int k = f64_tile(c, f64_tiles(P), [](int i, int* tx, int* ty) {
        *tx = f64_tile_x(i);
        *ty = f64_tile_y(i);
        return 2 * f64_role_threads(P, *tx, *ty) / 32;
    });
    if constexpr (f64_tiles(P) > 2)
        if (k == 2) return stage_f64_tile<P, DIV, FLUX, 2>(c, A, s, prep);
    return k == 1 ? stage_f64_tile<P, DIV, FLUX, 1>(c, A, s, prep) : stage_f64_tile<P, DIV, FLUX, 0>(c, A, s, prep);
}

template <class T, int P, int K>
static cudaError_t stage_adv_tile(const LaunchCfg& c, StageArgs<T> A, cudaStream_t s, bool prep)
{
    constexpr int TX = adv_tile_x(P, K), TY = adv_tile_y(P, K);
    const size_t smem = stage_smem<T, P, EQ_ADV, TX, TY, false>();
    auto kern = cpr_stage_adv_kernel<T, P, TX, TY>;
    if (prep) return allow_smem(kern, smem);
    A.rhx2 = T(2.0 / c.hx * c.ax);  // the operator's factors, the velocity in them
    A.rhy2 = T(2.0 / c.hy * c.ay);
    A.tiles_x = (c.nx + TX - 1) / TX;
    div_magic((unsigned)A.tiles_x, &A.qx.tx_magic, &A.qx.tx_shift);
    kern<<<A.tiles_x * ((c.ny + TY - 1) / TY), stage_threads(TX * TY * (P + 1)), smem, s>>>(A);
    return cudaGetLastError();
}

template <class T, int P>
static cudaError_t stage_adv(const LaunchCfg& c, const StageArgs<T>& A, cudaStream_t s, bool prep)
{
    if constexpr (sizeof(T) == 8) {
        const int k = f64_tile(c, 2, [](int i, int* tx, int* ty) {
            *tx = adv_tile_x(P, i);
            *ty = adv_tile_y(P, i);
            return stage_threads(*tx * *ty * (P + 1)) / 32;
        });
        if (k == 1) return stage_adv_tile<T, P, 1>(c, A, s, prep);
    }
    return stage_adv_tile<T, P, 0>(c, A, s, prep);
}

template <class T, int P, int EQ, int DIV, int FLUX>
static cudaError_t stage_one(const LaunchCfg& c, const StageArgs<T>& A, int ctas, cudaStream_t s, bool prep)
{
    if constexpr (EQ == EQ_ADV) return stage_adv<T, P>(c, A, s, prep);
    else if constexpr (sizeof(T) == 8) return stage_f64<P, DIV, FLUX>(c, A, s, prep);
    else {
    constexpr int N = P + 1, V = NVars<EQ>::value;
    constexpr int TX = stage_tile_x(P), TY = stage_tile_y(P);
    constexpr int NT = TX * TY * N;
    constexpr bool DELTA = stage_delta<T>();
    // FP32 Euler: the quad form for the stage updates; the stand-alone
    // residual, and every other type and equation, the general kernel
    constexpr bool QUAD = stage_quad<T, EQ, DELTA>;
    const size_t smem = sizeof(T) * StageLayout<N, V, TX, TY, DELTA>::TOTAL;
    [[maybe_unused]] const size_t smem_q = stage_smem<T, P, EQ, TX, TY, DELTA>();
    auto kern = cpr_stage_kernel<T, P, EQ, DIV, FLUX, TX, TY, DELTA>;
    // the prefetching instantiation only where the compensated FP32 stages
    // run on large states: Euler, LP divergence, Rusanov flux
    constexpr bool HAS_PF = sizeof(T) == 4 && EQ == EQ_EULER && DIV == DIV_LP && FLUX == FLUX_RUSANOV;
    auto kern_pf = cpr_stage_kernel<T, P, EQ, DIV, FLUX, TX, TY, DELTA, HAS_PF>;
    // and the one for grids of at most two CTAs per SM: FP32 Euler, every
    // divergence and flux
    constexpr bool HAS_WIDE = sizeof(T) == 4 && EQ == EQ_EULER;
    auto kern_w = cpr_stage_kernel<T, P, EQ, DIV, FLUX, TX, TY, DELTA, false, HAS_WIDE>;
    // CTAs per SM the wide instantiation is compiled for: the grid fits the
    // device at once up to that many per SM
    constexpr int WIDE_PER_SM = stage_min_blocks<T, N, true, TX * TY>();
    const bool wide = HAS_WIDE && c.sms > 0 && ctas <= WIDE_PER_SM * c.sms;
    if (prep) {
        auto limit = [](auto k, size_t bytes) { return allow_smem(k, bytes); };
        cudaError_t e = limit(kern, smem);
        if (e == cudaSuccess && HAS_PF) e = limit(kern_pf, QUAD ? smem_q : smem);
        if (e == cudaSuccess && HAS_WIDE) e = limit(kern_w, smem);
        if constexpr (QUAD)
            for (int mode = MODE_SO1; mode <= MODE_INC3 && e == cudaSuccess; ++mode) {
                auto lq = [&](auto k) { return limit(k, smem_q); };
                e = with_quad_kernel<P, DIV, FLUX, TX, TY>(mode, false, c.shared, lq);
                if (e == cudaSuccess) e = with_quad_kernel<P, DIV, FLUX, TX, TY>(mode, true, c.shared, lq);
            }
        return e;
    }
    if constexpr (QUAD) {
        if (A.mode != MODE_RESIDUAL) {
            auto launch = [&](auto k) {
                // a kernel compiled for its Shu-Osher stage: in order behind another
                if (DIV == DIV_LP && FLUX == FLUX_RUSANOV && !c.shared && quad_ordered(A.mode))
                    return launch_ordered(c, k, ctas, NT, smem_q, s, A);
                k<<<ctas, NT, smem_q, s>>>(A);
                return cudaGetLastError();
            };
            if (HAS_PF && A.pf_lo && !c.shared) return launch(kern_pf);
            return with_quad_kernel<P, DIV, FLUX, TX, TY>(A.mode, wide, c.shared, launch);
        }
    }
    if (wide) kern_w<<<ctas, NT, smem, s>>>(A);
    else kern<<<ctas, NT, smem, s>>>(A);
    return cudaGetLastError();
    }
}

template <class T, int P>
static cudaError_t stage_dispatch(const LaunchCfg& c, const StageArgs<T>& A, int ctas, cudaStream_t s, bool prep)
{
    // advection: every divergence and flux is one operator (cpr_stage_adv.cuh)
    if (c.eqn == EQ_ADV) return stage_one<T, P, EQ_ADV, DIV_LP, FLUX_UPWIND>(c, A, ctas, s, prep);
    if (c.flux == FLUX_ROE)
        return c.div == DIV_LP ? stage_one<T, P, EQ_EULER, DIV_LP, FLUX_ROE>(c, A, ctas, s, prep)
                               : stage_one<T, P, EQ_EULER, DIV_CHAIN, FLUX_ROE>(c, A, ctas, s, prep);
    return c.div == DIV_LP ? stage_one<T, P, EQ_EULER, DIV_LP, FLUX_RUSANOV>(c, A, ctas, s, prep)
                           : stage_one<T, P, EQ_EULER, DIV_CHAIN, FLUX_RUSANOV>(c, A, ctas, s, prep);
}

template <class T>
static StageArgs<T> make_stage_args(const LaunchCfg& c, int mode, const StagePtrs& b, bool do_wave)
{
    StageArgs<T> A;
    A.qs = static_cast<const T*>(b.qs);
    A.qb = static_cast<const T*>(b.qb);
    A.qn = static_cast<const T*>(b.qn);
    A.out = static_cast<T*>(b.out);
    A.lo = static_cast<T*>(b.lo);
    A.avg = static_cast<T*>(b.avg);
    A.ctrl = c.ctrl;
    A.npts = c.npts;
    A.nx = c.nx;
    A.ny = c.ny;
    A.bcx = c.bcx;
    A.bcy = c.bcy;
    A.tiles_x = (c.nx + stage_tile_x(c.p) - 1) / stage_tile_x(c.p);
    A.mode = mode;
    A.do_avg = b.avg != nullptr;
    A.do_wave = do_wave;
    // the five state arrays of the compensated stage exceed L2
    A.pf_lo = mode == MODE_INC3 && b.lo != nullptr &&
              (double)c.npts * (c.eqn == EQ_EULER ? 4 : 1) * sizeof(T) * 5.0 > (double)c.l2_bytes;
    A.rhx2 = T(2.0 / c.hx);
    A.rhy2 = T(2.0 / c.hy);
    A.ph.gamma = T(c.gamma);
    A.ph.ax = T(c.ax);
    A.ph.ay = T(c.ay);
    A.tab = host_tab<T>(c.tab);
    A.tp = host_tabpr<T>(c.tab);
    A.qx.tab = host_quadtab<T>(c.tab, (c.eqn == EQ_ADV || c.div == DIV_LP) && quad_joined<T>(c.p + 1));
    div_magic((unsigned)A.tiles_x, &A.qx.tx_magic, &A.qx.tx_shift);
    return A;
}

template <class T, int P>
cudaError_t launch_stage_p(const LaunchCfg& c, int mode, const StagePtrs& b, bool do_wave, cudaStream_t s)
{
    StageArgs<T> A = make_stage_args<T>(c, mode, b, do_wave);
    return stage_dispatch<T, P>(c, A, stage_ctas(c), s, false);
}

template <class T, int P>
cudaError_t prepare_stage_p(const LaunchCfg& c)
{
    StagePtrs b{};
    StageArgs<T> A = make_stage_args<T>(c, 0, b, false);
    return stage_dispatch<T, P>(c, A, 0, 0, true);
}

// Tile of the adjoint kernels: 8 x 4 elements (twice as many CTAs per SM as
// 8 x 8 ones in the same shared memory: 1024^2 p = 3 FP32 0.441 -> 0.411 ms per
// launch of the kernel with one word per variable); FP64 advection 8 x 8, or
// 8 x 4 where 8 x 8 would exceed the shared memory of one CTA.
template <class T, int P, int EQ>
struct VjpTile {
    static constexpr int X = 8;
    static constexpr int Y = sizeof(T) == 8 && EQ == EQ_ADV && P < 4 ? 8 : 4;
};

template <class T, int P, int EQ, int FLUX>
static cudaError_t vjp_one(const LaunchCfg& c, const VjpPtrs& b, cudaStream_t s, bool prep)
{
    constexpr int N = P + 1, V = NVars<EQ>::value;
    constexpr int TX = VjpTile<T, P, EQ>::X, TY = VjpTile<T, P, EQ>::Y;
    auto kern = [] {
        if constexpr (EQ == EQ_EULER) return cpr_vjp_quad_kernel<T, P, TX, TY>;
        else return cpr_residual_vjp_kernel<T, P, EQ, FLUX, TX, TY>;
    }();
    const size_t smem = EQ == EQ_EULER ? sizeof(Quad<T>) * VjpQuadLayout<T, N, TX, TY>::TOTAL
                                       : sizeof(T) * VjpLayout<N, V, TX, TY>::TOTAL;
    if (prep) return allow_smem(kern, smem);
    VjpArgs<T> A;
    A.q = static_cast<const T*>(b.q);
    A.rbar = static_cast<const T*>(b.rbar);
    A.out = static_cast<T*>(b.out);
    A.X0 = static_cast<const T*>(b.X0);
    A.X1 = static_cast<const T*>(b.X1);
    A.X2 = static_cast<const T*>(b.X2);
    A.c0 = T(b.c0);
    A.c1 = T(b.c1);
    A.c2 = T(b.c2);
    A.cv = T(b.cv);
    A.npts = c.npts;
    A.nx = c.nx;
    A.ny = c.ny;
    A.bcx = c.bcx;
    A.bcy = c.bcy;
    A.tiles_x = (c.nx + TX - 1) / TX;
    A.rhx2 = T(2.0 / c.hx);
    A.rhy2 = T(2.0 / c.hy);
    A.ph.gamma = T(c.gamma);
    A.ph.ax = T(c.ax);
    A.ph.ay = T(c.ay);
    A.tab = host_tab<T>(c.tab);
    for (int a = 0; a < kMaxN; ++a)
        for (int l = 0; l < kMaxN; ++l)
            A.MT[l][a] = (a < N && l < N)
                             ? T(c.tab.D[a][l] - c.tab.lm[l] * c.tab.dgl[a] - c.tab.lp[l] * c.tab.dgr[a])
                             : T(0);
    const int ctas = A.tiles_x * ((c.ny + TY - 1) / TY);
    if constexpr (EQ == EQ_EULER) return launch_ordered(c, kern, ctas, TX * TY * N, smem, s, A);
    kern<<<ctas, TX * TY * N, smem, s>>>(A);
    return cudaGetLastError();
}

template <class T, int P>
cudaError_t launch_vjp_p(const LaunchCfg& c, const VjpPtrs& b, cudaStream_t s, bool prep)
{
    if (c.eqn == EQ_EULER) return vjp_one<T, P, EQ_EULER, FLUX_RUSANOV>(c, b, s, prep);
    if (c.flux == FLUX_UPWIND) return vjp_one<T, P, EQ_ADV, FLUX_UPWIND>(c, b, s, prep);
    return vjp_one<T, P, EQ_ADV, FLUX_RUSANOV>(c, b, s, prep);
}

}  // namespace cpr

#define CPR_INSTANTIATE_STAGE(T, P)                                                                     \
    template cudaError_t cpr::launch_stage_p<T, P>(const LaunchCfg&, int, const StagePtrs&, bool, cudaStream_t); \
    template cudaError_t cpr::prepare_stage_p<T, P>(const LaunchCfg&);                                  \
    template cudaError_t cpr::launch_vjp_p<T, P>(const LaunchCfg&, const VjpPtrs&, cudaStream_t, bool);
