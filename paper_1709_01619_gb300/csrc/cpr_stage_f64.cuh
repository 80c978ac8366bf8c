// cpr_stage_f64.cuh -- the tile of the fused residual + SSP-RK3 stage for the
// FP64 Euler equations (the scheme and its stage modes: cpr_stage.cuh).
//
// Bound by the FP64 pipe: each of an SM's four schedulers feeds half an FP64
// lane per cycle, so one operation keeps a scheduler busy for 64 cycles per
// warp, and the rest of the kernel hides behind that as soon as every
// scheduler has a warp or two.  So
//   - the operations are few: the pressure, velocities and 1 / rho of a point
//     serve the fluxes of both directions (LP divergence), the line operators
//     take the mirrored, joined form (line_derivative), reciprocals and square
//     roots are the short ones of cpr_common.cuh: 140 operations or 222 flops
//     per point and stage for p = 3, counted, against the general tile's 297
//     flops;
//   - the warps are many and alike: the threads of a CTA have one of two roles,
//     x-lines (rows) and y-lines (columns), and share the points of a row in
//     the phases that work on points, so that a thread has half the
//     operations of a thread that owns a row and a column.  A grid that
//     leaves schedulers idle runs in half the time, and a large one fills the
//     last round of warps better.
// 128^2 p = 3, 12 steps: 4.49 -> 3.09 ms (86 us per stage; the busiest scheduler
// gets 8 of 4096 warps where 6.7 is the mean, and its FP64 pipe is busy 84 % of
// the launch, the rest are the barriers of a tile); 16^2 elements, us per stage, p = 1 to 4: 25 /
// 41 / 36 / 56 -> 11 / 15 / 17 / 20.  With one thread for a row and a column, the
// same operations took 18 / 22 / 26 / 32.
//
// Shared memory holds quads (QuadArr).  Phases, a barrier after each:
//   1 the points: stage input, both fluxes (LP); halo lines (edge states)
//   2 the lines: edge states, line operator
//   3 common flux on the lower face of every line; the tile's upper edge
//   4 jumps, corrections: the direction's part of the residual
//   5 the points: stage update, store, CFL maximum; averages
// The fused operations are written out, so that tiles of every size round
// alike (a batch and single problems give the same bits).
#pragma once

#include "cpr_stage_quad.cuh"

namespace cpr {

template <int N, int TX, int TY>
struct F64Layout {
    using Q = QuadLayout<N, TX, TY>;  // index functions
    static constexpr int E = TX * TY;
    static constexpr int SQ = E * N * N;          // stage input; the result when averages are wanted
    static constexpr int SF = SQ, SG = SQ;        // fluxes, then the parts of the residual
    static constexpr int XR = TY * (TX + 1) * N;  // right edge states, elements -1..TX-1
    static constexpr int XH = TY * N;             // left edge states of the right halo
    static constexpr int XG = E * N;              // twice the common flux on the right face
    static constexpr int YT = (TY + 1) * TX * N;
    static constexpr int YH = TX * N;
    static constexpr int YG = E * N;
    static constexpr int TOTAL = SQ + SF + SG + XR + XH + XG + YT + YH + YG;
};

// Threads of a role, and of the CTA: whole warps.
constexpr int f64_role_threads(int p, int tx, int ty) { return stage_threads(tx * ty * (p + 1)); }

// F* - f from twice the common flux, one operation per variable.
__device__ __forceinline__ Quad<double> f64_jump(const Quad<double>& G2, const Quad<double>& f)
{
    return qmk(fma(0.5, G2.a.v.x, -f.a.v.x), fma(0.5, G2.a.v.y, -f.a.v.y), fma(0.5, G2.b.v.x, -f.b.v.x),
               fma(0.5, G2.b.v.y, -f.b.v.y));
}

template <int P, int DIV, int FLUX, int TX, int TY>
__device__ __forceinline__ void stage_tile_f64(const StageArgs<double>& A, const Tab<double>& tb,
                                               const QuadArgs<double>& qx, int tile, int tid,
                                               unsigned char* smem_raw, int nslots)
{
    using Qd = Quad<double>;
    constexpr int N = P + 1, NN = N * N, H = (N + 1) / 2;
    constexpr int E = TX * TY, NT = E * N, NR = (NT + 31) / 32 * 32;
    static_assert(2 * (TX > TY ? TX : TY) * N <= NT, "one halo line per thread of a role");
    using L = F64Layout<N, TX, TY>;
    using Q = typename L::Q;
    const QuadArr<double, L::SQ> sq{reinterpret_cast<Pr<double>*>(smem_raw)};
    const QuadArr<double, L::SF> sf{sq.end()}, sg{sf.end()};
    const QuadArr<double, L::XR> xR{sg.end()};
    const QuadArr<double, L::XH> xH{xR.end()};
    const QuadArr<double, L::XG> xG{xH.end()};
    const QuadArr<double, L::YT> yT{xG.end()};
    const QuadArr<double, L::YH> yH{yT.end()};
    const QuadArr<double, L::YG> yG{yH.end()};
    const QuadArr<double, L::XR> avS = xR;  // row sums of the averages
    const QuadTab<double>& qt = qx.tab;

    const int mode = A.mode;
    if (mode != MODE_RESIDUAL && A.ctrl->done) return;  // t_end reached: uniform exit
    // a limited run: clear the marked-element count of the limiter pass that
    // follows this stage
    if (mode != MODE_RESIDUAL && A.do_avg && tile == 0 && tid == 0) A.ctrl->marked = 0;

    const bool yrole = tid >= NR;  // uniform over a warp
    const int lt = yrole ? tid - NR : tid;
    const bool active = lt < NT;
    const int tj = (int)div_invariant((unsigned)tile, (unsigned)A.tiles_x, A.qx.tx_magic, A.qx.tx_shift);
    const int i0 = (tile - tj * A.tiles_x) * TX, j0 = tj * TY;
    const int TXe = min(TX, A.nx - i0), TYe = min(TY, A.ny - j0);
    // points: row k of element el, the lower half of it for the x-role
    const int el = lt / N, k = lt % N, tx = el % TX, ty = el / TX;
    const bool valid = active && tx < TXe && ty < TYe;
    const long long off = ((long long)(j0 + ty) * A.nx + (i0 + tx)) * NN + k * N;
    const int a0 = yrole ? H : 0, na = yrole ? N - H : H;
    // lines: row k of el, or a column (odd N: a warp holds one column of
    // consecutive elements, against bank conflicts)
    constexpr bool KMAJ = N % 2 == 1;
    const int ell = yrole && KMAJ ? lt % E : el, kl = yrole && KMAJ ? lt / E : k;
    const int txl = ell % TX, tyl = ell / TX;
    const bool validl = active && txl < TXe && tyl < TYe;
    auto at = [&](int i) { return yrole ? Q::sq(ell, i, kl) : Q::sq(ell, kl, i); };

    // ---- phase 1 ---------------------------------------------------------------
    if (valid) {
#pragma unroll
        for (int i = 0; i < H; ++i) {
            if (i < na) {
                const double* p = A.qs + off + a0 + i;
                const Qd x = qmk(p[0], p[A.npts], p[2 * A.npts], p[3 * A.npts]);
                const int s = Q::sq(el, k, a0 + i);
                sq.st(s, x);
                if constexpr (DIV == DIV_LP) {
                    Qd f, g;
                    quad_flux_xy(x, A.ph, f, g);
                    sf.st(s, f);
                    sg.st(s, g);
                }
            }
        }
    }
    {
        // the edge states of the neighbour elements facing the tile: x-role
        // left and right, y-role lower and upper
        const int len = yrole ? TX * N : TY * N;
        const int side = lt >= len, r = side ? lt - len : lt;
        const int pos = r / N, kk = r % N;
        int gi = yrole ? i0 + pos : (side ? i0 + TXe : i0 - 1);
        int gj = yrole ? (side ? j0 + TYe : j0 - 1) : j0 + pos;
        bool have = lt < 2 * len && pos < (yrole ? TXe : TYe);
        if (gi < 0 || gi >= A.nx) {
            have = have && !A.bcx;
            gi = gi < 0 ? gi + A.nx : gi - A.nx;
        }
        if (gj < 0 || gj >= A.ny) {
            have = have && !A.bcy;
            gj = gj < 0 ? gj + A.ny : gj - A.ny;
        }
        if (have) {
            const double* p = A.qs + ((long long)gj * A.nx + gi) * NN + (yrole ? kk : kk * N);
            Qd h[N];
#pragma unroll
            for (int l = 0; l < N; ++l) {
                const double* pl = p + (yrole ? l * N : l);
                h[l] = qmk(pl[0], pl[A.npts], pl[2 * A.npts], pl[3 * A.npts]);
            }
            const Qd es = side ? edge_lo<N>(qt, h) : edge_hi<N>(qt, h);
            if (yrole) {
                if (side) yH.st(pos * N + kk, es);
                else yT.st(Q::yt(0, pos, kk), es);
            } else {
                if (side) xH.st(pos * N + kk, es);
                else xR.st(Q::xr(pos, 0, kk), es);
            }
        }
    }
    __syncthreads();

    // ---- phase 2 ---------------------------------------------------------------
    Qd r[N], e0, f0, f1;  // line operator; lower edge state; fluxes the jumps are taken from
    if (validl) {
        Qd x[N], e1;
#pragma unroll
        for (int i = 0; i < N; ++i) x[i] = sq.ld(at(i));
        if constexpr (DIV == DIV_LP) {
            e0 = edge_lo<N>(qt, x);
            e1 = edge_hi<N>(qt, x);
            const QuadArr<double, L::SF> fl{yrole ? sg.p : sf.p};
#pragma unroll
            for (int i = 0; i < N; ++i) x[i] = fl.ld(at(i));
            f0 = x[0];
            f1 = x[N - 1];
            line_derivative<N>(qt, x, r);
        } else if (yrole) {
            quad_line<N, 1, DIV>(qt, A.ph, x, r, e0, e1, f0, f1);
        } else {
            quad_line<N, 0, DIV>(qt, A.ph, x, r, e0, e1, f0, f1);
        }
        if (yrole) yT.st(Q::yt(tyl + 1, txl, kl), e1);
        else xR.st(Q::xr(tyl, txl + 1, kl), e1);
    }
    __syncthreads();

    // ---- phase 3 ---------------------------------------------------------------
    Qd j0q;  // jump on the lower face
    if (yrole) {
        if (validl) {
            const Qd dm = A.bcy && j0 + tyl == 0 ? e0 : yT.ld(Q::yt(tyl, txl, kl));
            const Qd G = quad_face2<FLUX, 1>(dm, e0, A.ph);
            if (tyl > 0) yG.st(Q::ef(ell - TX, kl), G);
            j0q = f64_jump(G, f0);
        }
        if (lt < TX * N && lt / N < TXe) {
            const int pos = lt / N, kk = lt % N;
            const Qd Em = yT.ld(Q::yt(TYe, pos, kk));
            const Qd dp = A.bcy && j0 + TYe == A.ny ? Em : yH.ld(pos * N + kk);
            yG.st(Q::ef((TYe - 1) * TX + pos, kk), quad_face2<FLUX, 1>(Em, dp, A.ph));
        }
    } else {
        if (validl) {
            const Qd dm = A.bcx && i0 + txl == 0 ? e0 : xR.ld(Q::xr(tyl, txl, kl));
            const Qd G = quad_face2<FLUX, 0>(dm, e0, A.ph);
            if (txl > 0) xG.st(Q::ef(ell - 1, kl), G);
            j0q = f64_jump(G, f0);
        }
        if (lt < TY * N && lt / N < TYe) {
            const int pos = lt / N, kk = lt % N;
            const Qd Em = xR.ld(Q::xr(pos, TXe, kk));
            const Qd dp = A.bcx && i0 + TXe == A.nx ? Em : xH.ld(pos * N + kk);
            xG.st(Q::ef(pos * TX + TXe - 1, kk), quad_face2<FLUX, 0>(Em, dp, A.ph));
        }
    }
    __syncthreads();

    // ---- phase 4 ---------------------------------------------------------------
    if (validl) {
        const Qd j1 = f64_jump(yrole ? yG.ld(Q::ef(ell, kl)) : xG.ld(Q::ef(ell, kl)), f1);
        const QuadArr<double, L::SF> part{yrole ? sg.p : sf.p};
#pragma unroll
        for (int i = 0; i < N; ++i)
            part.st(at(i), qfma(j1, -qt.dgl[N - 1 - i], qfma(j0q, qt.dgl[i], r[i])));
    }
    __syncthreads();

    // ---- phase 5 ---------------------------------------------------------------
    const bool wave = A.do_wave && !(A.ctrl->dt_fixed > 0.0);
    double m = 0.0;
    if (valid) {
        // the factor of R in the stage's result
        double w = mode == MODE_RESIDUAL ? 1.0 : A.ctrl->dt;
        if (mode == MODE_SO2) w *= 0.25;
        if (mode == MODE_SO3) w *= 2.0 / 3.0;
        const double sx = -A.rhx2 * w, sy = -A.rhy2 * w;
        const double c0 = mode == MODE_SO2 ? 0.25 : 1.0 / 3.0, c1 = mode == MODE_SO2 ? 0.75 : 2.0 / 3.0;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            if (i < na) {
                const int s = Q::sq(el, k, a0 + i);
                double o[4];
                qget(qfma(sf.ld(s), sx, qmul(sg.ld(s), sy)), o);
                const long long at0 = off + a0 + i;
                // the states last: two roundings of their size
                if (mode != MODE_RESIDUAL) {
                    double qs[4];
                    qget(sq.ld(s), qs);
                    if (mode == MODE_SO1) {
#pragma unroll
                        for (int v = 0; v < 4; ++v) o[v] = qs[v] + o[v];
                    } else {
                        // the smaller multiple first: its rounding is the smaller one
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const double qn = A.qn[v * A.npts + at0];
                            o[v] = fma(c1, mode == MODE_SO2 ? qn : qs[v], fma(c0, mode == MODE_SO2 ? qs[v] : qn, o[v]));
                        }
                    }
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) A.out[v * A.npts + at0] = o[v];
                if (A.do_avg) sq.st(s, qput(o));
                if (wave) {
                    const double sp = point_speed<EQ_EULER, true>(o, A.ph);
                    m = sp > m ? sp : m;
                }
            }
        }
    }

    // ---- fused element averages (Algorithm 9) -----------------------------
    if (A.do_avg) {
        __syncthreads();
        if (valid && !yrole) {
            double o[4][N], sv[4];
#pragma unroll
            for (int a = 0; a < N; ++a) {
                double x[4];
                qget(sq.ld(Q::sq(el, k, a)), x);
#pragma unroll
                for (int v = 0; v < 4; ++v) o[v][a] = x[v];
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) sv[v] = line_dot<N>(tb.cavg[k], o[v]);
            avS.st(Q::ef(el, k), qput(sv));
        }
        __syncthreads();
        const int ax = tid % TX, ay = tid / TX;
        if (tid < E && ax < TXe && ay < TYe) {
            Qd s = avS.ld(Q::ef(tid, 0));
#pragma unroll
            for (int b = 1; b < N; ++b) s = qadd(s, avS.ld(Q::ef(tid, b)));
            double sv[4];
            qget(s, sv);
            const long long ne = A.npts / NN, ea = (long long)(j0 + ay) * A.nx + (i0 + ax);
#pragma unroll
            for (int v = 0; v < 4; ++v) A.avg[v * ne + ea] = sv[v];
        }
    }
    if (A.do_wave) block_time_update<double>(m, A.ctrl, /*advance=*/true, nslots, wave);
}

// Tiles of a single problem's kernels (f64_tile picks one): 8 x 4, 4 x 4 and,
// for p = 4 whose 4 x 4 tile has six warps for four schedulers, 4 x 2 elements.
constexpr int f64_tiles(int p) { return p == 4 ? 3 : 2; }
constexpr int f64_tile_x(int k) { return k == 0 ? 8 : 4; }
constexpr int f64_tile_y(int k) { return k == 2 ? 2 : 4; }
// Resident CTAs that the registers are sized for: 16 warps per SM of 128
// registers for p = 3.
constexpr int f64_min_blocks(int p, int k) { return p != 3 ? 1 : k == 0 ? 2 : 4; }

template <int P, int DIV, int FLUX, int TX, int TY, int MINB>
__global__ void __launch_bounds__(2 * f64_role_threads(P, TX, TY), MINB) cpr_stage_f64_kernel(const StageArgs<double> A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_order();
    stage_tile_f64<P, DIV, FLUX, TX, TY>(A, A.tab, A.qx, blockIdx.x, threadIdx.x, smem_raw, gridDim.x);
}

}  // namespace cpr
