// cpr_stage_adv.cuh -- the tile of the fused residual + SSP-RK3 stage for linear
// advection (the scheme and its stage modes: cpr_stage.cuh).
//
// With the constant velocity (ax, ay) both divergences are one linear
// operator, and Rusanov's flux, whose lambda is |a|, is the upwind flux.  So
// no point flux and no face pass is left: along a line of an element
//   f'_a = c [ sum_l D'_al q_l + (e_L - q_0) g_L'_a + (e_R - q_{N-1}) g_R'_a ],
// c = a (-2 / h), D' the joined operator of line_derivative, and e_L, e_R the
// upwind edge state of the two faces: the upper edge of the lower element for
// a >= 0, else the lower edge of the upper one.  Either way the state of face
// f of a row of the tile is formed by one thread into slot f.
// FP32 with N < 4 (quad_joined) takes D and the element's own edge states in
// place of D', q_0 and q_{N-1}: every rounded entry of the operator is an error
// common to all elements and steps, and there the joined one has more of it.
//
// Thread (el, k): row k of element el in phases 1 and 4, a column of an element
// in phases 2 and 3.
//   1 own row into the tile copy, its outflow edge; the halo lines upwind of
//     the tile (the domain's transmissive edge takes the inner state)
//   2 column: outflow edge, D' q
//   3 column: jumps, the whole y-part over the column
//   4 row: jumps, both parts, stage update, store; averages
// For even N a warp holds whole elements, so only the edge states need a CTA
// barrier (after phase 2).
//
// Against the general tile, us per FP64 stage on 16^2 elements, p = 1 to 4: 6.1 /
// 9.1 / 13.3 / 12.1 -> 4.7 / 5.5 / 6.3 / 7.3, 96^2 6.2 / 9.3 / 13.5 / 19.3 -> 4.9 /
// 7.3 / 9.8 / 13.8; FP32 is bound by the launch (3.2 to 3.7 -> 3.1 to 3.6).
#pragma once

#include "cpr_stage_quad.cuh"

namespace cpr {

template <int N, int TX, int TY>
struct AdvLayout {
    static constexpr int NN = N * N, E = TX * TY;
    // N = 4: the element index shifts the rows, else the columns of a warp's
    // elements (stride 16 words) would meet in few banks
    static constexpr int SQ = E * NN;             // tile copy, then the y-part
    static constexpr int XE = TY * (TX + 1) * N;  // edge state of every x-face
    static constexpr int YE = (TY + 1) * TX * N;  // edge state of every y-face
    static constexpr int AV = E * N;              // row sums of the averages
    static constexpr int TOTAL = SQ + XE + YE + AV;
    __device__ static int sq(int el, int b, int a)
    {
        if constexpr (N == 4) return el * 16 + ((b ^ (el & 3)) << 2) + a;
        else return el * NN + b * N + a;
    }
    __device__ static int xe(int ty, int f, int k) { return (ty * (TX + 1) + f) * N + k; }
    __device__ static int ye(int f, int tx, int k) { return (f * TX + tx) * N + k; }
};

template <class T, int P, int TX, int TY>
__device__ __forceinline__ void stage_tile_adv(const StageArgs<T>& A, const Tab<T>& tb, const QuadArgs<T>& qx,
                                               int tile, int tid, unsigned char* smem_raw,
                                               int nslots)
{
    constexpr int N = P + 1, NN = N * N;
    constexpr int NT = TX * TY * N;
    using L = AdvLayout<N, TX, TY>;
    T* sq = reinterpret_cast<T*>(smem_raw);
    T* xE = sq + L::SQ;
    T* yE = xE + L::XE;
    T* avS = yE + L::YE;
    const QuadTab<T>& qt = qx.tab;
    constexpr bool J = quad_joined<T>(N);
    const int mode = A.mode;
    if (mode != MODE_RESIDUAL && A.ctrl->done) return;  // t_end reached: uniform exit
    // a limited run: clear the marked-element count of the limiter pass that
    // follows this stage
    if (mode != MODE_RESIDUAL && A.do_avg && tile == 0 && tid == 0) A.ctrl->marked = 0;

    const bool active = tid < NT;
    const int tj = (int)div_invariant((unsigned)tile, (unsigned)A.tiles_x, A.qx.tx_magic, A.qx.tx_shift);
    const int i0 = (tile - tj * A.tiles_x) * TX, j0 = tj * TY;
    const int TXe = min(TX, A.nx - i0), TYe = min(TY, A.ny - j0);
    const int el = tid / N, k = tid % N;
    const int tx = el % TX, ty = el / TX;
    const bool valid = active && tx < TXe && ty < TYe;
    const long long e = (long long)(j0 + ty) * A.nx + (i0 + tx);
    const long long off = e * NN + k * N;
    const bool addb = mode == MODE_INC2 || mode == MODE_INC3;
    const bool xup = A.ph.ax >= T(0), yup = A.ph.ay >= T(0);

    // ---- phase 1 ---------------------------------------------------------------
    T x[N];
    if (valid) {
        gload_row<N>(A.qs + off, x);
        if (addb) {
            T b[N];
            gload_row<N>(A.qb + off, b);
#pragma unroll
            for (int a = 0; a < N; ++a) x[a] += b[a];
        }
    }
    for (int t = tid; t < (TX + TY) * N; t += (NT + 31) / 32 * 32) {
        // the line of the element upwind of the tile
        const bool xd = t < TY * N;
        const int r = xd ? t : t - TY * N;
        const int pos = r / N, kk = r % N;
        const bool upw = xd ? xup : yup;
        int gi = xd ? (upw ? i0 - 1 : i0 + TXe) : i0 + pos;
        int gj = xd ? j0 + pos : (upw ? j0 - 1 : j0 + TYe);
        bool have = pos < (xd ? TYe : TXe);
        if (gi < 0 || gi >= A.nx) {
            have = have && !A.bcx;
            gi = gi < 0 ? gi + A.nx : gi - A.nx;
        }
        if (gj < 0 || gj >= A.ny) {
            have = have && !A.bcy;
            gj = gj < 0 ? gj + A.ny : gj - A.ny;
        }
        if (have) {
            const long long eh = ((long long)gj * A.nx + gi) * NN + (xd ? kk * N : kk);
            T h[N];
#pragma unroll
            for (int l = 0; l < N; ++l) {
                h[l] = A.qs[eh + (xd ? l : l * N)];
                if (addb) h[l] += A.qb[eh + (xd ? l : l * N)];
            }
            const T es = upw ? edge_hi<N>(qt, h) : edge_lo<N>(qt, h);
            if (xd) xE[L::xe(pos, upw ? 0 : TXe, kk)] = es;
            else yE[L::ye(upw ? 0 : TYe, pos, kk)] = es;
        }
    }
    if (valid) {
#pragma unroll
        for (int a = 0; a < N; ++a) sq[L::sq(el, k, a)] = x[a];
        xE[L::xe(ty, xup ? tx + 1 : tx, k)] = xup ? edge_hi<N>(qt, x) : edge_lo<N>(qt, x);
        // transmissive inflow edge: the element's own state there
        if (A.bcx && xup && i0 + tx == 0) xE[L::xe(ty, 0, k)] = edge_lo<N>(qt, x);
        if (A.bcx && !xup && i0 + tx == A.nx - 1) xE[L::xe(ty, TXe, k)] = edge_hi<N>(qt, x);
    }
    // phases 2 to 4 read from the tile copy what threads of the same element wrote
    constexpr bool KMAJ = N % 2 == 1;
    constexpr bool WARP = !KMAJ && 32 % N == 0;
    if constexpr (WARP) __syncwarp();
    else __syncthreads();

    // ---- phase 2 ---------------------------------------------------------------
    const int elc = KMAJ ? tid % (TX * TY) : el, kc = KMAJ ? tid / (TX * TY) : k;
    const int txc = elc % TX, tyc = elc / TX;
    const bool validc = active && txc < TXe && tyc < TYe;
    T ry[N], c0, c1;
    if (validc) {
        T c[N];
#pragma unroll
        for (int b = 0; b < N; ++b) c[b] = sq[L::sq(elc, b, kc)];
        c0 = J ? c[0] : edge_lo<N>(qt, c);
        c1 = J ? c[N - 1] : edge_hi<N>(qt, c);
        yE[L::ye(yup ? tyc + 1 : tyc, txc, kc)] = yup ? edge_hi<N>(qt, c) : edge_lo<N>(qt, c);
        if (A.bcy && yup && j0 + tyc == 0) yE[L::ye(0, txc, kc)] = edge_lo<N>(qt, c);
        if (A.bcy && !yup && j0 + tyc == A.ny - 1) yE[L::ye(TYe, txc, kc)] = edge_hi<N>(qt, c);
        line_derivative<N>(qt, c, ry);
    }
    __syncthreads();

    // ---- phase 3 ---------------------------------------------------------------
    if (validc) {
        const T jb = yE[L::ye(tyc, txc, kc)] - c0, jt = yE[L::ye(tyc + 1, txc, kc)] - c1;
#pragma unroll
        for (int b = 0; b < N; ++b)
            sq[L::sq(elc, b, kc)] = fma(jt, -qt.dgl[N - 1 - b], fma(jb, qt.dgl[b], ry[b]));
    }
    T rx[N];
    if (valid) {
        const T jl = xE[L::xe(ty, tx, k)] - (J ? x[0] : edge_lo<N>(qt, x));
        const T jr = xE[L::xe(ty, tx + 1, k)] - (J ? x[N - 1] : edge_hi<N>(qt, x));
        line_derivative<N>(qt, x, rx);
#pragma unroll
        for (int a = 0; a < N; ++a) rx[a] = fma(jr, -qt.dgl[N - 1 - a], fma(jl, qt.dgl[a], rx[a]));
    }
    if constexpr (WARP) __syncwarp();
    else __syncthreads();

    // ---- phase 4 ---------------------------------------------------------------
    T o[N];
    if (valid) {
        // R (2 / h here holds the velocity, rounded once), then the step: dt and
        // the velocity rounded into one factor would be one more common error.
        // FP32, 100 fixed steps on 48 x 45, mean error against 64 bits of eight
        // states, in 1e-8, p = 1 / 2: 20.5 / 12.2 -> 18.1 / 8.6 without it, 11.8 / 6.9
        // with the operator of N < 4 above (the general tile 12.0 / 9.8).
#pragma unroll
        for (int a = 0; a < N; ++a) o[a] = fma(-A.rhx2, rx[a], -A.rhy2 * sq[L::sq(el, k, a)]);
        T w = mode == MODE_RESIDUAL ? T(1) : T(A.ctrl->dt);
        if (mode == MODE_SO2 || mode == MODE_INC2) w *= T(0.25);
        if (mode == MODE_INC1) {
#pragma unroll
            for (int a = 0; a < N; ++a) o[a] *= w;
        } else if (mode == MODE_SO1) {
#pragma unroll
            for (int a = 0; a < N; ++a) o[a] = fma(w, o[a], x[a]);
        } else if (mode == MODE_SO2 || mode == MODE_SO3) {
            if (sizeof(T) == 8 && mode == MODE_SO3) w *= T(2.0 / 3.0);
            T qn[N];
            gload_row<N>(A.qn + off, qn);
#pragma unroll
            for (int a = 0; a < N; ++a) {
                if (mode == MODE_SO2) o[a] = fma(T(0.75), qn[a], fma(T(0.25), x[a], w * o[a]));
                // FP32: as q + 2/3 ((q2 - q) + dt R), whose weights sum to one
                // (stage_tile_quad)
                else if (sizeof(T) == 4) o[a] = fma(T(2.0 / 3.0), fma(w, o[a], x[a] - qn[a]), qn[a]);
                // (the smaller multiple first: its rounding is the smaller one)
                else o[a] = fma(T(2.0 / 3.0), x[a], fma(T(1.0 / 3.0), qn[a], w * o[a]));
            }
        } else if (addb) {
            T b[N];
            gload_row<N>(A.qb + off, b);
            if (mode == MODE_INC2) {
#pragma unroll
                for (int a = 0; a < N; ++a) o[a] = fma(T(0.25), b[a], w * o[a]);
            } else {
                T hi[N], lo[N];
                gload_row<N>(A.qs + off, hi);
                gload_row<N>(A.lo + off, lo);
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    compensated_add(hi[a], lo[a], T(2.0 / 3.0) * fma(w, o[a], b[a]));
                    o[a] = hi[a];
                }
                gstore_row<N>(A.lo + off, lo);
            }
        }
        gstore_row<N>(A.out + off, o);
    }

    // ---- fused element averages (Algorithm 9) -----------------------------
    if (A.do_avg) {
        if (valid) avS[el * N + k] = line_dot<N>(tb.cavg[k], o);
        __syncthreads();
        if (valid && k == 0) {
            T s = avS[el * N];
#pragma unroll
            for (int b = 1; b < N; ++b) s = s + avS[el * N + b];
            A.avg[e] = s;
        }
    }

    // ---- max signal speed for the next CFL step ------------------------------
    if (A.do_wave) {
        const bool cfl = !(A.ctrl->dt_fixed > 0.0);
        T m = T(0);
        if (cfl && valid) m = point_speed<EQ_ADV>(o, A.ph);
        block_time_update<T>(m, A.ctrl, /*advance=*/true, nslots, cfl);
    }
}

// Tiles: the common one, and for small FP64 grids 4 x 4 elements.
constexpr int adv_tile_x(int p, int k) { return k == 0 ? stage_tile_x(p) : 4; }
constexpr int adv_tile_y(int p, int k) { return k == 0 ? stage_tile_y(p) : 4; }

template <class T, int P, int TX, int TY>
__global__ void __launch_bounds__(stage_threads(TX * TY * (P + 1))) cpr_stage_adv_kernel(const StageArgs<T> A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    stage_tile_adv<T, P, TX, TY>(A, A.tab, A.qx, blockIdx.x, threadIdx.x, smem_raw, gridDim.x);
}

}  // namespace cpr
