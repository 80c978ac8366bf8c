// cpr_stage_quad.cuh -- the tile of the fused residual + SSP-RK3 stage for the
// FP32 Euler equations (the scheme and its stage modes: cpr_stage.cuh).
//
// The four variables of a point are kept together: shared memory holds one
// 16-byte quad (rho, rho u, rho v, e) per point, edge state, edge flux or
// jump, so that each of them is one 16-byte access instead of four words, and
// the line operators run on pairs of variables (packed FP32 instructions)
// with a table entry broadcast to both lanes: no lane is padding for any
// order and no sum runs across lanes.
//
// Against the same phases with one word per variable (thread instructions per
// thread of the first increment stage: p = 2 1185 -> 695, p = 3 1080 -> 848,
// p = 4 1450 -> 961), per pass, and with the later changes noted below: 1024^2
// p = 3 5.27 -> 4.51 -> 4.32 ms (8 steps), 1365 x 1363 p = 2 5.67 -> 4.70 -> 4.58
// ms (6 steps), 821 x 819 p = 4 5.64 -> 5.03 -> 4.91 ms (6 steps), 128^2 p = 3
// 1.34 -> 1.11 -> 1.07 ms (64 steps, L2-resident).  Bound: at 1024^2 HBM in the
// second and third stage (5.2 TB/s moved); for odd N the L1 / shared-memory data
// pipe (80 % busy for N = 3); on grids that fit the device at once latency.
#pragma once

#include "cpr_common.cuh"
#include "cpr_reduce.cuh"

namespace cpr {

template <class T>
struct alignas(16) Quad {
    Pr<T> a, b;  // (rho, rho u), (rho v, e)
};

template <class T>
__device__ __forceinline__ Quad<T> qmk(T x, T y, T z, T w) { return {pmk(x, y), pmk(z, w)}; }
template <class T>
__device__ __forceinline__ Quad<T> qmul(const Quad<T>& x, T c) { return {pmul(pbc(c), x.a), pmul(pbc(c), x.b)}; }
template <class T>
__device__ __forceinline__ Quad<T> qfma(const Quad<T>& x, T c, const Quad<T>& y)
{
    return {pfma(pbc(c), x.a, y.a), pfma(pbc(c), x.b, y.b)};
}
template <class T>
__device__ __forceinline__ Quad<T> qadd(const Quad<T>& x, const Quad<T>& y) { return {padd(x.a, y.a), padd(x.b, y.b)}; }
template <class T>
__device__ __forceinline__ Quad<T> qsub(const Quad<T>& x, const Quad<T>& y) { return {psub(x.a, y.a), psub(x.b, y.b)}; }
template <class T>
__device__ __forceinline__ void qget(const Quad<T>& x, T* v)
{
    v[0] = x.a.v.x;
    v[1] = x.a.v.y;
    v[2] = x.b.v.x;
    v[3] = x.b.v.y;
}
template <class T>
__device__ __forceinline__ Quad<T> qput(const T* v) { return qmk(v[0], v[1], v[2], v[3]); }

// The same on a single variable.
template <class T>
__device__ __forceinline__ T qmul(T x, T c) { return c * x; }
template <class T>
__device__ __forceinline__ T qfma(T x, T c, T y) { return fma(c, x, y); }
template <class T>
__device__ __forceinline__ T qadd(T x, T y) { return x + y; }
template <class T>
__device__ __forceinline__ T qsub(T x, T y) { return x - y; }

// Edge states of a line of N quads (or of N values of one variable) at -1 (lo) and +1 (hi).  The solution
// points are symmetric, so l_l(+1) = l_{N-1-l}(-1): one table serves both.
// Every edge state of the kernel, the element's own and the one a neighbour
// CTA forms from its halo line, is one of these two sums in this order.
template <int N, class T, class X>
__device__ __forceinline__ X edge_lo(const QuadTab<T>& t, const X (&x)[N])
{
    X s = qmul(x[0], t.lm[0]);
#pragma unroll
    for (int l = 1; l < N; ++l) s = qfma(x[l], t.lm[l], s);
    return s;
}
template <int N, class T, class X>
__device__ __forceinline__ X edge_hi(const QuadTab<T>& t, const X (&x)[N])
{
    X s = qmul(x[N - 1], t.lm[0]);
#pragma unroll
    for (int l = 1; l < N; ++l) s = qfma(x[N - 1 - l], t.lm[l], s);
    return s;
}

// A line operator with the mirror symmetry of the points applied to a line:
// the derivative of the interpolant, or the one of the LP divergence below.
// Its rows sum to zero, so it is a combination of the N - 1 differences of
// neighbouring values (exact for values within a factor of two, where the
// plain row sum rounds every product of an O(1) value); and it changes sign
// under the mirror image of the line, so sums and differences of mirrored
// differences serve two points at once: 8 / 13 / 22 operations per pair of
// variables for N = 3 / 4 / 5 against 9 / 16 / 25 of the row sums.
//
// LP divergence: sum_l D_al f_l + (F*_L - f_L) g_L'_a + (F*_R - f_R) g_R'_a with
// the interpolated edge fluxes f_L = sum_l l_l(-1) f_l, f_R likewise.  Written
// with f_0 and f_{N-1} in place of f_L and f_R, the rest of the edge terms
// joins the matrix,
//   D'_al = D_al + (delta_l0 - l_l(-1)) g_L'_a + (delta_l,N-1 - l_l(+1)) g_R'_a,
// which keeps both properties (the l(+-1) sum to one).  So no edge flux is
// interpolated, N / 2 operations per point and pair of variables, and their
// rounding is gone.  FP32 with N >= 4 (1024^2 p = 3 4.50 -> 4.46 ms for 8 steps,
// 128^2 1.115 -> 1.104 ms for 64; error against 64 bits 5.3e-8 -> 4.5e-8 and
// 1.1e-7 -> 9e-8); for N = 3, where the registers are full, it spills (1365 x
// 1363 4.73 -> 4.77 ms).
template <int N, class T, class X>
__device__ __forceinline__ void line_derivative(const QuadTab<T>& t, const X (&f)[N], X (&r)[N])
{
    constexpr int M = N - 1, H = M / 2;
    X s[H > 0 ? H : 1], d[H > 0 ? H : 1], mid;
#pragma unroll
    for (int m = 0; m < H; ++m) {
        const X lo = qsub(f[m + 1], f[m]), hi = qsub(f[N - 1 - m], f[N - 2 - m]);
        s[m] = qadd(lo, hi);
        d[m] = qsub(lo, hi);
    }
    if constexpr (M % 2 == 1) mid = qsub(f[H + 1], f[H]);
#pragma unroll
    for (int a = 0; a < (N + 1) / 2; ++a) {
        X p;
        if constexpr (M % 2 == 1) {
            p = qmul(mid, t.cm[a]);
#pragma unroll
            for (int m = 0; m < H; ++m) p = qfma(s[m], t.ce[a][m], p);
        } else {
            p = qmul(s[0], t.ce[a][0]);
#pragma unroll
            for (int m = 1; m < H; ++m) p = qfma(s[m], t.ce[a][m], p);
        }
        if (2 * a == N - 1) {
            r[a] = p;
        } else {
            X lo = p, hi = p;
#pragma unroll
            for (int m = 0; m < H; ++m) {
                lo = qfma(d[m], t.co[a][m], lo);
                hi = qfma(d[m], -t.co[a][m], hi);
            }
            r[a] = lo;
            r[N - 1 - a] = hi;
        }
    }
}

// S quads in shared memory.  Every access is of 16 bytes: a whole FP32 quad,
// or one of the two pairs of an FP64 quad, which lie in planes of their own so
// that both types meet the same banks.
template <class T, int S>
struct QuadArr {
    Pr<T>* p;
    __device__ __forceinline__ Quad<T> ld(int i) const
    {
        if constexpr (sizeof(T) == 4) return reinterpret_cast<const Quad<T>*>(p)[i];
        else return {p[i], p[S + i]};
    }
    __device__ __forceinline__ void st(int i, const Quad<T>& x) const
    {
        if constexpr (sizeof(T) == 4) {
            reinterpret_cast<Quad<T>*>(p)[i] = x;
        } else {
            p[i] = x.a;
            p[S + i] = x.b;
        }
    }
    __device__ __forceinline__ Pr<T>* end() const { return p + 2 * S; }
};

// Shared memory of a tile, in quads.
template <int N, int TX, int TY>
struct QuadLayout {
    static constexpr int NN = N * N, E = TX * TY;
    static constexpr int SQ = E * NN;             // tile copy of the stage input, then the y-part of the residual
    static constexpr int XR = TY * (TX + 1) * N;  // right edge states, elements -1..TX-1
    static constexpr int XH = TY * N;             // left edge states of the right halo
    static constexpr int XF = E * N;              // right edge fluxes, then the right jumps
    static constexpr int YT = (TY + 1) * TX * N;  // top edge states, elements -1..TY-1
    static constexpr int YH = TX * N;             // bottom edge states of the upper halo
    static constexpr int YF = E * N;              // top edge fluxes, then the top jumps
    static constexpr int TOTAL = SQ + XR + XH + XF + YT + YH + YF;
    // Point (b, a) of element el.  A quarter warp's accesses (eight threads,
    // 16 bytes each) must hit distinct 16-byte columns of the 128-byte bank
    // row, for the rows (thread = row b, one store per a) and for the columns
    // (thread = column a, one load per b).  N = 4: eight threads hold two
    // elements; XOR of the row into the column and of the element's parity
    // into the row.  N = 2: four elements.  N = 3, 5: the odd element stride
    // does it for the rows, and for the columns when a warp holds one column
    // of consecutive elements (the k-major identity of phase 2).
    __device__ static int sq(int el, int b, int a)
    {
        if constexpr (N == 4) return el * 16 + ((b ^ (el & 1)) << 2) + (a ^ b);
        else if constexpr (N == 2) return el * 4 + ((b * 2 + a) ^ (((el >> 1) & 1) * 3));
        else return el * NN + b * N + a;
    }
    __device__ static int xr(int ty, int f, int k) { return (ty * (TX + 1) + f) * N + k; }
    __device__ static int yt(int g, int tx, int k) { return (g * TX + tx) * N + k; }
    __device__ static int ef(int el, int k) { return el * N + k; }
};

// Row of N values of every variable (point offset off) as quads; addb adds
// the increment array.
template <int N, class T>
__device__ __forceinline__ void load_row_quads(const T* __restrict__ q, const T* __restrict__ qb, bool addb,
                                               long long npts, long long off, Quad<T> (&x)[N])
{
    T r[4][N];
#pragma unroll
    for (int v = 0; v < 4; ++v) gload_row<N>(q + v * npts + off, r[v]);
    if (addb) {
        T b[4][N];
#pragma unroll
        for (int v = 0; v < 4; ++v) gload_row<N>(qb + v * npts + off, b[v]);
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int a = 0; a < N; ++a) r[v][a] += b[v][a];
    }
#pragma unroll
    for (int a = 0; a < N; ++a) x[a] = qmk(r[0][a], r[1][a], r[2][a], r[3][a]);
}

// Column of N values (stride N) of every variable as quads.
template <int N, class T>
__device__ __forceinline__ void load_col_quads(const T* __restrict__ q, const T* __restrict__ qb, bool addb,
                                               long long npts, long long off, Quad<T> (&x)[N])
{
    T r[4][N];
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int l = 0; l < N; ++l) r[v][l] = q[v * npts + off + l * N];
    if (addb) {
        T b[4][N];
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int l = 0; l < N; ++l) b[v][l] = qb[v * npts + off + l * N];
#pragma unroll
        for (int v = 0; v < 4; ++v)
#pragma unroll
            for (int l = 0; l < N; ++l) r[v][l] += b[v][l];
    }
#pragma unroll
    for (int a = 0; a < N; ++a) x[a] = qmk(r[0][a], r[1][a], r[2][a], r[3][a]);
}

// Flux of Eq. 4 through DIR at one point; SPEED: also the signal speed
// |Vn| + c.  FP32: the mass flux is rho Vn with the rounded velocity that the
// momentum and energy fluxes carry, not the momentum itself.  Errors against 64
// bits, mean of eight vortex states, with the momentum -> this way, in 1e-8: 60
// fixed steps p = 1 to 4 6.0 / 8.1 / 8.1 / 8.8 -> 5.7 / 7.7 / 7.0 / 7.6, p = 1 with
// Lobatto points and chain rule 8.0 -> 7.6; FV, 40 steps, second / third order,
// 23.7 / 6.1 -> 23.0 / 5.7.  No dearer: 1024^2 p = 3 4.39 -> 4.34 ms.
template <int DIR, bool SPEED = false, class T>
__device__ __forceinline__ Quad<T> quad_flux(const Quad<T>& q, const Phys<T>& ph, T* s = nullptr)
{
    T v[4], u, w, r;
    qget(q, v);
    const T p = pressure<true>(v, ph.gamma, u, w, r);
    const T vn = DIR == 0 ? u : w;
    if constexpr (SPEED) *s = ::fabs(vn) + sqrt_of<true>(ph.gamma * p * r);
    const T h = (v[3] + p) * vn, m = sizeof(T) == 4 ? v[0] * vn : v[DIR + 1];
    if constexpr (DIR == 0) return qmk(m, fma(v[1], u, p), v[2] * u, h);
    else return qmk(m, v[1] * w, fma(v[2], w, p), h);
}

// Both fluxes of Eq. 4 at one point (q may be f).
template <class T>
__device__ __forceinline__ void quad_flux_xy(const Quad<T>& q, const Phys<T>& ph, Quad<T>& f, Quad<T>& g)
{
    T v[4];
    qget(q, v);
    const T r = rcp_of<true>(v[0]), u = v[1] * r, w = v[2] * r;
    const T mw = v[1] * w;
    const T p = (ph.gamma - T(1)) * fma(T(-0.5), fma(v[1], u, v[2] * w), v[3]), h = v[3] + p;
    f = qmk(v[1], fma(v[1], u, p), mw, h * u);
    g = qmk(v[2], mw, fma(v[2], w, p), h * w);
}

// Twice the common flux through a face between the lower state m and the
// upper state p (the factor 1/2 joins the jump's subtraction, half_jump).
template <int FLUX, int DIR, class T>
__device__ __forceinline__ Quad<T> quad_face2(const Quad<T>& m, const Quad<T>& p, const Phys<T>& ph)
{
    if constexpr (FLUX == FLUX_RUSANOV) {
        T sm, sp;
        const Quad<T> fm = quad_flux<DIR, true>(m, ph, &sm), fp = quad_flux<DIR, true>(p, ph, &sp);
        const T lam = sm >= sp ? sm : sp;
        return qfma(qsub(m, p), lam, qadd(fm, fp));
    } else {
        T a[4], b[4], F[4];
        qget(m, a);
        qget(p, b);
        roe_flux<DIR, true>(a, b, ph, F);
        return qmul(qput(F), T(2));
    }
}
// F* - f from twice the common flux.
template <class T>
__device__ __forceinline__ Quad<T> half_jump(const Quad<T>& G2, const Quad<T>& f)
{
    return {pfma(G2.a, pbc(T(0.5)), pmul(f.a, pbc(T(-1)))), pfma(G2.b, pbc(T(0.5)), pmul(f.b, pbc(T(-1))))};
}

// x-line or y-line of one thread: line operator r, edge states lo, hi and the
// fluxes flo, fhi that the common fluxes are compared with (joined operator:
// those of the first and last point; else of the edges) of the line x
// (consumed).
template <int N, int DIR, int DIV, class T>
__device__ __forceinline__ void quad_line(const QuadTab<T>& t, const Phys<T>& ph, Quad<T> (&x)[N], Quad<T> (&r)[N],
                                          Quad<T>& lo, Quad<T>& hi, Quad<T>& flo, Quad<T>& fhi)
{
    lo = edge_lo<N>(t, x);
    hi = edge_hi<N>(t, x);
    if constexpr (DIV == DIV_LP) {
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = quad_flux<DIR>(x[a], ph);
        if constexpr (quad_joined<T>(N)) {
            flo = x[0];
            fhi = x[N - 1];
        } else {
            flo = edge_lo<N>(t, x);
            fhi = edge_hi<N>(t, x);
        }
        line_derivative<N>(t, x, r);
    } else {
        Quad<T> dq[N];
        line_derivative<N>(t, x, dq);
#pragma unroll
        for (int a = 0; a < N; ++a) {
            T q[4], d[4], o[4];
            qget(x[a], q);
            qget(dq[a], d);
            flux_jvp<EQ_EULER, DIR, true>(q, d, ph, o);
            r[a] = qput(o);
        }
        flo = quad_flux<DIR>(lo, ph);
        fhi = quad_flux<DIR>(hi, ph);
    }
}

// One tile of a stage update (modes 1-6): the work of one CTA (the tile
// index, the idle threads and nslots: stage_tile of cpr_stage.cuh).  MODE: the
// stage mode, or 0 for the one in the arguments.
//
// Thread (el, k) is row k of element el in phases 1 and 4 and a column of an
// element in phases 2 and 3.
//   1 halo lines (edge states of the neighbour elements facing the tile, one
//     line of all variables per thread), own row: into the tile copy, x-line
//   2 column from the tile copy: y-line
//   3 common flux on the element's left and lower face points, one evaluation
//     per face point (the tile's right / upper edge faces go to threads of
//     their own), and the jumps F* - f of both elements: the neighbour's over
//     its edge flux, the own lower one into the y-derivative, which goes over
//     the dead tile copy
//   4 row k: corrections, stage update, store; averages, CFL maximum
template <int P, int DIV, int FLUX, int TX, int TY, bool PF, int MODE>
__device__ __forceinline__ void stage_tile_quad(const StageArgs<float>& A, const Tab<float>& tb, const QuadArgs<float>& qx,
                                                int tile, int tid, unsigned char* smem_raw, int nslots)
{
    constexpr int N = P + 1, NN = N * N;
    constexpr int NT = TX * TY * N;
    using L = QuadLayout<N, TX, TY>;
    Quad<float>* sq = reinterpret_cast<Quad<float>*>(smem_raw);
    Quad<float>* xR = sq + L::SQ;
    Quad<float>* xH = xR + L::XR;
    Quad<float>* xF = xH + L::XH;
    Quad<float>* yT = xF + L::XF;
    Quad<float>* yH = yT + L::YT;
    Quad<float>* yF = yH + L::YH;
    Quad<float>* avS = xR;  // row partial sums of the averages, over the edge states after phase 3
    static_assert(L::XR >= TX * TY * N, "the partial sums of the averages fit the right edge states");

    const int mode = MODE > 0 ? MODE : A.mode;
    // t_end reached (uniform over the grid): tested after the first barrier,
    // so that the flag's load and the state's are under way together (nothing
    // is written to global memory before): 128^2 p = 3 1.103 -> 1.066 ms for 64
    // steps, 1024^2 4.488 -> 4.410 ms for 8; the FP64 and advection tiles and the
    // limiter did not gain
    const int done = A.ctrl->done;

    const bool active = tid < NT;
    const QuadTab<float>& qt = qx.tab;
    const int tj = (int)div_invariant((unsigned)tile, (unsigned)A.tiles_x, A.qx.tx_magic, A.qx.tx_shift);
    const int i0 = (tile - tj * A.tiles_x) * TX;
    const int j0 = tj * TY;
    const int TXe = min(TX, A.nx - i0), TYe = min(TY, A.ny - j0);
    const int el = tid / N, k = tid % N;
    const int tx = el % TX, ty = el / TX;
    const bool valid = active && tx < TXe && ty < TYe;
    const long long e = (long long)(j0 + ty) * A.nx + (i0 + tx);
    const long long off = e * NN + k * N;
    const bool addb = mode == MODE_INC2 || mode == MODE_INC3;
    const bool lwall = A.bcx && i0 + tx == 0;

    // ---- phase 1: halo lines; own row -> tile copy and x-line ---------------
    if (PF && valid && k == 0 && (tx & 1) == 0) {
        // the low part is first read in phase 4, from HBM when the state
        // does not fit in L2: start it towards L2 now, one prefetch per
        // 128-byte line (two elements' rows of one variable)
#pragma unroll
        for (int v = 0; v < 4; ++v) asm volatile("prefetch.global.L2 [%0];" ::"l"(A.lo + v * A.npts + e * NN));
    }
    Quad<float> x[N], rx[N], eL, fL;
    if (valid) load_row_quads<N>(A.qs, A.qb, addb, A.npts, off, x);
    {
        constexpr int NXH = 2 * TY * N, LINES = NXH + 2 * TX * N;
        static_assert(LINES <= NT, "at most one halo line per thread");
        const int t = tid - (NT - LINES);
        if (active && t >= 0) {
            const bool xdir = t < NXH;
            const int r0 = xdir ? t : t - NXH;
            const int side = r0 >= (xdir ? TY * N : TX * N);
            const int r = side ? r0 - (xdir ? TY * N : TX * N) : r0;
            const int pos = r / N, kk = r % N;  // pos: tile row (x) or tile column (y)
            int gi = xdir ? (side ? i0 + TXe : i0 - 1) : i0 + pos;
            int gj = xdir ? j0 + pos : (side ? j0 + TYe : j0 - 1);
            bool have = pos < (xdir ? TYe : TXe);
            if (gi < 0 || gi >= A.nx) {
                have = have && !A.bcx;
                gi = gi < 0 ? gi + A.nx : gi - A.nx;
            }
            if (gj < 0 || gj >= A.ny) {
                have = have && !A.bcy;
                gj = gj < 0 ? gj + A.ny : gj - A.ny;
            }
            if (have) {
                const long long eh = ((long long)gj * A.nx + gi) * NN;
                Quad<float> h[N];
                if (xdir) load_row_quads<N>(A.qs, A.qb, addb, A.npts, eh + kk * N, h);
                else load_col_quads<N>(A.qs, A.qb, addb, A.npts, eh + kk, h);
                const Quad<float> es = side ? edge_lo<N>(qt, h) : edge_hi<N>(qt, h);
                if (xdir) {
                    if (side) xH[pos * N + kk] = es;
                    else xR[L::xr(pos, 0, kk)] = es;
                } else {
                    if (side) yH[pos * N + kk] = es;
                    else yT[L::yt(0, pos, kk)] = es;
                }
            }
        }
    }
    if (valid) {
#pragma unroll
        for (int a = 0; a < N; ++a) sq[L::sq(el, k, a)] = x[a];
        Quad<float> eR, fR;
        quad_line<N, 0, DIV>(qt, A.ph, x, rx, eL, eR, fL, fR);
        xR[L::xr(ty, tx + 1, k)] = eR;
        xF[L::ef(el, k)] = fR;
    }
    // Phase 2 reads only the points of one element from the tile copy.  For
    // even N the column identity is the row identity and a warp holds whole
    // elements, so a warp barrier orders its own rows.  Everything else that
    // phase 1 writes is read after the next CTA barrier.
    constexpr bool KMAJ = N % 2 == 1;
    if constexpr (!KMAJ && 32 % N == 0) __syncwarp();
    else __syncthreads();
    if (done) return;
    // a limited run: clear the marked-element count of the limiter pass
    // that follows this stage (stream order keeps it apart from the last one)
    if (A.do_avg && tile == 0 && tid == 0) A.ctrl->marked = 0;

    // ---- phase 2: y-line (column kc of element elc) --------------------------
    const int elc = KMAJ ? tid % (TX * TY) : el, kc = KMAJ ? tid / (TX * TY) : k;
    const int txc = elc % TX, tyc = elc / TX;
    const bool validc = active && txc < TXe && tyc < TYe;
    const bool bwall = A.bcy && j0 + tyc == 0;
    Quad<float> ry[N], eB, gB;
    if (validc) {
        Quad<float> c[N], eT, gT;
#pragma unroll
        for (int b = 0; b < N; ++b) c[b] = sq[L::sq(elc, b, kc)];
        quad_line<N, 1, DIV>(qt, A.ph, c, ry, eB, eT, gB, gT);
        yT[L::yt(tyc + 1, txc, kc)] = eT;
        yF[L::ef(elc, kc)] = gT;
    }
    __syncthreads();

    // ---- phase 3: common fluxes ----------------------------------------------
    if (validc) {
        // lower face: the jump F* - f of this element into its y-derivative,
        // the neighbour's over its top edge flux
        const Quad<float> dm = bwall ? eB : yT[L::yt(tyc, txc, kc)];
        const Quad<float> G = quad_face2<FLUX, 1>(dm, eB, A.ph);
        const Quad<float> J = half_jump(G, gB);
        if (tyc > 0) {
            Quad<float>* pj = yF + L::ef(elc - TX, kc);
            *pj = half_jump(G, *pj);
        }
#pragma unroll
        for (int b = 0; b < N; ++b) sq[L::sq(elc, b, kc)] = qfma(J, qt.dgl[b], ry[b]);
    }
    Quad<float> JL;
    if (valid) {
        const Quad<float> dm = lwall ? eL : xR[L::xr(ty, tx, k)];
        const Quad<float> G = quad_face2<FLUX, 0>(dm, eL, A.ph);
        JL = half_jump(G, fL);
        if (tx > 0) {
            Quad<float>* pj = xF + L::ef(el - 1, k);
            *pj = half_jump(G, *pj);
        }
    }
    if (tid < (TX + TY) * N) {
        // right face of the tile's last column (x) / upper face of its last row
        const bool xe = tid < TY * N;
        const int r = xe ? tid : tid - TY * N;
        const int pos = r / N, kk = r % N;
        if (pos < (xe ? TYe : TXe)) {
            const bool wall = xe ? (A.bcx && i0 + TXe == A.nx) : (A.bcy && j0 + TYe == A.ny);
            const Quad<float> Em = xe ? xR[L::xr(pos, TXe, kk)] : yT[L::yt(TYe, pos, kk)];
            const Quad<float> dp = wall ? Em : (xe ? xH[pos * N + kk] : yH[pos * N + kk]);
            const Quad<float> G = xe ? quad_face2<FLUX, 0>(Em, dp, A.ph) : quad_face2<FLUX, 1>(Em, dp, A.ph);
            Quad<float>* pj = xe ? xF + L::ef(pos * TX + TXe - 1, kk) : yF + L::ef((TYe - 1) * TX + pos, kk);
            *pj = half_jump(G, *pj);
        }
    }
    __syncthreads();

    // ---- phase 4: R on row k, stage update, store ----------------------------
    float o[4][N];
    if (valid) {
        // g_R'(eta_k) = -g_L'(eta_{N-1-k}): one select chain instead of an
        // indexed parameter load
        float grk = -qt.dgl[N - 1];
#pragma unroll
        for (int b = 1; b < N; ++b) grk = k == b ? -qt.dgl[N - 1 - b] : grk;
        // the factor of R in the stage's result: dt (increment modes: dt / 4
        // and 2 dt / 3 of the second and third stage)
        float w = (float)A.ctrl->dt;
        if (mode == MODE_INC2) w *= 0.25f;
        if (mode == MODE_INC3) w *= 2.0f / 3.0f;
        const float sx = -A.rhx2 * w, sy = -A.rhy2 * w;
        const Quad<float> JR = xF[L::ef(el, k)];
#pragma unroll
        for (int a = 0; a < N; ++a) {
            Quad<float> y = sq[L::sq(el, k, a)];
            y = qfma(yF[L::ef(el, a)], grk, y);
            Quad<float> z = qfma(JL, qt.dgl[a], rx[a]);
            z = qfma(JR, -qt.dgl[N - 1 - a], z);
            float yv[4], zv[4];
            qget(qmul(y, sy), yv);
            qget(z, zv);
#pragma unroll
            for (int v = 0; v < 4; ++v) o[v][a] = fmaf(sx, zv[v], yv[v]);
        }
        if (mode == MODE_INC1) {
        } else if (mode <= MODE_SO3) {
            // q1 = q + dt R, then q + c ((q_i - q) + dt R), c = 1/4, 2/3: one
            // rounding of the state's size (the difference is exact within a
            // factor of two), and weights that sum to one, where 1/3 and 2/3 in FP32 exceed it by
            // 3e-8, a growth of every step (limited runs of 8 steps, error
            // against 64 bits over twelve states: p = 1 1.15e-7 -> 4.9e-8, p = 2
            // 1.14e-7 -> 5.8e-8, p = 3 1.09e-7 -> 7.7e-8)
            const float c = mode == MODE_SO2 ? 0.25f : 2.0f / 3.0f;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                float qs[N], qn[N];
                gload_row<N>(A.qs + v * A.npts + off, qs);
                if (mode == MODE_SO1) {
#pragma unroll
                    for (int a = 0; a < N; ++a) o[v][a] = qs[a] + o[v][a];
                } else {
                    gload_row<N>(A.qn + v * A.npts + off, qn);
#pragma unroll
                    for (int a = 0; a < N; ++a) o[v][a] = fmaf(c, o[v][a] + (qs[a] - qn[a]), qn[a]);
                }
            }
        } else {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                float b[N];
                gload_row<N>(A.qb + v * A.npts + off, b);
                if (mode == MODE_INC2) {
#pragma unroll
                    for (int a = 0; a < N; ++a) o[v][a] = fmaf(0.25f, b[a], o[v][a]);
                } else {
                    float hi[N], lo[N];
                    gload_row<N>(A.qs + v * A.npts + off, hi);
                    gload_row<N>(A.lo + v * A.npts + off, lo);
#pragma unroll
                    for (int a = 0; a < N; ++a) {
                        compensated_add(hi[a], lo[a], fmaf(2.0f / 3.0f, b[a], o[v][a]));
                        o[v][a] = hi[a];
                    }
                    gstore_row<N>(A.lo + v * A.npts + off, lo);
                }
            }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) gstore_row<N>(A.out + v * A.npts + off, o[v]);
    }

    // ---- fused element averages (Algorithm 9) -----------------------------
    if (A.do_avg) {
        if (valid) {
            float s[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) s[v] = line_dot<N>(tb.cavg[k], o[v]);
            avS[L::ef(el, k)] = qput(s);
        }
        __syncthreads();
        const int ax = tid % TX, ay = tid / TX;
        if (tid < TX * TY && ax < TXe && ay < TYe) {
            Quad<float> s = avS[L::ef(tid, 0)];
#pragma unroll
            for (int b = 1; b < N; ++b) s = qadd(s, avS[L::ef(tid, b)]);
            float sv[4];
            qget(s, sv);
            const long long ne = A.npts / NN, ea = (long long)(j0 + ay) * A.nx + (i0 + ax);
#pragma unroll
            for (int v = 0; v < 4; ++v) A.avg[v * ne + ea] = sv[v];
        }
    }

    // ---- fused max signal speed for the next CFL step ---------------------
    // (only CFL runs need the speed; a run of fixed steps only closes the
    // step; the branch is uniform over the grid)
    if (A.do_wave) {
        const bool cfl = !(A.ctrl->dt_fixed > 0.0);
        float m = 0.f;
        if (cfl && valid) {
#pragma unroll
            for (int a = 0; a < N; ++a) {
                const float q[4] = {o[0][a], o[1][a], o[2][a], o[3][a]};
                const float s = point_speed<EQ_EULER, true>(q, A.ph);
                m = s > m ? s : m;
            }
        }
        block_time_update<float>(m, A.ctrl, /*advance=*/true, nslots, cfl);
    }
}

// Resident CTAs per SM of a single problem's kernels.  p = 4: 4 CTAs of 32
// elements (96 registers, no spills) instead of the 6 (64 registers, 56 bytes
// of spills) that batches keep: 821 x 819 p = 4 303 -> 281 us per stage, the
// 64-instance batch 31.5 -> 32.5 ms per 24 steps.  p = 1: 7 CTAs (72 registers,
// which LP with Rusanov's flux takes anyway) for every grid; with the 76 to 85 of
// the other divergences and fluxes, grids around 256^2 need a second round of
// CTAs: Roe 10.6 -> 8.2 us per stage (the general tile 10.1), 768^2 57.7 -> 52.7.
template <int P, bool WIDE, int ELEMS>
constexpr int quad_min_blocks()
{
    return P == 1             ? 7 * 64 / ELEMS
           : P == 4 && !WIDE ? 128 / ELEMS
                             : stage_min_blocks<float, P + 1, WIDE, ELEMS>();
}

// The kernels that the step adjoint launches behind one another: those compiled
// for a Shu-Osher stage.
__host__ __device__ constexpr bool quad_ordered(int mode) { return mode >= MODE_SO1 && mode <= MODE_SO3; }

template <int P, int DIV, int FLUX, int TX, int TY, int MINB, int MODE>
__global__ void __launch_bounds__(TX * TY * (P + 1), MINB) cpr_stage_quad_kernel(const StageArgs<float> A)
{
    static_assert((TX * TY * (P + 1)) % 32 == 0, "whole warps: the warp-level reductions use every lane");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if constexpr (quad_ordered(MODE)) grid_order();
    stage_tile_quad<P, DIV, FLUX, TX, TY, false, MODE>(A, A.tab, A.qx, blockIdx.x, threadIdx.x, smem_raw, gridDim.x);
}

}  // namespace cpr
