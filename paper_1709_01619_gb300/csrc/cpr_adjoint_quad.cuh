// cpr_adjoint_quad.cuh -- the transposed residual of cpr_adjoint.cuh for the
// Euler equations, with the four variables of a point kept together
// (cpr_stage_quad.cuh): out = c0 X0 + c1 X1 + c2 X2 + cv (dR/dq)^T rbar.
//
// Every part of the transpose that is linear in the cotangent alone (the
// transposed line operator M, the edge sums) needs no flux.  So the column
// threads only apply M^T along y and leave the result in shared memory over
// the column of cotangents it came from, and the row threads apply both flux
// Jacobians of a point at once: pressure, velocities and 1 / rho are formed
// once per point instead of once per direction.  The faces on the tile's right
// and upper edge go to threads of their own (as in the stage kernel): in every
// warp's tail they cost a second pass over the face transpose.
//
// Thread (el, k) is row k of element el in phases 1 and 4, column k in phases 2
// and 3 (and row k again for the left faces).
//   1 own rows of q and rbar into the tile copies; edge states, edge
//     cotangents and M^T of the row; halo lines
//   2 column: edge states, edge cotangents, M^T of the column
//   3 face transposes: left and lower face of every element, the tile's
//     right and upper edge
//   4 Jacobians of the row's points, face contributions, epilogue
//
// Against one word per variable and both Jacobians of a point apart, a gradient
// through 20 steps on 256^2 elements, p = 3: 3.72 -> 2.96 ms (60 of these
// launches, and 120 stages).
#pragma once

#include "cpr_adjoint.cuh"
#include "cpr_stage_quad.cuh"

namespace cpr {

template <class T, int N, int TX, int TY>
struct VjpQuadLayout {
    static constexpr int E = TX * TY;
    static constexpr int SQ = E * N * N;          // q
    static constexpr int SR = E * N * N;          // rbar, then M^T along y
    static constexpr int XR = TY * (TX + 1) * N;  // right edge, elements -1..TX-1: states; cotangents
    static constexpr int XH = TY * N;             // left edge of the right halo: state; cotangent
    static constexpr int YT = (TY + 1) * TX * N;
    static constexpr int YH = TX * N;
    static constexpr int EF = E * N;              // per element and line: right face, top face, bottom face
    static constexpr int TOTAL = SQ + SR + 2 * (XR + XH + YT + YH) + 3 * EF;
};

// What the Jacobians of a point need.
template <class T>
struct PointState {
    T ir, u, v, p, m, n, H;  // 1 / rho, velocities, pressure, momenta, e + p
};
template <class T>
__device__ __forceinline__ PointState<T> point_state(const Quad<T>& q, const Phys<T>& ph)
{
    T x[4];
    qget(q, x);
    PointState<T> s;
    s.p = pressure<true>(x, ph.gamma, s.u, s.v, s.ir);
    s.m = x[1];
    s.n = x[2];
    s.H = x[3] + s.p;
    return s;
}

// (dF_DIR/dq)^T w at the state s.  With C = w1 rho u + w2 rho v + w3 H the
// factor of the normal velocity's differential and P = w_n + w3 V_n that of
// the pressure's:
//   dV_n = (-V_n, n_x, n_y, 0) / rho,  dp = (gamma - 1)((u^2 + v^2) / 2, -u, -v, 1).
template <int DIR, class T>
__device__ __forceinline__ Quad<T> jacobian_t(const PointState<T>& s, const Quad<T>& w4, const Phys<T>& ph)
{
    T w[4];
    qget(w4, w);
    const T vn = DIR == 0 ? s.u : s.v;
    const T C = (w[1] * s.m + w[2] * s.n + w[3] * s.H) * s.ir;
    const T G = (ph.gamma - T(1)) * (w[3] * vn + (DIR == 0 ? w[1] : w[2]));
    const T ek = T(0.5) * (s.u * s.u + s.v * s.v);
    const T o0 = G * ek - C * vn;
    const T o1 = vn * w[1] - G * s.u, o2 = vn * w[2] - G * s.v;
    return qmk(o0, DIR == 0 ? o1 + (w[0] + C) : o1, DIR == 1 ? o2 + (w[0] + C) : o2, vn * w[3] + G);
}

// Transpose of Rusanov's flux through a face between the lower state qm and
// the upper state qp (lambda the larger one-sided speed, differentiated on the
// branch that the forward flux takes): the cotangents bm, bp for cotangent w.
template <int DIR, class T>
__device__ __forceinline__ void face_t(const Quad<T>& qm, const Quad<T>& qp, const Quad<T>& w, const Phys<T>& ph,
                                       Quad<T>& bm, Quad<T>& bp)
{
    const PointState<T> a = point_state(qm, ph), b = point_state(qp, ph);
    const T cm = sqrt_of<true>(ph.gamma * a.p * a.ir), cp = sqrt_of<true>(ph.gamma * b.p * b.ir);
    const T va = DIR == 0 ? a.u : a.v, vb = DIR == 0 ? b.u : b.v;
    const T sm = ::fabs(va) + cm, sp = ::fabs(vb) + cp;
    const bool low = sm >= sp;
    const T lam = low ? sm : sp;
    const Quad<T> hw = qmul(w, T(0.5));
    bm = qfma(hw, lam, jacobian_t<DIR>(a, hw, ph));
    bp = qfma(hw, -lam, jacobian_t<DIR>(b, hw, ph));
    // d lambda: -(w, qp - qm) / 2 times the gradient of |V_n| + c at the
    // state that sets lambda
    T h[4], d[4];
    qget(hw, h);
    qget(qsub(qm, qp), d);
    const T t = h[0] * d[0] + h[1] * d[1] + h[2] * d[2] + h[3] * d[3];
    const T ir = low ? a.ir : b.ir, u = low ? a.u : b.u, v = low ? a.v : b.v, p = low ? a.p : b.p;
    const T c = low ? cm : cp, vn = DIR == 0 ? u : v;
    const T g1 = ph.gamma - T(1);
    const T k = T(0.5) * ph.gamma * ir * rcp_of<true>(c);
    const T si = vn >= T(0) ? ir : -ir;
    const T kg = k * g1;
    const Quad<T> gs = qmk(k * (g1 * (T(0.5) * (u * u + v * v)) - p * ir) - si * vn,
                           (DIR == 0 ? si : T(0)) - kg * u, (DIR == 1 ? si : T(0)) - kg * v, kg);
    bm = qfma(gs, low ? t : T(0), bm);
    bp = qfma(gs, low ? T(0) : t, bp);
}

// sum_a c_a x_a over a line of quads.
template <int N, class T>
__device__ __forceinline__ Quad<T> quad_dot(const T* c, const Quad<T> (&x)[N])
{
    Quad<T> s = qmul(x[0], c[0]);
#pragma unroll
    for (int l = 1; l < N; ++l) s = qfma(x[l], c[l], s);
    return s;
}

// Resident CTAs per SM that the registers are sized for (tiles of 32
// elements, no spills).  FP32 p = 3: 5 (96 registers) 1.00, 4 1.04, 6 (80
// registers) 1.06 times the gradient case's time.
template <class T>
constexpr int vjp_quad_min_blocks(int p)
{
    return sizeof(T) == 8 ? 1 : (p == 1 ? 8 : p == 2 ? 7 : p == 3 ? 5 : 4);
}

template <class T, int P, int TX, int TY>
__global__ void __launch_bounds__(TX * TY * (P + 1), vjp_quad_min_blocks<T>(P)) cpr_vjp_quad_kernel(const VjpArgs<T> A)
{
    constexpr int N = P + 1, NN = N * N, NT = TX * TY * N;
    using L = VjpQuadLayout<T, N, TX, TY>;
    using Q = QuadLayout<N, TX, TY>;  // index functions of the tile and edge arrays
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const QuadArr<T, L::SQ> sq{reinterpret_cast<Pr<T>*>(smem_raw)};
    const QuadArr<T, L::SR> sr{sq.end()};
    const QuadArr<T, L::XR> xRq{sr.end()}, xRw{xRq.end()};
    const QuadArr<T, L::XH> xHq{xRw.end()}, xHw{xHq.end()};
    const QuadArr<T, L::YT> yTq{xHw.end()}, yTw{yTq.end()};
    const QuadArr<T, L::YH> yHq{yTw.end()}, yHw{yHq.end()};
    const QuadArr<T, L::EF> xQ{yHw.end()}, yQ{xQ.end()}, yB{yQ.end()};  // right, top, bottom face

    grid_order();
    const int tid = threadIdx.x;
    const int tj = blockIdx.x / A.tiles_x;
    const int i0 = (blockIdx.x - tj * A.tiles_x) * TX, j0 = tj * TY;
    const int TXe = min(TX, A.nx - i0), TYe = min(TY, A.ny - j0);
    const int el = tid / N, k = tid % N;
    const int tx = el % TX, ty = el / TX;
    const bool valid = tx < TXe && ty < TYe;
    const long long e = (long long)(j0 + ty) * A.nx + (i0 + tx);
    const long long off = e * NN + k * N;
    const Tab<T>& tb = A.tab;

    // ---- phase 1 ---------------------------------------------------------------
    Quad<T> x[N], w[N], eL, wL;
    if (valid) {
        load_row_quads<N>(A.q, A.q, false, A.npts, off, x);
        load_row_quads<N>(A.rbar, A.rbar, false, A.npts, off, w);
    }
    {
        constexpr int NXH = 2 * TY * N, LINES = NXH + 2 * TX * N;
        static_assert(LINES <= NT && (TX + TY) * N <= NT, "one halo line or edge face per thread");
        const int t = tid - (NT - LINES);
        if (t >= 0) {
            const bool xdir = t < NXH;
            const int r0 = xdir ? t : t - NXH;
            const int side = r0 >= (xdir ? TY * N : TX * N);
            const int r = side ? r0 - (xdir ? TY * N : TX * N) : r0;
            const int pos = r / N, kk = r % N;
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
                Quad<T> hq[N], hw[N];
                if (xdir) {
                    load_row_quads<N>(A.q, A.q, false, A.npts, eh + kk * N, hq);
                    load_row_quads<N>(A.rbar, A.rbar, false, A.npts, eh + kk * N, hw);
                } else {
                    load_col_quads<N>(A.q, A.q, false, A.npts, eh + kk, hq);
                    load_col_quads<N>(A.rbar, A.rbar, false, A.npts, eh + kk, hw);
                }
                // the edge facing the tile: right / top edge of the lower
                // halo, left / bottom edge of the upper halo
                const T sc = xdir ? -A.rhx2 : -A.rhy2;
                const Quad<T> dq = side ? quad_dot<N>(tb.lm, hq) : quad_dot<N>(tb.lp, hq);
                const Quad<T> dw = qmul(side ? quad_dot<N>(tb.dgl, hw) : quad_dot<N>(tb.dgr, hw), sc);
                if (xdir) {
                    if (side) {
                        xHq.st(pos * N + kk, dq);
                        xHw.st(pos * N + kk, dw);
                    } else {
                        xRq.st(Q::xr(pos, 0, kk), dq);
                        xRw.st(Q::xr(pos, 0, kk), dw);
                    }
                } else {
                    if (side) {
                        yHq.st(pos * N + kk, dq);
                        yHw.st(pos * N + kk, dw);
                    } else {
                        yTq.st(Q::yt(0, pos, kk), dq);
                        yTw.st(Q::yt(0, pos, kk), dw);
                    }
                }
            }
        }
    }
    Quad<T> fb[N];  // M^T along the row
    if (valid) {
#pragma unroll
        for (int a = 0; a < N; ++a) {
            sq.st(Q::sq(el, k, a), x[a]);
            sr.st(Q::sq(el, k, a), w[a]);
        }
        eL = quad_dot<N>(tb.lm, x);
        xRq.st(Q::xr(ty, tx + 1, k), quad_dot<N>(tb.lp, x));
        wL = qmul(quad_dot<N>(tb.dgl, w), -A.rhx2);
        xRw.st(Q::xr(ty, tx + 1, k), qmul(quad_dot<N>(tb.dgr, w), -A.rhx2));
#pragma unroll
        for (int l = 0; l < N; ++l) fb[l] = qmul(quad_dot<N>(A.MT[l], w), -A.rhx2);
    }
    // the columns of an element are read by its own threads: one warp for
    // even N (see the stage kernel)
    constexpr bool KMAJ = N % 2 == 1;
    if constexpr (!KMAJ && 32 % N == 0) __syncwarp();
    else __syncthreads();

    // ---- phase 2 ---------------------------------------------------------------
    const int elc = KMAJ ? tid % (TX * TY) : el, kc = KMAJ ? tid / (TX * TY) : k;
    const int txc = elc % TX, tyc = elc / TX;
    const bool validc = txc < TXe && tyc < TYe;
    Quad<T> eB, wB;
    if (validc) {
        Quad<T> c[N];
#pragma unroll
        for (int b = 0; b < N; ++b) c[b] = sq.ld(Q::sq(elc, b, kc));
        eB = quad_dot<N>(tb.lm, c);
        yTq.st(Q::yt(tyc + 1, txc, kc), quad_dot<N>(tb.lp, c));
#pragma unroll
        for (int b = 0; b < N; ++b) c[b] = sr.ld(Q::sq(elc, b, kc));
        wB = qmul(quad_dot<N>(tb.dgl, c), -A.rhy2);
        yTw.st(Q::yt(tyc + 1, txc, kc), qmul(quad_dot<N>(tb.dgr, c), -A.rhy2));
#pragma unroll
        for (int l = 0; l < N; ++l) sr.st(Q::sq(elc, l, kc), qmul(quad_dot<N>(A.MT[l], c), -A.rhy2));
    }
    __syncthreads();

    // ---- phase 3 ---------------------------------------------------------------
    // A face's cotangent is the sum of both sides'; its lower state's
    // cotangent goes to the lower element's slot.
    Quad<T> own;  // left face: the element's own state
    if (valid) {
        const bool wall = A.bcx && i0 + tx == 0;
        Quad<T> qm = eL, W = wL, bm;
        if (!wall) {
            qm = xRq.ld(Q::xr(ty, tx, k));
            W = qadd(W, xRw.ld(Q::xr(ty, tx, k)));
        }
        face_t<0>(qm, eL, W, A.ph, bm, own);
        if (wall) own = qadd(own, bm);
        if (tx > 0) xQ.st(Q::ef(el - 1, k), bm);
    }
    if (validc) {
        const bool wall = A.bcy && j0 + tyc == 0;
        Quad<T> qm = eB, W = wB, bm, bp;
        if (!wall) {
            qm = yTq.ld(Q::yt(tyc, txc, kc));
            W = qadd(W, yTw.ld(Q::yt(tyc, txc, kc)));
        }
        face_t<1>(qm, eB, W, A.ph, bm, bp);
        yB.st(Q::ef(elc, kc), wall ? qadd(bp, bm) : bp);
        if (tyc > 0) yQ.st(Q::ef(elc - TX, kc), bm);
    }
    if (tid < (TX + TY) * N) {
        // right face of the tile's last column (x) / upper face of its last row
        const bool xe = tid < TY * N;
        const int r = xe ? tid : tid - TY * N;
        const int pos = r / N, kk = r % N;
        if (pos < (xe ? TYe : TXe)) {
            const bool wall = xe ? (A.bcx && i0 + TXe == A.nx) : (A.bcy && j0 + TYe == A.ny);
            const Quad<T> qm = xe ? xRq.ld(Q::xr(pos, TXe, kk)) : yTq.ld(Q::yt(TYe, pos, kk));
            Quad<T> W = xe ? xRw.ld(Q::xr(pos, TXe, kk)) : yTw.ld(Q::yt(TYe, pos, kk));
            Quad<T> qp = qm, bm, bp;
            if (!wall) {
                qp = xe ? xHq.ld(pos * N + kk) : yHq.ld(pos * N + kk);
                W = qadd(W, xe ? xHw.ld(pos * N + kk) : yHw.ld(pos * N + kk));
            }
            if (xe) face_t<0>(qm, qp, W, A.ph, bm, bp);
            else face_t<1>(qm, qp, W, A.ph, bm, bp);
            if (wall) bm = qadd(bm, bp);
            if (xe) xQ.st(Q::ef(pos * TX + TXe - 1, kk), bm);
            else yQ.st(Q::ef((TYe - 1) * TX + pos, kk), bm);
        }
    }
    __syncthreads();

    // ---- phase 4 ---------------------------------------------------------------
    if (valid) {
        T lmk = tb.lm[0], lpk = tb.lp[0];  // by selects instead of indexed parameter loads
#pragma unroll
        for (int b = 1; b < N; ++b) {
            lmk = k == b ? tb.lm[b] : lmk;
            lpk = k == b ? tb.lp[b] : lpk;
        }
        const Quad<T> right = xQ.ld(Q::ef(el, k));
        T o[4][N];
#pragma unroll
        for (int a = 0; a < N; ++a) {
            const PointState<T> s = point_state(sq.ld(Q::sq(el, k, a)), A.ph);
            Quad<T> y = qadd(jacobian_t<0>(s, fb[a], A.ph), jacobian_t<1>(s, sr.ld(Q::sq(el, k, a)), A.ph));
            y = qfma(own, tb.lm[a], y);
            y = qfma(right, tb.lp[a], y);
            y = qfma(yB.ld(Q::ef(el, a)), lmk, y);
            y = qmul(qfma(yQ.ld(Q::ef(el, a)), lpk, y), A.cv);
            T r[4];
            qget(y, r);
#pragma unroll
            for (int v = 0; v < 4; ++v) o[v][a] = r[v];
        }
        auto add = [&](const T* X, T c) {
            if (!X) return;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                T z[N];
                gload_row<N>(X + v * A.npts + off, z);
#pragma unroll
                for (int a = 0; a < N; ++a) o[v][a] = fma(c, z[a], o[v][a]);
            }
        };
        add(A.X0, A.c0);
        add(A.X1, A.c1);
        add(A.X2, A.c2);
#pragma unroll
        for (int v = 0; v < 4; ++v) gstore_row<N>(A.out + v * A.npts + off, o[v]);
    }
}

}  // namespace cpr
