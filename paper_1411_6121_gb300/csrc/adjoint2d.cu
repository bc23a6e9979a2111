// adjoint2d.cu -- hand-written discrete adjoint of the 2D (D2Q9) DUGKS step, and the
// checkpointed reverse sweep behind dugks_record / dugks_adjoint.
//
// One step Phi: g~^n -> g~^{n+1} (Appendix steps 1-10 of arXiv 1411.6121 in deviation form,
// as dugks_step.cuh computes it) depends on the acceleration field G(x) and on the wall
// velocities u_w. For lambda' = dL/dg~^{n+1} one reverse step forms
//     lambda = (dPhi/dg~^n)^T lambda',  dL/dG += (dPhi/dG)^T lambda',  dL/du_w += (dPhi/du_w)^T lambda'
// by running the sub-steps backwards in three gather-form kernels:
//   adj_cells_fwd (per cell)       recomputes the cell moments (eq. (27)) and
//                                  fbar+ (step 1, eq. (24));
//   adj_faces_all (per interface)  recomputes steps 3-7 and pulls lambda' back through the
//                                  flux (steps 8-9), the interface relaxation (step 7,
//                                  eq. (20)), the interface moments (step 6) and the
//                                  wall condition (step 5: eq. (32), or eq. (31)), down to the
//                                  adjoint of the step-4 values and of the interface
//                                  acceleration;
//   adj_cells_all (per cell)       transposes the reconstruction (steps 3-4, eq. (23))
//                                  and the ghost extrapolation (step 2), then pulls the
//                                  adjoint of fbar+ back through step 1 and the cell moments
//                                  to g~^n and G; then it makes adj_cells_fwd's work for the
//                                  next reverse step, which leaves adj_cells_fwd to the first
//                                  reverse step of each checkpoint segment.
// The interior of each kernel takes a fast path with compile-time velocities; the band along
// walls, x_c interfaces and periodic seams takes the general path, one item per half-warp with
// one velocity per lane. Every output element is a gather written by one thread, or by one lane
// after a fixed-order butterfly over the velocities (no atomics), so the sweep is bitwise
// reproducible. Arithmetic in the storage type of the handle (float or double). The adjoint
// covers the incompressible model (eq. (6)).
//
// Interfaces: normal to x, (i, j) with i in [0, nx], j in [0, ny), between cells (i-1, j)
// and (i, j), index i + (nx+1) j; normal to y, (i, j) with i in [0, nx), j in [0, ny],
// between (i, j-1) and (i, j), index i + nx j. The forward step evaluates interface 0 and
// interface n of a periodic axis separately (equal values): the first feeds cell 0, the
// second cell n-1, and so they are two interfaces here as well.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <vector>

#include "../../include/dugks.h"
#include "dugks_internal.h"
#include "handle.h"

namespace dugks {

namespace {

constexpr int Q = 9;
using L9 = Lat<9>;

template <class T>
struct AdjParams {
    int n[2];                // nx, ny
    int per[2];              // periodic along x / y
    int64_t px, dstride;     // layout of the stored state (row pitch, direction stride)
    int bc[4];               // DUGKS_BC_* of the faces -x, +x, -y, +y
    T mw[4][2];              // wall momentum rho0 u_w / c of a velocity condition
    T drw[4];                // rho_a - rho0 = p_w / RT of a pressure condition
    T drw1[4];               // its oscillating part: + drw1 cos(omega (t_n + h))
    T rho0, inv_rho0, dmw;   // dmw = d m_w / d u_w = rho0 / c
    T b1, c1, b7, c7, kappa, two_kappa, wcell, wface;
    T g[2];                  // uniform acceleration
    const float *field;      // [2][ncell] acceleration field or null
    T ctc, cthc;             // cos(omega t_n) / c and cos(omega (t_n + h)) / c
    T cwh;                   // cos(omega (t_n + h))
    const T *state;          // g~^n (padded layout)
    T *phi;                  // [Q][ncell] fbar+ of the cells
    T *mom;                  // [3][ncell] drho, m_x, m_y of the cells (m in units of c)
    const T *nstate;         // g~^{n-1} for the next reverse step's recompute, or null
    T nctc;                  // cos(omega t_{n-1}) / c
    T *nmom;                 // its cell moments (the other moments buffer)
    const T *lam1;           // lambda' [Q][ncell]
    T *fb[2];                // adjoint of the step-4 values [Q][nface_d]
    T *gb[2];                // adjoint of the interface acceleration Gh [2][nface_d]
    T *lam0;                 // lambda [Q][ncell]
    double *dG;              // [2][ncell] dL/dfield accumulator (null: not wanted)
    double *dW;              // [2 (ny + nx)][2] dL/du_w accumulator per wall interface
};

template <class T>
__device__ __forceinline__ int64_t ncell(const AdjParams<T> &a) {
    return (int64_t)a.n[0] * a.n[1];
}
template <class T>
__device__ __forceinline__ int64_t nface(const AdjParams<T> &a, int d) {
    return d == 0 ? (int64_t)(a.n[0] + 1) * a.n[1] : (int64_t)a.n[0] * (a.n[1] + 1);
}
template <class T>
__device__ __forceinline__ int64_t fidx(const AdjParams<T> &a, int d, int i, int j) {
    return d == 0 ? i + (int64_t)(a.n[0] + 1) * j : i + (int64_t)a.n[0] * j;
}

// ---- step 2: extended positions -1 .. n along one axis (reading R3: ghost = 2 f(0) - f(1)
// at a wall, the periodic image otherwise), as two cells and their weights (the second 0 where the
// position is a real cell or an image): branch-free, so the loads of an item are all in flight
// together ----
template <class T>
__device__ __forceinline__ void ext2(int x, int n, int per, int c[2], T w[2]) {
    const bool lo = x < 0, out = lo || x >= n, wall = out && !per;
    c[0] = wall ? (lo ? 0 : n - 1) : (out ? (lo ? n - 1 : 0) : x);
    c[1] = wall ? (lo ? 1 : n - 2) : c[0];
    w[0] = wall ? T(2) : T(1);
    w[1] = wall ? T(-1) : T(0);
}

// ---- equilibrium (eq. (6), deviation form, m = rho0 u / c) ----
template <class T>
__device__ __forceinline__ T geq(const AdjParams<T> &a, int k, T dr, const T m[2]) {
    const T em = (T)L9::e(k, 0) * m[0] + (T)L9::e(k, 1) * m[1];
    const T mm = m[0] * m[0] + m[1] * m[1];
    return L9::wt<T>(k) * (dr + T(3) * em + (T(4.5) * em * em - T(1.5) * mm) * a.inv_rho0);
}

// Moments of a distribution with the force weight w (dt/2 at cells, h/2 at interfaces).
template <class T>
__device__ __forceinline__ void moments2(const AdjParams<T> &a, const T f[Q], const T Gh[2], T w, T &dr, T m[2]) {
    dr = T(0);
    m[0] = m[1] = T(0);
    for (int k = 0; k < Q; k++) {
        dr += f[k];
        m[0] += (T)L9::e(k, 0) * f[k];
        m[1] += (T)L9::e(k, 1) * f[k];
    }
    m[0] += a.rho0 * Gh[0] * w;
    m[1] += a.rho0 * Gh[1] * w;
}

// ---- the general path, velocity-parallel: one half-warp per item of the boundary frame,
// lane k of the half (k < Q) holding velocity k and lanes k >= Q zeros. Sums over the
// velocities are butterflies over the half-warp: every lane ends with the same bits and the
// order is fixed. The two halves of a warp work on different items and may diverge, so the
// shuffles name only their own half. ----
__device__ __forceinline__ int half_lane() { return threadIdx.x & 15; }
template <class T>
__device__ __forceinline__ T wsum(T v) {
    const unsigned m = 0xffffu << (threadIdx.x & 16);
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) v += __shfl_xor_sync(m, v, o, 16);
    return v;
}

// The lane's velocity: k < Q, lanes beyond it repeat velocity 0 and take part with zeros.
template <class T>
struct LaneVel {
    int k, ie[2];
    bool act;
    T e[2], W;
    __device__ __forceinline__ LaneVel() {
        const int lane = half_lane();
        act = lane < Q;
        k = act ? lane : 0;
        ie[0] = k / 3 - 1;
        ie[1] = k - 3 * (k / 3) - 1;
        e[0] = (T)ie[0];
        e[1] = (T)ie[1];
        W = ie[0] && ie[1] ? T(1) / T(36) : (ie[0] || ie[1] ? T(1) / T(9) : T(4) / T(9));
    }
};
template <class T>
__device__ __forceinline__ T geq_lane(const LaneVel<T> &l, T inv_rho0, T dr, const T m[2]) {
    const T em = l.e[0] * m[0] + l.e[1] * m[1], mm = m[0] * m[0] + m[1] * m[1];
    return l.W * (dr + T(3) * em + (T(4.5) * em * em - T(1.5) * mm) * inv_rho0);
}
template <class T>
__device__ __forceinline__ void geq_dm_lane(const LaneVel<T> &l, T inv_rho0, const T m[2], T out[2]) {
    const T em9 = T(9) * (l.e[0] * m[0] + l.e[1] * m[1]);
#pragma unroll
    for (int c = 0; c < 2; c++) out[c] = l.W * (T(3) * l.e[c] + (em9 * l.e[c] - T(3) * m[c]) * inv_rho0);
}

// Relaxation P_k = f_k + b (geq_k - f_k) + c S_k with S_k = 3 (Gh.e_k - Gh.m/rho0) f_eq,k
// (steps 1 and 7). Given the weight w = dL/dP_k of the lane's velocity, dL/d(drho), dL/dm and dL/dGh
// through the moment dependence (the direct part (1 - b) w is left to the caller), summed over
// the velocities.
template <class T>
__device__ __forceinline__ void relax_T_lane(const AdjParams<T> &a, const LaneVel<T> &l, T w, T dr, const T m[2],
                                             const T Gh[2], T b, T c, T &bdr, T bm[2], T bG[2]) {
    const T gm = (Gh[0] * m[0] + Gh[1] * m[1]) * a.inv_rho0;
    const T s = T(3) * (Gh[0] * l.e[0] + Gh[1] * l.e[1] - gm);
    const T feq = l.W * a.rho0 + geq_lane(l, a.inv_rho0, dr, m);
    T dg[2];
    geq_dm_lane(l, a.inv_rho0, m, dg);
    const T cw = w * (b + c * s), fq = w * c * T(3) * feq;  // w dP/dgeq
    bdr = wsum(cw * l.W);
#pragma unroll
    for (int i = 0; i < 2; i++) {
        bm[i] = wsum(cw * dg[i] - fq * (Gh[i] * a.inv_rho0));
        bG[i] = wsum(fq * (l.e[i] - m[i] * a.inv_rho0));
    }
}

// ---- acceleration at cells and interfaces (reading R2) ----
template <class T>
__device__ __forceinline__ T field_at(const AdjParams<T> &a, int comp, int x, int y) {
    return a.field ? (T)a.field[comp * ncell(a) + x + (int64_t)a.n[0] * y] : T(0);
}
template <class T>
__device__ __forceinline__ void cell_Gh(const AdjParams<T> &a, int x, int y, T Gh[2]) {
    for (int c = 0; c < 2; c++) Gh[c] = (a.g[c] + field_at(a, c, x, y)) * a.ctc;
}
// ---- fast paths: interfaces and cells whose stencils lie inside the domain, away from
// walls and periodic seams (no ghosts, images, NEQ or x_c coupling). Same arithmetic as the
// general path, with compile-time velocities and direct neighbour reads. ----

// relax_T with a compile-time velocity loop; D >= 0 restricts it to the velocities that
// cross an interface normal to axis D (the others have zero weight there).
template <class T, int D>
__device__ __forceinline__ void relax_T_c(const AdjParams<T> &a, const T wk[Q], T dr, const T m[2], const T Gh[2],
                                          T b, T c, T &bdr, T bm[2], T bG[2]) {
    const T gm = (Gh[0] * m[0] + Gh[1] * m[1]) * a.inv_rho0;
    const T mm = m[0] * m[0] + m[1] * m[1];
    sfor<Q>([&](auto kc) {
        constexpr int k = kc;
        constexpr int e0 = L9::e(k, 0), e1 = L9::e(k, 1);
        if constexpr (D < 0 || L9::e(k, D < 0 ? 0 : D) != 0) {
            const T W = L9::wt<T>(k);
            const T em = T(e0) * m[0] + T(e1) * m[1];
            const T s = T(3) * (Gh[0] * T(e0) + Gh[1] * T(e1) - gm);
            const T feq = W * a.rho0 + W * (dr + T(3) * em + (T(4.5) * em * em - T(1.5) * mm) * a.inv_rho0);
            const T w = wk[k];
            const T cw = w * (b + c * s) * W;  // w dP/dgeq times W
            const T fq = w * c * T(3) * feq;
            bdr += cw;
            bm[0] += cw * (T(3) * T(e0) + (T(9) * em * T(e0) - T(3) * m[0]) * a.inv_rho0) - fq * Gh[0] * a.inv_rho0;
            bm[1] += cw * (T(3) * T(e1) + (T(9) * em * T(e1) - T(3) * m[1]) * a.inv_rho0) - fq * Gh[1] * a.inv_rho0;
            bG[0] += fq * (T(e0) - m[0] * a.inv_rho0);
            bG[1] += fq * (T(e1) - m[1] * a.inv_rho0);
        }
    });
}

// The fast regions. Interfaces normal to d: both cells, their tangential neighbours and
// the cells' own interfaces are in the domain without wrapping, and the interface is neither
// a wall nor the x_c of one. Cells: every interface of the stencil transposed in adj_cells
// is in the domain and the cell feeds no ghost or periodic image. Everything else (a frame
// along the boundary) takes the general path.
struct Rect {
    int W, H;            // index space W x H
    int x0, x1, y0, y1;  // fast rectangle, inclusive (empty when x0 > x1 or y0 > y1)
};
__host__ __device__ inline Rect face_rect(int d, int nx, int ny, int perx, int pery) {
    if (d == 0) {
        const int m = perx ? 1 : 2;
        return Rect{nx + 1, ny, m, nx - m, 1, ny - 2};
    }
    const int m = pery ? 1 : 2;
    return Rect{nx, ny + 1, 1, nx - 2, m, ny - m};
}
__host__ __device__ inline Rect cell_rect(int nx, int ny, int perx, int pery) {
    const int mx = perx ? 1 : 2, my = pery ? 1 : 2;
    return Rect{nx, ny, mx, nx - 1 - mx, my, ny - 1 - my};
}
__host__ __device__ inline bool rect_empty(const Rect &r) { return r.x0 > r.x1 || r.y0 > r.y1; }
__host__ __device__ inline int64_t rect_count(const Rect &r) {
    return rect_empty(r) ? 0 : (int64_t)(r.x1 - r.x0 + 1) * (r.y1 - r.y0 + 1);
}
__host__ __device__ inline int64_t frame_count(const Rect &r) { return (int64_t)r.W * r.H - rect_count(r); }
// The t-th element (row-major) of the index space outside the fast rectangle. 32-bit counts: the
// sweep's some 45 values per cell leave room for fewer than 2^31 cells.
__device__ inline void frame_at(const Rect &r, unsigned t, int &x, int &y) {
    const unsigned W = (unsigned)r.W;
    const bool none = rect_empty(r);
    const unsigned below = none ? ~0u : (unsigned)r.y0 * W, above = none ? 0u : (unsigned)(r.H - 1 - r.y1) * W;
    if (t < below || t - below < above) {
        y = (int)(t / W);
        x = (int)(t - (unsigned)y * W);
        if (t >= below) y += r.y1 + 1 - r.y0;
    } else {
        t -= below + above;
        const unsigned side = (unsigned)(r.x0 + (r.W - 1 - r.x1));  // frame columns of a middle row
        const unsigned row = t / side;
        const int c = (int)(t - row * side);
        y = r.y0 + (int)row;
        x = c < r.x0 ? c : r.x1 + 1 + (c - r.x0);
    }
}

template <class T, int d>
__device__ __forceinline__ void face_fast(const AdjParams<T> &a, int i, int j, int64_t f, int64_t nf) {
    const int nx = a.n[0];
    const int64_t nc = ncell(a);
    const int64_t cR = i + (int64_t)nx * j;
    const int64_t cL = d == 0 ? cR - 1 : cR - nx;
    const int64_t ts = d == 0 ? nx : 1;  // step to the tangential neighbour
    T F[Q];
    sfor<Q>([&](auto kc) {
        constexpr int k = kc;
        constexpr int ed = L9::e(k, d), et = L9::e(k, 1 - d);
        const T *ph = a.phi + k * nc;
        const T l = ph[cL], r = ph[cR];
        T v = T(0.5) * (l + r);
        if constexpr (ed != 0) v -= a.kappa * T(ed) * (r - l);
        if constexpr (et != 0) v -= T(0.25) * a.kappa * T(et) * ((ph[cL + ts] + ph[cR + ts]) - (ph[cL - ts] + ph[cR - ts]));
        F[k] = v;
    });
    T Gh[2];
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const T fl = a.field ? T(0.5) * ((T)a.field[c * nc + cL] + (T)a.field[c * nc + cR]) : T(0);
        Gh[c] = (a.g[c] + fl) * a.cthc;
    }
    T dr, m[2];
    moments2(a, F, Gh, a.wface, dr, m);
    T fbar[Q];
    sfor<Q>([&](auto kc) {
        constexpr int k = kc;
        constexpr int ed = L9::e(k, d);
        if constexpr (ed != 0) fbar[k] = a.two_kappa * T(ed) * (a.lam1[k * nc + cR] - a.lam1[k * nc + cL]);
        else fbar[k] = T(0);
    });
    T bdr = T(0), bm[2] = {T(0), T(0)}, Gb[2] = {T(0), T(0)};
    relax_T_c<T, d>(a, fbar, dr, m, Gh, a.b7, a.c7, bdr, bm, Gb);
    T *fb = a.fb[d];
    sfor<Q>([&](auto kc) {
        constexpr int k = kc;
        fb[k * nf + f] = (T(1) - a.b7) * fbar[k] + bdr + T(L9::e(k, 0)) * bm[0] + T(L9::e(k, 1)) * bm[1];
    });
    a.gb[d][f] = Gb[0] + a.rho0 * a.wface * bm[0];
    a.gb[d][nf + f] = Gb[1] + a.rho0 * a.wface * bm[1];
}

template <class T>
__device__ __forceinline__ void cell_fast(const AdjParams<T> &a, int x, int y, int64_t c) {
    const int nx = a.n[0];
    const int64_t nc = ncell(a), n0 = nface(a, 0), n1 = nface(a, 1);
    const int64_t ix = x + (int64_t)(nx + 1) * y;  // x interface (x, y): the cell's -x interface
    const int64_t iy = x + (int64_t)nx * y;        // y interface (x, y): the cell's -y interface
    const int64_t sx = nx + 1, sy = nx;            // row strides of the interface arrays
    const T h = T(0.5), q = T(0.25) * a.kappa;
    T pb[Q];
    sfor<Q>([&](auto kc) {
        constexpr int k = kc;
        constexpr int ex = L9::e(k, 0), ey = L9::e(k, 1);
        const T *f0 = a.fb[0] + k * n0, *f1 = a.fb[1] + k * n1;
        T v = T(4) / T(3) * a.lam1[k * nc + c];
        v += (h + a.kappa * T(ex)) * f0[ix + 1] + (h - a.kappa * T(ex)) * f0[ix];
        if constexpr (ey != 0) v += q * T(ey) * ((f0[ix + 1 + sx] + f0[ix + sx]) - (f0[ix + 1 - sx] + f0[ix - sx]));
        v += (h + a.kappa * T(ey)) * f1[iy + sy] + (h - a.kappa * T(ey)) * f1[iy];
        if constexpr (ex != 0) v += q * T(ex) * ((f1[iy + 1 + sy] + f1[iy + 1]) - (f1[iy - 1 + sy] + f1[iy - 1]));
        pb[k] = v;
    });
    const T dr = a.mom[c];
    const T m[2] = {a.mom[nc + c], a.mom[2 * nc + c]};
    T Gh[2];
    cell_Gh(a, x, y, Gh);
    T bdr = T(0), bm[2] = {T(0), T(0)}, bG[2] = {T(0), T(0)};
    relax_T_c<T, -1>(a, pb, dr, m, Gh, a.b1, a.c1, bdr, bm, bG);
    sfor<Q>([&](auto kc) {
        constexpr int k = kc;
        a.lam0[k * nc + c] = -a.lam1[k * nc + c] / T(3) + (T(1) - a.b1) * pb[k] + bdr + T(L9::e(k, 0)) * bm[0] +
                             T(L9::e(k, 1)) * bm[1];
    });
    if (a.dG) {
#pragma unroll
        for (int comp = 0; comp < 2; comp++) {
            const T fs = T(0.5) * (a.gb[0][comp * n0 + ix] + a.gb[0][comp * n0 + ix + 1]) +
                         T(0.5) * (a.gb[1][comp * n1 + iy] + a.gb[1][comp * n1 + iy + sy]);
            a.dG[comp * nc + c] += (double)((bG[comp] + a.rho0 * a.wcell * bm[comp]) * a.ctc + fs * a.cthc);
        }
    }
}

// ---- kernels ----
// fbar+ (step 1, eq. (24)) and the moments (eq. (27)) of cell c of `state` into
// a.phi and `mom`, with ctc = cos(omega t) / c at that state's time. Not inlined: the
// recompute kernel and the cells kernel that carries the next step's recompute run the same
// code, so the sweep's bits do not depend on which of them computed a step.
template <class T>
__device__ __noinline__ void fwd_cell(const AdjParams<T> &a, const T *state, T ctc, T *mom, int64_t c) {
    const int64_t nc = ncell(a);
    const int y = (int)((unsigned)c / (unsigned)a.n[0]), x = (int)c - y * a.n[0];
    T g[Q], Gh[2], dr, m[2];
#pragma unroll
    for (int k = 0; k < Q; k++) g[k] = state[k * a.dstride + (int64_t)y * a.px + x];
#pragma unroll
    for (int comp = 0; comp < 2; comp++) Gh[comp] = (a.g[comp] + field_at(a, comp, x, y)) * ctc;
    moments2(a, g, Gh, a.wcell, dr, m);
    const T gm = (Gh[0] * m[0] + Gh[1] * m[1]) * a.inv_rho0;
#pragma unroll
    for (int k = 0; k < Q; k++) {
        const T q = geq(a, k, dr, m);
        const T s = T(3) * (Gh[0] * (T)L9::e(k, 0) + Gh[1] * (T)L9::e(k, 1) - gm);
        a.phi[k * nc + c] = g[k] + a.b1 * (q - g[k]) + a.c1 * s * (L9::wt<T>(k) * a.rho0 + q);
    }
    mom[c] = dr;
    mom[nc + c] = m[0];
    mom[2 * nc + c] = m[1];
}

template <class T>
__global__ void __launch_bounds__(256) adj_cells_fwd(const AdjParams<T> a) {
    const int64_t nc = ncell(a);
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x)
        fwd_cell(a, a.state, a.ctc, a.mom, c);
}

// The t-th interface of the frame of both axes, one velocity per lane of the calling half-warp. The
// interface next to a wall is x_c of the wall's (reading R4) and has the wall's item as well: both
// take their step-4 values from the same two cells of each line, and what the wall passes to x_c
// (step 5) stays in the lane. The time of this kernel and of the cells' is the latency of one frame item
// wherever the interior is small (512 x 256 channel: 30.6 us per reverse step when a wall, an
// x_c and a corner each formed their neighbours' values anew, 13 us of each kernel in the frame
// alone; now 22).
template <class T>
__device__ __noinline__ void faces_frame_item(const AdjParams<T> &a, unsigned t) {
    const Rect r0 = face_rect(0, a.n[0], a.n[1], a.per[0], a.per[1]);
    const Rect r1 = face_rect(1, a.n[0], a.n[1], a.per[0], a.per[1]);
    const unsigned c0 = (unsigned)frame_count(r0);
    const int d = t < c0 ? 0 : 1;
    int i, j;
    frame_at(d == 0 ? r0 : r1, d == 0 ? t : t - c0, i, j);
    const int n = d == 0 ? a.n[0] : a.n[1], nt = d == 0 ? a.n[1] : a.n[0];
    const int per = d == 0 ? a.per[0] : a.per[1], pert = d == 0 ? a.per[1] : a.per[0];
    const int pos = d == 0 ? i : j, tp = d == 0 ? j : i;
    if (!per && (pos == 0 || pos == n)) return;  // a wall: its x_c's item makes it
    const LaneVel<T> l;
    const int lane = half_lane(), ien = d == 0 ? l.ie[0] : l.ie[1];
    const T en = d == 0 ? l.e[0] : l.e[1], et = d == 0 ? l.e[1] : l.e[0];
    const int64_t nc = ncell(a);
    const unsigned nx = (unsigned)a.n[0], sn = d == 0 ? 1u : nx, st = d == 0 ? nx : 1u;
    // the two cells, and their tangential neighbours
    const unsigned lo = sn * (unsigned)(pos > 0 ? pos - 1 : n - 1), hi = sn * (unsigned)(pos < n ? pos : 0);
    const unsigned own = st * (unsigned)tp;
    int cp[2], cm[2];
    T wp[2], wm[2];
    ext2<T>(tp + 1, nt, pert, cp, wp);
    ext2<T>(tp - 1, nt, pert, cm, wm);
    const T *ph = a.phi + l.k * nc, *lam = a.lam1 + l.k * nc;
    auto line = [&](unsigned c, T &v, T &dv) __attribute__((always_inline)) {
        v = ph[c + own];
        dv = (wp[0] * ph[c + st * (unsigned)cp[0]] + wp[1] * ph[c + st * (unsigned)cp[1]]) -
             (wm[0] * ph[c + st * (unsigned)cm[0]] + wm[1] * ph[c + st * (unsigned)cm[1]]);
        if (!l.act) v = dv = T(0);
    };
    T A, dA, B, dB;
    line(lo, A, dA);
    line(hi, B, dB);
    const T lamA = l.act ? lam[lo + own] : T(0), lamB = l.act ? lam[hi + own] : T(0);
    T fA[2] = {T(0), T(0)}, fB[2] = {T(0), T(0)};
    if (a.field) {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            fA[c] = (T)a.field[c * nc + lo + own];
            fB[c] = (T)a.field[c * nc + hi + own];
        }
    }
    const T k4 = T(0.25) * a.kappa * et, kn = a.kappa * en, rw = a.rho0 * a.wface;
    const int64_t nf = nface(a, d);
    T *fb = a.fb[d] + l.k * nf, *gb = a.gb[d];
    auto face_at = [&](int p) __attribute__((always_inline)) { return d == 0 ? fidx(a, 0, p, tp) : fidx(a, 1, tp, p); };
    auto store = [&](int64_t f, T Fb, T G0, T G1) __attribute__((always_inline)) {
        if (l.act) fb[f] = Fb;
        if (lane < 2) gb[lane * nf + f] = lane ? G1 : G0;
    };
    // ---- the interface itself: steps 3-7 forward, then steps 9-6 backward. Steps 8-9: velocity k
    // enters the update of the low cell with -2 kappa e_d and of the high cell with +2 kappa e_d ----
    const T F = T(0.5) * (A + B) - kn * (B - A) - k4 * (dA + dB);
    T Gh[2], m[2], Gb[2], bdr, bm[2];
#pragma unroll
    for (int c = 0; c < 2; c++) Gh[c] = (a.g[c] + T(0.5) * (fA[c] + fB[c])) * a.cthc;
    const T dr = wsum(F);
#pragma unroll
    for (int c = 0; c < 2; c++) m[c] = wsum(l.e[c] * F) + rw * Gh[c];
    const T fbar = a.two_kappa * en * ((pos < n ? lamB : T(0)) - (pos > 0 ? lamA : T(0)));
    relax_T_lane(a, l, fbar, dr, m, Gh, a.b7, a.c7, bdr, bm, Gb);
    T Fb = (T(1) - a.b7) * fbar + bdr + l.e[0] * bm[0] + l.e[1] * bm[1];
#pragma unroll
    for (int c = 0; c < 2; c++) Gb[c] += rw * bm[c];
    // ---- the wall interfaces whose x_c it is ----
#pragma unroll 1
    for (int sd = 0; sd < 2; sd++) {
        if (per || pos != (sd == 0 ? 1 : n - 1)) continue;
        const int wid = 2 * d + sd, type = a.bc[wid];
        const T sg = sd == 0 ? T(1) : T(-1);  // the incoming velocities' e_d
        const T C = sd == 0 ? A : B, dC = sd == 0 ? dA : dB;  // the wall's cell; its ghost (step 2) is 2 C - other
        const T G = T(2) * C - (sd == 0 ? B : A), dG = T(2) * dC - (sd == 0 ? dB : dA);
        const bool incoming = l.act && (sd == 0 ? ien > 0 : ien < 0), bb = type == DUGKS_BC_BOUNCE_BACK;
        const bool vel = type == DUGKS_BC_NEQ_VELOCITY;
        T Fw = T(0.5) * (G + C) - kn * sg * (C - G) - k4 * (dG + dC);
        const unsigned mask = 0xffffu << (threadIdx.x & 16);
        const int64_t slot = d == 0 ? (sd == 0 ? 0 : a.n[1]) + j : 2 * (int64_t)a.n[1] + (sd == 0 ? 0 : a.n[0]) + i;
        const bool wantW = a.dW && (bb || vel) && lane < 2;
        const double dW0 = wantW ? a.dW[2 * slot + lane] : 0.0;
        const T mw[2] = {a.mw[wid][0], a.mw[wid][1]};
        T Gw[2], mwf[2], Gwb[2], Wb[2], ma[2];
#pragma unroll
        for (int c = 0; c < 2; c++) {
            Gw[c] = (a.g[c] + (sd == 0 ? fA[c] : fB[c])) * a.cthc;
            ma[c] = vel ? mw[c] : m[c];
        }
        // step 5: eq. (31), or eq. (32) with drho_a, m_a of a velocity or a pressure condition
        const T Fo = __shfl_sync(mask, Fw, Q - 1 - l.k, 16);
        const T dra = vel ? dr : a.drw[wid] + a.drw1[wid] * a.cwh;
        const T Fin = bb ? Fo + T(6) * l.W * (l.e[0] * mw[0] + l.e[1] * mw[1])
                         : geq_lane(l, a.inv_rho0, dra, ma) + F - geq_lane(l, a.inv_rho0, dr, m);
        if (incoming) Fw = Fin;
        const T drw = wsum(Fw);
#pragma unroll
        for (int c = 0; c < 2; c++) mwf[c] = wsum(l.e[c] * Fw) + rw * Gw[c];
        const T fw = a.two_kappa * en * (sd == 0 ? lamA : -lamB);
        T bd, b[2];
        relax_T_lane(a, l, fw, drw, mwf, Gw, a.b7, a.c7, bd, b, Gwb);
        T Fwb = (T(1) - a.b7) * fw + bd + l.e[0] * b[0] + l.e[1] * b[1];
        // step 5 backward: the weight of an incoming velocity passes to its opposite and u_w (eq. (31)),
        // or to x_c's value and moments and to u_w (the W_k terms of a velocity condition and the m terms of a
        // pressure condition cancel)
        const T w = incoming ? Fwb : T(0);
        if (incoming) Fwb = T(0);
        T dw[2];
        if (bb) {
            Fwb += __shfl_sync(mask, w, Q - 1 - l.k, 16);
#pragma unroll
            for (int c = 0; c < 2; c++) dw[c] = T(6) * l.W * l.e[c];
        } else {
            T xd = T(0), xm[2] = {T(0), T(0)};
            geq_dm_lane(l, a.inv_rho0, mw, dw);
            if (vel) {
                T dc[2];
                geq_dm_lane(l, a.inv_rho0, m, dc);
#pragma unroll
                for (int c = 0; c < 2; c++) xm[c] = -wsum(w * dc[c]);
            } else {
                xd = -wsum(w * l.W);
            }
            Fb += w + xd + l.e[0] * xm[0] + l.e[1] * xm[1];
#pragma unroll
            for (int c = 0; c < 2; c++) Gb[c] += rw * xm[c];
        }
        if (a.dW && (bb || vel)) {
#pragma unroll
            for (int c = 0; c < 2; c++) Wb[c] = wsum(w * dw[c] * a.dmw);
            if (wantW) a.dW[2 * slot + lane] = dW0 + (double)(lane ? Wb[1] : Wb[0]);
        }
        store(face_at(sd == 0 ? 0 : n), Fwb, Gwb[0] + rw * b[0], Gwb[1] + rw * b[1]);
    }
    store(face_at(pos), Fb, Gb[0], Gb[1]);
}

// The frame item of a thread: eight per block of 128 threads, one per half-warp. From the block's number,
// not the thread's: 16 threads an item pass 32 bits at 2^28 items (a long strip of 10^8 cells is all frame).
__host__ __device__ constexpr unsigned frame_item(unsigned block, unsigned thread) { return block * 8u + (thread >> 4); }
static_assert(frame_item(0, 127) == 7 && frame_item(1u << 25, 0) == 1u << 28 && frame_item((1u << 28) - 1, 127) == (1u << 31) - 1,
              "frame items up to 2^31 - 1 have blocks and threads of their own");

// Every interface of both axes in one launch of 128-thread blocks: the frame blocks first
// (eight frame interfaces per block, one per half-warp), then 32 x 4 tiles of the interior
// rectangle of x interfaces (nt0 tiles, tx0 per row), then those of y interfaces (tx1 per row).
template <class T>
__global__ void __launch_bounds__(128, 6) adj_faces_all(const AdjParams<T> a, int64_t nframe, int nfb, int nt0,
                                                         int tx0, int tx1) {
    if ((int)blockIdx.x < nfb) {
        const unsigned t = frame_item(blockIdx.x, threadIdx.x);
        if (t < nframe) faces_frame_item(a, t);
        return;
    }
    int b = (int)blockIdx.x - nfb;
    const int d = b < nt0 ? 0 : 1;
    if (d) b -= nt0;
    const int tx = d ? tx1 : tx0;
    const Rect r = face_rect(d, a.n[0], a.n[1], a.per[0], a.per[1]);
    const int i = r.x0 + (b % tx) * 32 + (threadIdx.x & 31), j = r.y0 + (b / tx) * 4 + (threadIdx.x >> 5);
    if (i > r.x1 || j > r.y1) return;
    const int64_t f = fidx(a, d, i, j);
    if (d == 0) face_fast<T, 0>(a, i, j, f, nface(a, 0));
    else face_fast<T, 1>(a, i, j, f, nface(a, 1));
}

// Transposes of the reconstruction and of step 2 along one axis, for the cell at x of n: the (at most
// four) interfaces across the axis whose step-4 values it enters as one of the two cells, directly or
// through a ghost or an image, as weights of the normal part (h -+ kappa e: w1), of the
// tangential part (w2) and of the interface acceleration (wg; reading R2); and its rows as a
// tangential neighbour, above, own (through a ghost) and below, with weights t.
template <class T>
struct AxisT {
    int f[4], row[3];  // f < 0: absent
    T w1[4], w2[4], wg[4], t[3];
    __device__ __forceinline__ AxisT(int x, int n, int per, T ke) {
        const T hp = T(0.5) + ke, hm = T(0.5) - ke;
        const bool lo = !per && x == 0, hi = !per && x == n - 1, lo1 = !per && x == 1, hi1 = !per && x == n - 2;
        const bool pl = per && x == 0, ph = per && x == n - 1;
        f[0] = x;
        w1[0] = hm + (lo ? T(2) * hp : T(0));
        w2[0] = lo ? T(3) : T(1);
        wg[0] = lo ? T(1) : T(0.5);
        f[1] = x + 1;
        w1[1] = hp + (hi ? T(2) * hm : T(0));
        w2[1] = hi ? T(3) : T(1);
        wg[1] = hi ? T(1) : T(0.5);
        f[2] = lo1 || ph ? 0 : -1;
        w1[2] = ph ? hp : -hp;
        w2[2] = ph ? T(1) : T(-1);
        wg[2] = ph ? T(0.5) : T(0);
        f[3] = hi1 || pl ? n : -1;
        w1[3] = pl ? hm : -hm;
        w2[3] = pl ? T(1) : T(-1);
        wg[3] = pl ? T(0.5) : T(0);
        row[0] = x + 1 < n ? x + 1 : (per ? 0 : x);
        row[1] = x;
        row[2] = x > 0 ? x - 1 : (per ? n - 1 : x);
        t[0] = hi ? T(0) : (hi1 ? T(2) : T(1));
        t[1] = (lo ? T(2) : T(0)) - (hi ? T(2) : T(0));
        t[2] = lo ? T(0) : (lo1 ? T(-2) : T(-1));
    }
};

// The t-th frame cell (cells whose stencil meets a wall ghost, a periodic image or a
// wall-clamped interface acceleration), one velocity per lane of the calling half-warp. Every
// load's address is known at the start.
template <class T>
__device__ __noinline__ void cells_frame_item(const AdjParams<T> &a, unsigned t) {
    const int64_t nc = ncell(a), n0 = nface(a, 0), n1 = nface(a, 1);
    const Rect r = cell_rect(a.n[0], a.n[1], a.per[0], a.per[1]);
    int x, y;
    frame_at(r, t, x, y);
    const LaneVel<T> l;
    const int lane = half_lane();
    const unsigned nx = (unsigned)a.n[0], c = (unsigned)x + nx * (unsigned)y;
    const AxisT<T> ax(x, a.n[0], a.per[0], a.kappa * l.e[0]), ay(y, a.n[1], a.per[1], a.kappa * l.e[1]);
    const T dr = a.mom[c];
    const T m[2] = {a.mom[nc + c], a.mom[2 * nc + c]};
    T Gh[2];
    cell_Gh(a, x, y, Gh);
    const T l1 = a.lam1[l.k * nc + c];
    const int comp = lane & 1;
    const bool wantG = a.dG && lane < 2;
    const double g0 = wantG ? a.dG[comp * nc + c] : 0.0;
    // adjoint of fbar+ of this cell: eq. (25) (4/3 fbar+) and the interface values it enters
    const T *f0 = a.fb[0] + l.k * n0, *f1 = a.fb[1] + l.k * n1;
    const T *g0x = a.gb[0] + comp * n0, *g1y = a.gb[1] + comp * n1;
    const T q = T(0.25) * a.kappa;
    T pb = T(4) / T(3) * l1, gs = T(0);
#pragma unroll
    for (int s = 0; s < 4; s++) {
        if (s >= 2 && ax.f[s] < 0) continue;
        const T *p = f0 + ax.f[s];
        const unsigned sr = nx + 1, o = sr * (unsigned)y;
        const T v = p[o], u = ay.t[0] * p[sr * (unsigned)ay.row[0]] + ay.t[1] * v + ay.t[2] * p[sr * (unsigned)ay.row[2]];
        pb += ax.w1[s] * v + q * l.e[1] * ax.w2[s] * u;
        if (wantG) gs += ax.wg[s] * g0x[ax.f[s] + o];
    }
#pragma unroll
    for (int s = 0; s < 4; s++) {
        if (s >= 2 && ay.f[s] < 0) continue;
        const T *p = f1 + (int64_t)nx * ay.f[s];
        const T v = p[x], u = ax.t[0] * p[ax.row[0]] + ax.t[1] * v + ax.t[2] * p[ax.row[2]];
        pb += ay.w1[s] * v + q * l.e[0] * ay.w2[s] * u;
        if (wantG) gs += ay.wg[s] * g1y[(int64_t)nx * ay.f[s] + x];
    }
    if (!l.act) pb = T(0);
    // step 1 (eq. (24)) and the cell moments (eq. (27))
    T bdr, bm[2], bG[2];
    relax_T_lane(a, l, pb, dr, m, Gh, a.b1, a.c1, bdr, bm, bG);
    if (l.act) a.lam0[l.k * nc + c] = -l1 / T(3) + (T(1) - a.b1) * pb + bdr + l.e[0] * bm[0] + l.e[1] * bm[1];
    if (wantG)
        a.dG[comp * nc + c] = g0 + (double)(((comp ? bG[1] : bG[0]) + a.rho0 * a.wcell * (comp ? bm[1] : bm[0])) * a.ctc +
                                            gs * a.cthc);
}

// All cells in one launch of 128-thread blocks: frame blocks first (a half-warp per frame cell),
// then 32 x 4 tiles of the fast rectangle (tx x ty blocks).
// With a.nstate set, the blocks then recompute the next reverse step's fbar+ and moments,
// one cell per thread in the blocks' order, so that the blocks of a last, partial wave have none
// (512 x 256: 3% of a reverse step against giving them to the interior tiles first): this
// step's interfaces no longer read a.phi, and each cell's moments go to the other buffer, so
// no block reads what another overwrites.
template <class T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 7 : 5) adj_cells_all(const AdjParams<T> a, int nfb, int tx, int ty) {
    const Rect r = cell_rect(a.n[0], a.n[1], a.per[0], a.per[1]);
    if ((int)blockIdx.x < nfb) {  // eight frame cells per block, one per half-warp
        const unsigned t = frame_item(blockIdx.x, threadIdx.x);
        if (t < frame_count(r)) cells_frame_item(a, t);
    } else {
        const int b = blockIdx.x - nfb;
        const int x = r.x0 + (b % tx) * 32 + (threadIdx.x & 31), y = r.y0 + (b / tx) * 4 + (threadIdx.x >> 5);
        if (x <= r.x1 && y <= r.y1) cell_fast(a, x, y, x + (int64_t)a.n[0] * y);
    }
    if (a.nstate) {
        const int64_t nc = ncell(a);
        for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x)
            fwd_cell(a, a.nstate, a.nctc, a.nmom, c);
    }
}

// Loss seed from dL/d(moments) [3][ncell] (p, u_x, u_y as dugks_moments returns them):
// p = RT sum g~, u = c/rho0 sum e g~ + G cos(omega t) dt/2 (eq. (27)).
template <class T>
__global__ void adj_seed(const AdjParams<T> a, const float *dLdm, T rt, T c_over_rho0, double gdt) {
    const int64_t nc = ncell(a);
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x) {
        const T gp = (T)dLdm[c], gu0 = (T)dLdm[nc + c], gu1 = (T)dLdm[2 * nc + c];
        for (int k = 0; k < Q; k++)
            a.lam0[k * nc + c] = rt * gp + c_over_rho0 * ((T)L9::e(k, 0) * gu0 + (T)L9::e(k, 1) * gu1);
        if (a.dG) {
            a.dG[c] += (double)gu0 * gdt;
            a.dG[nc + c] += (double)gu1 * gdt;
        }
    }
}

// dL/du_w per face [6][3] from the per-wall-interface slots (-x: ny, +x: ny, -y: nx, +y: nx
// slots of 2 components), each sum in slot order (deterministic); zero for the faces that
// are not velocity walls.
__global__ void adj_wall_sum(const double *slots, double *out, int nx, int ny, int vx0, int vx1, int vy0, int vy1) {
    const int t = threadIdx.x;  // face * 3 + component
    if (t >= 18) return;
    const int f = t / 3, comp = t % 3;
    const int vel[4] = {vx0, vx1, vy0, vy1};
    double s = 0.0;
    if (f < 4 && comp < 2 && vel[f]) {
        const int first = f == 0 ? 0 : f == 1 ? ny : f == 2 ? 2 * ny : 2 * ny + nx;
        const int count = f < 2 ? ny : nx;
        for (int i = 0; i < count; i++) s += slots[2 * (first + i) + comp];
    }
    out[t] = s;
}

__global__ void adj_to_float(const double *src, float *dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (float)src[i];
}

// Face types whose wall velocity enters the step (and so has a gradient).
static int moving_wall(int type) { return type == DUGKS_BC_NEQ_VELOCITY || type == DUGKS_BC_BOUNCE_BACK; }

int blocks_for(int64_t n, int threads) {
    const int64_t b = (n + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 1 << 20));
}

// Work buffers carved from one allocation (element size es, 256-byte aligned pieces).
struct AdjBufs {
    void *phi, *mom[2], *fb[2], *gb[2], *lam[2];
};

size_t al256(size_t b) { return (b + 255) / 256 * 256; }

size_t scratch_bytes(int64_t nx, int64_t ny, size_t es) {
    const int64_t nc = nx * ny, n0 = (nx + 1) * ny, n1 = nx * (ny + 1);
    return al256(es * Q * nc) + 2 * al256(es * 3 * nc) + al256(es * Q * n0) + al256(es * Q * n1) + al256(es * 2 * n0) +
           al256(es * 2 * n1) + 2 * al256(es * Q * nc);
}

AdjBufs carve(void *base, int64_t nx, int64_t ny, size_t es) {
    const int64_t nc = nx * ny, n0 = (nx + 1) * ny, n1 = nx * (ny + 1);
    char *p = (char *)base;
    AdjBufs B;
    B.phi = p; p += al256(es * Q * nc);
    B.mom[0] = p; p += al256(es * 3 * nc);
    B.mom[1] = p; p += al256(es * 3 * nc);
    B.fb[0] = p; p += al256(es * Q * n0);
    B.fb[1] = p; p += al256(es * Q * n1);
    B.gb[0] = p; p += al256(es * 2 * n0);
    B.gb[1] = p; p += al256(es * 2 * n1);
    B.lam[0] = p; p += al256(es * Q * nc);
    B.lam[1] = p;
    return B;
}

template <class T>
AdjParams<T> base_params(const dugks_t h, const AdjBufs &B) {
    AdjParams<T> a;
    memset(&a, 0, sizeof a);
    const StepParams p = handle_params(h);
    a.n[0] = (int)h->nx;
    a.n[1] = (int)h->ny;
    a.per[0] = h->bcs.face[0].type == DUGKS_BC_PERIODIC;
    a.per[1] = h->bcs.face[2].type == DUGKS_BC_PERIODIC;
    a.px = p.px;
    a.dstride = p.dstride;
    for (int w = 0; w < 4; w++) {
        a.bc[w] = p.bc[w];
        a.mw[w][0] = (T)(p.bc_u[w][0] * p.rho0 * p.inv_c);
        a.mw[w][1] = (T)(p.bc_u[w][1] * p.rho0 * p.inv_c);
        a.drw[w] = (T)p.bc_drho[w];
        a.drw1[w] = (T)p.bc_drho1[w];
    }
    a.rho0 = (T)p.rho0;
    a.inv_rho0 = (T)(1.0 / p.rho0);
    a.dmw = (T)(p.rho0 * p.inv_c);
    a.b1 = (T)p.b1;
    a.c1 = (T)p.c1;
    a.b7 = (T)p.b7;
    a.c7 = (T)p.c7;
    a.kappa = (T)p.kappa;
    a.two_kappa = (T)p.two_kappa;
    a.wcell = (T)p.wcell;
    a.wface = (T)p.wface;
    a.g[0] = (T)p.g[0];
    a.g[1] = (T)p.g[1];
    a.field = p.field;
    a.phi = (T *)B.phi;
    a.mom = (T *)B.mom[0];
    for (int d = 0; d < 2; d++) {
        a.fb[d] = (T *)B.fb[d];
        a.gb[d] = (T *)B.gb[d];
    }
    a.dG = h->tape.dG;
    a.dW = h->tape.dW;
    return a;
}

// cos(omega t) / c at the time t of a state, as the recompute of that state uses it.
template <class T>
T force_factor(const dugks_t h, double t) {
    return (T)(cos(h->force.omega * t) * (1.0 / h->c));
}

// One reverse step at the state g~^n held in `state` (t_n = tn): lambda' in lam1 -> lam0,
// with the cell moments of g~^n in `mom`. Launches: the cell recompute unless the previous
// reverse step's cells kernel made it (have_fwd), all interfaces (frame blocks first), and
// all cells (frame blocks first), which also recompute g~^{n-1} = `next` (at time tnext) into
// a.phi and `nmom` when `next` is given.
template <class T>
cudaError_t reverse_step(AdjParams<T> a, const dugks_t h, const void *state, double tn, const void *lam1,
                         void *lam0, void *mom, bool have_fwd, const void *next, double tnext, void *nmom,
                         int64_t *launches) {
    const double om = h->force.omega, inv_c = 1.0 / h->c;
    a.ctc = force_factor<T>(h, tn);
    a.cthc = (T)(cos(om * (tn + 0.5 * h->dt)) * inv_c);
    a.cwh = (T)cos(om * (tn + 0.5 * h->dt));
    a.state = (const T *)state;
    a.lam1 = (const T *)lam1;
    a.lam0 = (T *)lam0;
    a.mom = (T *)mom;
    a.nstate = (const T *)next;
    a.nmom = (T *)nmom;
    a.nctc = next ? force_factor<T>(h, tnext) : T(0);
    cudaStream_t st = h->stream;
    const int nx = (int)h->nx, ny = (int)h->ny;
    const int64_t nc = h->ncell;
    int64_t n = 0;
    if (!have_fwd) {
        adj_cells_fwd<T><<<blocks_for(nc, 256), 256, 0, st>>>(a);
        n++;
    }
    {
        const Rect r0 = face_rect(0, nx, ny, a.per[0], a.per[1]), r1 = face_rect(1, nx, ny, a.per[0], a.per[1]);
        const int64_t nframe = frame_count(r0) + frame_count(r1);
        const int nfb = (int)((nframe + 7) / 8);
        const int tx0 = rect_empty(r0) ? 0 : (r0.x1 - r0.x0 + 32) / 32, ty0 = rect_empty(r0) ? 0 : (r0.y1 - r0.y0 + 4) / 4;
        const int tx1 = rect_empty(r1) ? 0 : (r1.x1 - r1.x0 + 32) / 32, ty1 = rect_empty(r1) ? 0 : (r1.y1 - r1.y0 + 4) / 4;
        const int nb = nfb + tx0 * ty0 + tx1 * ty1;
        if (nb > 0) {
            adj_faces_all<T><<<nb, 128, 0, st>>>(a, nframe, nfb, tx0 * ty0, tx0, tx1);
            n++;
        }
    }
    {
        const Rect rc = cell_rect(nx, ny, a.per[0], a.per[1]);
        const int tx = rect_empty(rc) ? 0 : (rc.x1 - rc.x0 + 32) / 32, ty = rect_empty(rc) ? 0 : (rc.y1 - rc.y0 + 4) / 4;
        const int nfb = (int)((frame_count(rc) + 7) / 8);
        const int nb = nfb + tx * ty;
        if (nb > 0) {
            adj_cells_all<T><<<nb, 128, 0, st>>>(a, nfb, tx, ty);
            n++;
        }
    }
    *launches += n;
    return cudaGetLastError();
}

// The work of one checkpoint segment of `len` steps whose first state is in seg[0] (copied
// from the checkpoint) and whose clock starts at `start`: recompute the states into
// seg[1 .. len-1], then the reverse steps len-1 .. 0 with lambda ping-ponging from
// lam[cur]. Returns the number of launches through *launches.
template <class T>
cudaError_t enqueue_segment(dugks_t h, const AdjParams<T> &a, const AdjBufs &B, int64_t start, int64_t len, int cur,
                            int64_t *launches) {
    AdjointTape &t = h->tape;
    for (int64_t j = 1; j < len; j++) {
        StepParams p = handle_params(h);
        p.src = t.seg[(size_t)j - 1];
        p.dst = t.seg[(size_t)j];
        p.step_ctr = t.zero;
        p.step_off = (int)(t.step0 + start + j - 1);
        cudaError_t e = handle_launch_step(h, p);
        if (e != cudaSuccess) return e;
        (*launches)++;
    }
    // step j's cell moments are in mom[j & 1]; each cells kernel but the segment's last also
    // recomputes step j - 1
    for (int64_t j = len - 1; j >= 0; j--) {
        const double tn = (double)(t.step0 + start + j) * h->dt;
        const double tprev = (double)(t.step0 + start + j - 1) * h->dt;
        cudaError_t e = reverse_step<T>(a, h, t.seg[(size_t)j], tn, B.lam[cur], B.lam[cur ^ 1], B.mom[j & 1],
                                        j < len - 1, j > 0 ? t.seg[(size_t)j - 1] : nullptr, tprev,
                                        B.mom[(j - 1) & 1], launches);
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    return cudaSuccess;
}

template <class T>
int enqueue_adjoint(dugks_t h, const float *dL_dmom, float *dL_dfield, void *dL_dstate0) {
    AdjointTape &t = h->tape;
    const size_t es = sizeof(T);
    const AdjBufs B = carve(t.scratch, h->nx, h->ny, es);
    const int64_t nc = h->ncell;
    const int64_t nwall = 2 * (h->nx + h->ny);
    cudaStream_t st = h->stream;
    cudaError_t e = cudaMemsetAsync(t.dG, 0, sizeof(double) * 2 * nc, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.dW, 0, sizeof(double) * 2 * nwall, st);
    if (e != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "adjoint: %s", cudaGetErrorString(e));
    AdjParams<T> a = base_params<T>(h, B);
    {  // seed at the end of the rollout
        const double tend = (double)(t.step0 + t.steps) * h->dt;
        AdjParams<T> s = a;
        s.lam0 = (T *)B.lam[0];
        adj_seed<T><<<blocks_for(nc, 256), 256, 0, st>>>(s, dL_dmom, (T)h->rt, (T)(h->c / h->rho0),
                                                          cos(h->force.omega * tend) * 0.5 * h->dt);
        h->launches++;
    }
    int cur = 0;
    const int64_t every = t.every;
    const int64_t nseg = (t.steps + every - 1) / every;
    // With a time-independent acceleration every segment of the same length and starting
    // parity is the same sequence of launches on the same buffers: capture it once as a
    // CUDA graph and replay it per segment.
    const bool graphs = h->use_graph && h->force.omega == 0.0 && nseg >= 3;
    // What a captured segment bakes in besides its length and parity: the forward step's and
    // the adjoint's parameter records (with omega = 0 neither depends on the segment's
    // time), the segment state buffers and the kernel selection. A graph of an earlier call
    // is reused while all of these are unchanged (its work has completed: the caller's
    // stream was synchronised before this call).
    std::vector<unsigned char> sig;
    if (graphs) {
        StepParams p0 = handle_params(h);
        p0.src = p0.dst = nullptr;
        p0.step_ctr = t.zero;
        auto put = [&](const void *q, size_t n) {
            const unsigned char *c = (const unsigned char *)q;
            sig.insert(sig.end(), c, c + n);
        };
        put(&p0, sizeof p0);
        put(&a, sizeof a);
        const int sel[4] = {h->kernel, h->tile_x, h->tile_y, h->store};
        put(sel, sizeof sel);
        for (void *q : t.seg) put(&q, sizeof q);
    }
    int rc = DUGKS_OK;
    for (int64_t sg = nseg - 1; sg >= 0 && rc == DUGKS_OK; sg--) {
        const int64_t start = sg * every;
        const int64_t len = std::min<int64_t>(every, t.steps - start);
        e = cudaMemcpyAsync(t.seg[0], t.ckpt[(size_t)sg], h->state_bytes, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) { rc = handle_fail(h, DUGKS_E_CUDA, "adjoint: %s", cudaGetErrorString(e)); break; }
        int64_t nl = 0;
        if (graphs) {
            AdjointTape::SegGraph *hit = nullptr;
            for (auto &gr : t.graphs)
                if (gr.len == len && gr.cur == cur) hit = &gr;
            if (hit && hit->sig != sig) {  // captured with other buffers or parameters
                cudaGraphExecDestroy(hit->exec);
                *hit = t.graphs.back();
                t.graphs.pop_back();
                hit = nullptr;
            }
            if (!hit) {
                cudaGraph_t g;
                e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
                if (e == cudaSuccess) {
                    cudaError_t e2 = enqueue_segment<T>(h, a, B, start, len, cur, &nl);
                    e = cudaStreamEndCapture(st, &g);
                    if (e2 != cudaSuccess) e = e2;
                }
                cudaGraphExec_t ge = nullptr;
                if (e == cudaSuccess) {
                    e = cudaGraphInstantiate(&ge, g, 0);
                    cudaGraphDestroy(g);
                }
                if (e != cudaSuccess) { rc = handle_fail(h, DUGKS_E_CUDA, "adjoint graph: %s", cudaGetErrorString(e)); break; }
                t.graphs.push_back(AdjointTape::SegGraph{len, cur, sig, ge, nl});
                hit = &t.graphs.back();
            }
            nl = hit->launches;
            e = cudaGraphLaunch(hit->exec, st);
        } else {
            e = enqueue_segment<T>(h, a, B, start, len, cur, &nl);
        }
        if (e != cudaSuccess) { rc = handle_fail(h, DUGKS_E_CUDA, "adjoint step: %s", cudaGetErrorString(e)); break; }
        h->launches += nl;
        if (len & 1) cur ^= 1;
    }
    if (rc != DUGKS_OK) {
        cudaStreamSynchronize(st);
        return rc;
    }
    if (dL_dfield) {
        adj_to_float<<<blocks_for(2 * nc, 256), 256, 0, st>>>(t.dG, dL_dfield, 2 * nc);
        h->launches++;
    }
    if (dL_dstate0) {
        e = cudaMemcpyAsync(dL_dstate0, B.lam[cur], es * Q * nc, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "adjoint: %s", cudaGetErrorString(e));
    }
    adj_wall_sum<<<1, 32, 0, st>>>(t.dW, t.dW_face, (int)h->nx, (int)h->ny,
                                   moving_wall(h->bcs.face[0].type), moving_wall(h->bcs.face[1].type),
                                   moving_wall(h->bcs.face[2].type), moving_wall(h->bcs.face[3].type));
    h->launches++;
    e = cudaMemcpyAsync(t.h_wall, t.dW_face, sizeof(double) * 18, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "adjoint: %s", cudaGetErrorString(e));
    return DUGKS_OK;
}

}  // namespace

void adjoint_release(dugks_t h) {
    AdjointTape &t = h->tape;
    for (void *p : t.ckpt) cudaFree(p);
    for (void *p : t.seg) cudaFree(p);
    t.ckpt.clear();
    t.seg.clear();
    cudaFree(t.scratch);
    cudaFree(t.dG);
    cudaFree(t.dW);
    cudaFree(t.zero);
    cudaFree(t.dW_face);
    if (t.h_wall) cudaFreeHost(t.h_wall);
    for (auto &gr : t.graphs) cudaGraphExecDestroy(gr.exec);
    t.graphs.clear();
    t.scratch = nullptr;
    t.dG = t.dW = t.dW_face = t.h_wall = nullptr;
    t.zero = nullptr;
    t.steps = 0;
}

}  // namespace dugks

using namespace dugks;

static int check_adjoint_support(dugks_t h) {
    if (h->q != DUGKS_D2Q9 || h->dim != 2)
        return handle_fail(h, DUGKS_E_UNSUPPORTED, "record/adjoint: built for D2Q9 only");
    if (h->store != DUGKS_STORE_F32 && h->store != DUGKS_STORE_F64)
        return handle_fail(h, DUGKS_E_UNSUPPORTED, "record/adjoint: F32 or F64 storage only");
    if (h->model != DUGKS_MODEL_INCOMPRESSIBLE)
        return handle_fail(h, DUGKS_E_UNSUPPORTED, "record/adjoint: the incompressible model only");
    if (h->d_metric) return handle_fail(h, DUGKS_E_UNSUPPORTED, "record/adjoint: uniform meshes only");
    return DUGKS_OK;
}

extern "C" int dugks_record(dugks_t h, int64_t nsteps, int32_t every) {
    if (!h) return DUGKS_E_INVAL;
    if (nsteps < 1 || every < 1) return handle_fail(h, DUGKS_E_INVAL, "record: nsteps and every must be >= 1");
    int rc = check_adjoint_support(h);
    if (rc != DUGKS_OK) return rc;
    if (h->step + nsteps > 2147483647LL) return handle_fail(h, DUGKS_E_INVAL, "record: step index past 2^31 - 1");
    AdjointTape &t = h->tape;
    t.steps = 0;
    // an earlier asynchronous adjoint may still read the buffers reused below
    cudaError_t es0 = cudaStreamSynchronize(h->stream);
    if (es0 != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "record: %s", cudaGetErrorString(es0));
    const int64_t nseg = (nsteps + every - 1) / every;
    const int64_t nbuf = std::min<int64_t>(every, nsteps);  // seg[0] receives the checkpoint
    cudaError_t e = cudaSuccess;
    auto resize = [&](std::vector<void *> &v, int64_t count) {
        while ((int64_t)v.size() > count) {
            cudaFree(v.back());
            v.pop_back();
        }
        while (e == cudaSuccess && (int64_t)v.size() < count) {
            void *p = nullptr;
            e = cudaMalloc(&p, h->state_bytes);
            if (e == cudaSuccess) e = cudaMemsetAsync(p, 0, h->state_bytes, h->stream);  // zero padding columns
            if (e == cudaSuccess) v.push_back(p);
            else cudaFree(p);
        }
    };
    resize(t.ckpt, nseg);
    resize(t.seg, nbuf);
    const size_t es = h->store == DUGKS_STORE_F64 ? 8 : 4;
    if (e == cudaSuccess && !t.scratch) {
        t.scratch_bytes = scratch_bytes(h->nx, h->ny, es);
        e = cudaMalloc(&t.scratch, t.scratch_bytes);
        if (e == cudaSuccess) e = cudaMalloc((void **)&t.dG, sizeof(double) * 2 * h->ncell);
        if (e == cudaSuccess) e = cudaMalloc((void **)&t.dW, sizeof(double) * 4 * (h->nx + h->ny));
        if (e == cudaSuccess) e = cudaMalloc((void **)&t.zero, sizeof(long long));
        if (e == cudaSuccess) e = cudaMalloc((void **)&t.dW_face, sizeof(double) * 18);
        if (e == cudaSuccess) e = cudaMallocHost((void **)&t.h_wall, sizeof(double) * 18);
        if (e == cudaSuccess) e = cudaMemsetAsync(t.zero, 0, sizeof(long long), h->stream);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        adjoint_release(h);
        return handle_fail(h, e == cudaErrorMemoryAllocation ? DUGKS_E_NOMEM : DUGKS_E_CUDA, "record: %s",
                           cudaGetErrorString(e));
    }
    t.step0 = h->step;
    t.every = every;
    for (int64_t s = 0; s < nseg; s++) {
        e = cudaMemcpyAsync(t.ckpt[(size_t)s], h->buf[h->cur], h->state_bytes, cudaMemcpyDeviceToDevice, h->stream);
        if (e != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "record: %s", cudaGetErrorString(e));
        rc = dugks_step(h, std::min<int64_t>(every, nsteps - s * every));
        if (rc != DUGKS_OK) return rc;
    }
    t.steps = nsteps;
    return DUGKS_OK;
}

static int adjoint_enqueue_checked(dugks_t h, const float *dL_dmom, float *dL_dfield, void *dL_dstate0) {
    if (!h || !dL_dmom) return DUGKS_E_INVAL;
    int rc = check_adjoint_support(h);
    if (rc != DUGKS_OK) return rc;
    if (h->tape.steps < 1) return handle_fail(h, DUGKS_E_INVAL, "adjoint: no recorded rollout (call dugks_record)");
    // the previous call's graphs and buffers are reused: its work must have completed
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "adjoint: %s", cudaGetErrorString(e));
    return h->store == DUGKS_STORE_F64 ? enqueue_adjoint<double>(h, dL_dmom, dL_dfield, dL_dstate0)
                                       : enqueue_adjoint<float>(h, dL_dmom, dL_dfield, dL_dstate0);
}

extern "C" int dugks_adjoint_async(dugks_t h, const float *dL_dmom, float *dL_dfield, void *dL_dstate0) {
    return adjoint_enqueue_checked(h, dL_dmom, dL_dfield, dL_dstate0);
}

extern "C" int dugks_adjoint_wall(dugks_t h, double *dL_dwall) {
    if (!h || !dL_dwall) return DUGKS_E_INVAL;
    if (!h->tape.h_wall) return handle_fail(h, DUGKS_E_INVAL, "adjoint_wall: no adjoint has run");
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "adjoint_wall: %s", cudaGetErrorString(e));
    for (int i = 0; i < 18; i++) dL_dwall[i] = h->tape.h_wall[i];
    return DUGKS_OK;
}

extern "C" int dugks_adjoint(dugks_t h, const float *dL_dmom, float *dL_dfield, double *dL_dwall,
                             void *dL_dstate0) {
    int rc = adjoint_enqueue_checked(h, dL_dmom, dL_dfield, dL_dstate0);
    if (rc != DUGKS_OK) return rc;
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return handle_fail(h, DUGKS_E_CUDA, "adjoint: %s", cudaGetErrorString(e));
    if (dL_dwall)
        for (int i = 0; i < 18; i++) dL_dwall[i] = h->tape.h_wall[i];
    return DUGKS_OK;
}
