// dugks_step2d_lean.cuh -- the fused DUGKS time step for D2Q9 with few arithmetic operations per
// cell, for FP64 storage and for non-uniform meshes (F32 and F64 storage) of the incompressible model.
//
// GB300 runs FP64 at a 64th of its FP32 rate (16 cycles of an SM per warp instruction), so an FP64
// step costs its FP64 instructions and nothing else. The reference kernel (dugks_step.cuh) takes
// about 2,000 per cell; this one about 380, by the following.
//  * Everything that two cells or two interfaces share is formed once: a block is 32 x RY threads,
//    one per cell (lanes along x); the inner 30 x (RY - 2) cells are updated. A thread forms its
//    cell's step 1, its +x and its +y interface; x neighbours exchange by shuffles, y neighbours
//    through shared memory.
//  * Steps 3-4 only for the six velocities that cross an interface. With w the weight of the high
//    cell, F = L + (w - h c e_n / dc) (R - L) - h c e_t / dt [T(L) + w (T(R) - T(L))], where the
//    tangential part T(f) = (1 - w-) (f - f-) + w+ (f+ - f) belongs to a cell (the difference of the
//    interface's two cross points, reading R18; w-, w+ the weights at the cell's two interfaces along
//    that axis). Uniform meshes: w = 1/2, dc = dt = dx.
//  * The interface moments in moment space, by the same formula from the cells' moments.
//  * Without a force the equilibrium part of f across a cell is combined from five numbers per
//    interface (dugks_step2d.cuh); with one, from the brackets of the crossing velocities.
// Measured (us per step, reference kernel / this one): 128^2 graded cavity F64 62 / 29, the FP64 pipe 79%
// busy with 315,344 warp instructions (616 operations per cell with the tiles' halos).
#pragma once

#include "dugks_step.cuh"

namespace dugks {

namespace lean {

constexpr int TXI = 30, MAX_RY = 8;
__host__ __device__ constexpr int ex(int k) { return Lat<9>::e(k, 0); }
__host__ __device__ constexpr int ey(int k) { return Lat<9>::e(k, 1); }
// positions among the velocities with e_x != 0 (0, 1, 2, 6, 7, 8), with e_y != 0 (0, 2, 3, 5, 6, 8), and
// among the diagonals (0, 2, 6, 8)
__host__ __device__ constexpr int xi(int k) { return k < 3 ? k : k - 3; }
__host__ __device__ constexpr int yi(int k) { return k - k / 3 - (k % 3 == 2); }
__host__ __device__ constexpr int di(int k) { return k < 3 ? k / 2 : k / 2 - 1; }
// Published per row and lane: fbar+ with e_y != 0; the six moments M0, M_x, M_y, M_xx, M_yy, M_xy; the
// x tangential parts of the diagonals and of M_x, M_xy, M_xx; then the +y interface's step-4 values
// and moments, and its numbers; the acceleration field.
constexpr int PF = 0, PM = 6, PT = 12, PFY = 19, PMY = 25, PN = 28, PFLD = 34;
template <bool FORCE>
constexpr int slots() { return FORCE ? PFLD + 2 : PFLD; }
template <class T, bool FORCE>
constexpr size_t smem_bytes(int ry) { return sizeof(T) * 32 * slots<FORCE>() * ry; }

template <class T>
__device__ __forceinline__ T up1(T v) { return __shfl_up_sync(0xffffffffu, v, 1); }
template <class T>
__device__ __forceinline__ T down1(T v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// The numbers of an interface from its moments fm (drho, j_n, j_t) and acceleration / c (dugks_step2d.cuh).
template <class T, bool FORCE>
__device__ __forceinline__ void face_numbers(const Coef<T> &cf, const T fm[3], T Gn, T Gt, T out[6]) {
    const T c45 = T(4.5) * cf.inv_rho0;
    T mn = fm[1], mt = fm[2];
    if constexpr (FORCE) {
        mn = fmaT(Gn, cf.wface * cf.rho0, mn);
        mt = fmaT(Gt, cf.wface * cf.rho0, mt);
    }
    const T base = fmaT(T(-1.5) * cf.inv_rho0, fmaT(mn, mn, mt * mt), fm[0]);
    const T s = c45 * mn, P = fmaT(s, mn, base), R = fmaT(c45 * mt, mt, P), S = (s + s) * mt;
    if constexpr (!FORCE) {
        out[0] = P;
        out[1] = R;
        out[2] = S;
        out[3] = mn;
        out[4] = mt;
    } else {
        const T c73 = T(3) * cf.c7, gm = c73 * (fmaT(Gn, mn, Gt * mt) * cf.inv_rho0);
        auto pair = [&](T q, T em, T ge, T &yp, T &yn) __attribute__((always_inline)) {
            const T Xp = fmaT(T(3), em, q), Xn = fmaT(T(-3), em, q), g3 = c73 * ge;
            yp = fmaT(g3 - gm, cf.rho0 + Xp, cf.b7 * Xp);
            yn = fmaT(-g3 - gm, cf.rho0 + Xn, cf.b7 * Xn);
        };
        pair(P, mn, Gn, out[0], out[1]);
        pair(R + S, mn + mt, Gn + Gt, out[2], out[3]);
        pair(R - S, mn - mt, Gn - Gt, out[4], out[5]);
    }
}

// Step 5 at a wall of side sg (the incoming velocities' e_n: +1 low wall, -1 high) with the wall's
// face index wid normal to axis d: F[i], t = i - 1, of the incoming velocities and the moments fm of
// the wall interface are replaced. Fo: the opposites at the wall; Fc, cm, Gc: x_c's values, moments and
// acceleration / c (n, t).
template <class T, bool FORCE, int d>
__device__ __forceinline__ void wall_face(const StepParams &p, const Coef<T> &cf, int wid, T sg, const T Fo[3],
                                          const T Fc[3], const T cm[3], T Gcn, T Gct, T F[3], T fm[3]) {
    const T ir = cf.inv_rho0;
    T mw[2];
    if constexpr (sizeof(T) == 4) {
        mw[0] = p.fwm[wid][d];
        mw[1] = p.fwm[wid][1 - d];
    } else {
        mw[0] = p.bc_u[wid][d] * p.rho0 * p.inv_c;
        mw[1] = p.bc_u[wid][1 - d] * p.rho0 * p.inv_c;
    }
    T mc[2] = {cm[1], cm[2]};
    if constexpr (FORCE) {
        mc[0] = fmaT(Gcn, cf.wface * cf.rho0, mc[0]);
        mc[1] = fmaT(Gct, cf.wface * cf.rho0, mc[1]);
    }
    const int type = p.bc[wid];
    const bool vel = type == 1;
    const T dra = vel ? cm[0] : wall_drho<T>(p, cf, wid);
    const T ma[2] = {vel ? mw[0] : mc[0], vel ? mw[1] : mc[1]};
    const T ba = fmaT(T(-1.5) * ir, fmaT(ma[0], ma[0], ma[1] * ma[1]), dra);
    const T bcc = fmaT(T(-1.5) * ir, fmaT(mc[0], mc[0], mc[1] * mc[1]), cm[0]);
    T dv[3], sum = T(0);
    sfor<3>([&](auto ic) {
        constexpr int i = ic, t = i - 1, k = t == 0 ? 7 : 8;  // a velocity of the same weight
        auto geq = [&](const T *m, T b) __attribute__((always_inline)) {
            const T em = fmaT(sg, m[0], T(t) * m[1]);
            return wmul<9, T>(k, fmaT(em, T(3), fmaT(ir * em, T(4.5) * em, b)));
        };
        const T v = type == 3 ? Fo[i] + wmul<9, T>(k, T(6) * fmaT(sg, mw[0], T(t) * mw[1]))
                              : geq(ma, ba) + (Fc[i] - geq(mc, bcc));
        dv[i] = v - F[i];
        F[i] = v;
        sum += dv[i];
    });
    fm[0] += sum;
    fm[1] = fmaT(sg, sum, fm[1]);
    fm[2] += dv[2] - dv[0];
}

// S: storage, NU: non-uniform mesh (p.metric).
template <class S, bool NU, bool FORCE>
__global__ void __launch_bounds__(32 * MAX_RY) fused_step2d_lean(const __grid_constant__ StepParams p) {
    using T = typename Arith<S>::T;
    constexpr int NS = slots<FORCE>(), NN = FORCE ? 6 : 5;
    extern __shared__ __align__(16) unsigned char smem_lean[];
    chain_wait();
    const Coef<T> cf(p);
    const int lane = threadIdx.x, row = threadIdx.y, ry = blockDim.y;
    const int nx = p.nx, ny = p.ny, strips = (nx + TXI - 1) / TXI;
    const int x0 = (int)(blockIdx.x % (unsigned)strips) * TXI, y0 = (int)(blockIdx.x / (unsigned)strips) * (ry - 2);
    const int gx = x0 - 1 + lane, gy = y0 - 1 + row;
    const int64_t ncell = (int64_t)nx * ny;
    const bool perx = p.bc[0] == 0, pery = p.bc[2] == 0;
    const S *src = reinterpret_cast<const S *>(p.src);
    S *dst = reinterpret_cast<S *>(p.dst);
    T *own = reinterpret_cast<T *>(smem_lean) + row * NS * 32 + lane;
    auto pub = [&](int dr, int i) __attribute__((always_inline)) -> T & { return own[(dr * NS + i) * 32]; };
    // the cell a column / row takes its data from: wrapped on a periodic axis, clamped beyond a wall
    const int cx = perx ? ((gx % nx) + nx) % nx : min(max(gx, 0), nx - 1);
    const int cy = pery ? ((gy % ny) + ny) % ny : min(max(gy, 0), ny - 1);
    const bool real = (gy >= 0 && gy < ny) || (pery && gy >= -1 && gy <= ny);
    const bool ywalls = !pery && (y0 == 0 || y0 + ry - 2 >= ny);  // the tile holds a ghost row
    const bool ghost = ywalls && (gy == -1 || gy == ny);
    const bool xlo = !perx && x0 == 0, xhi = !perx && x0 + TXI >= nx;

    // metrics: weights of the high cell at the cell's two interfaces per axis, h c / (centre distance) at
    // its high one, h c / width, 2 h c / width (dt c / width)
    T wxm, wxp, wym, wyp, nxp, nyp, tx, ty, dcx, dcy;
    if constexpr (NU) {
        const T hc = (T)(0.5 * p.dt / p.inv_c);
        auto met = [&](int a, int i) __attribute__((always_inline)) { return (T)__ldg(p.metric[a] + i); };
        const int ix = min(max(gx, -1), nx - 1), iy = min(max(gy, -1), ny - 1);
        wxm = met(0, max(ix, 0));
        wxp = met(0, ix + 1);
        wym = met(1, max(iy, 0));
        wyp = met(1, iy + 1);
        nxp = hc * met(0, nx + 1 + ix + 1);
        nyp = hc * met(1, ny + 1 + iy + 1);
        tx = hc * met(0, 2 * nx + 2 + cx);
        ty = hc * met(1, 2 * ny + 2 + cy);
    } else {
        wxm = wxp = wym = wyp = T(0.5);
        nxp = nyp = tx = ty = cf.kappa;
    }
    dcx = tx + tx;
    dcy = ty + ty;

    // ---- step 1 and the x tangential parts ----
    T f[9], u0[9], m[6], Tx[7];  // Tx: diagonals, then M_x, M_xy, M_xx
    T fld[2] = {T(0), T(0)};
    // ghost columns beyond x walls (step 2): 2 f0 - f1, or linear through the two centres
    auto x_ghost = [&](T v) __attribute__((always_inline)) -> T {
        if (xlo) {
            const T a = down1(v), b = __shfl_down_sync(0xffffffffu, v, 2);
            if (gx == -1) v = NU ? fmaT((T)p.eg[0][0], b - a, a) : ghost_value(a, b);
        }
        if (xhi) {
            const T a = up1(v), b = __shfl_up_sync(0xffffffffu, v, 2);
            if (gx == nx) v = NU ? fmaT((T)p.eg[0][1], b - a, a) : ghost_value(a, b);
        }
        return v;
    };
    // T along x of the columns' values v (header)
    auto tang_x = [&](T v) __attribute__((always_inline)) -> T {
        const T e = down1(v), w = up1(v);
        return NU ? fmaT(wxp, e - v, (T(1) - wxm) * (v - w)) : T(0.5) * (e - w);
    };
    if (real) {
        {
            T g[9], Gh[3] = {T(0), T(0), T(0)}, drho, mm[3];
            const int64_t off = (int64_t)cy * p.px + cx;
#pragma unroll
            for (int k = 0; k < 9; k++) g[k] = (T)Store<S>::ldc(src + k * p.dstride + off);
            if constexpr (FORCE) {
                const int64_t c = (int64_t)cx + (int64_t)nx * cy;
                if (p.field) {
                    fld[0] = (T)__ldg(p.field + c);
                    fld[1] = (T)__ldg(p.field + ncell + c);
                }
#pragma unroll
                for (int a = 0; a < 2; a++) Gh[a] = ((sizeof(T) == 4 ? (T)p.fg[a] : (T)p.g[a]) + fld[a]) * cf.ct;
            }
            moments<9, T, true>(g, Gh, cf.wcell * cf.rho0, drho, mm);
            relax<9, T, FORCE>(g, drho, mm, Gh, cf.rho0, cf.inv_rho0, cf.b1, cf.c1, f);
#pragma unroll
            for (int k = 0; k < 9; k++) u0[k] = fmaT(T(1) / T(3), f[k] - g[k], f[k]);  // eq. (25)
        }
        const T xp = (f[6] + f[7]) + f[8], xn = (f[0] + f[1]) + f[2], yp = (f[2] + f[5]) + f[8], yn = (f[0] + f[3]) + f[6];
        m[0] = ((f[3] + f[4]) + f[5]) + (xp + xn);
        m[1] = xp - xn;
        m[2] = yp - yn;
        m[3] = xp + xn;
        m[4] = yp + yn;
        m[5] = (f[0] - f[2]) - (f[6] - f[8]);
        if (xlo || xhi) {
#pragma unroll
            for (int k = 0; k < 9; k++) f[k] = x_ghost(f[k]);
#pragma unroll
            for (int i = 0; i < 6; i++) m[i] = x_ghost(m[i]);
        }
        sfor<9>([&](auto kc) {
            constexpr int k = kc;
            if constexpr (ex(k) != 0 && ey(k) != 0) Tx[di(k)] = tang_x(f[k]);
            if constexpr (ey(k) != 0) pub(0, PF + yi(k)) = f[k];
        });
        Tx[4] = tang_x(m[1]);
        Tx[5] = tang_x(m[5]);
        Tx[6] = tang_x(m[3]);
#pragma unroll
        for (int i = 0; i < 6; i++) pub(0, PM + i) = m[i];
#pragma unroll
        for (int i = 0; i < 7; i++) pub(0, PT + i) = Tx[i];
        if constexpr (FORCE) {
            pub(0, PFLD) = fld[0];
            pub(0, PFLD + 1) = fld[1];
        }
    }
    if (ywalls) {
        __syncthreads();
        if (ghost) {  // ghost rows (step 2); everything published is linear in fbar+
            const int d = gy < 0 ? 1 : -1, sd = gy < 0 ? 0 : 1;
            for (int i = 0; i < PFY; i++) {
                const T a = pub(d, i), b = pub(2 * d, i);
                pub(0, i) = NU ? fmaT((T)p.eg[1][sd], b - a, a) : ghost_value(a, b);
            }
            if constexpr (FORCE) {  // a wall interface takes the one adjacent cell's acceleration
                pub(0, PFLD) = pub(d, PFLD);
                pub(0, PFLD + 1) = pub(d, PFLD + 1);
            }
        }
    }
    __syncthreads();

    const bool upd = row >= 1 && row <= ry - 2 && gy < ny;            // warp-uniform
    const bool yface = row <= ry - 2 && (real || gy == -1) && gy < ny;  // owns the interface above
    // acceleration / c at an interface: interpolated between the two cells (reading R2, R18)
    auto face_G = [&](int c, T a, T b, T w) __attribute__((always_inline)) -> T {
        if constexpr (FORCE)
            return ((sizeof(T) == 4 ? (T)p.fg[c] : (T)p.g[c]) + (NU ? fmaT(w, b - a, a) : T(0.5) * (a + b))) * cf.cth;
        else return T(0);
    };
    auto field = [&](int dr, int c) __attribute__((always_inline)) -> T {
        if constexpr (FORCE) return pub(dr, PFLD + c);
        else return T(0);
    };
    // ---- the +y interface: step-4 values of the crossing velocities, moments (drho, j_y, j_x) ----
    T Fy[6], my[3], Gy[2] = {T(0), T(0)};
    if (yface) {
        const T cp = wyp - nyp, cm = wyp + nyp;  // w -+ h c / dc for e_y = +-1
        sfor<9>([&](auto kc) {
            constexpr int k = kc;
            if constexpr (ey(k) != 0) {
                const T L = pub(0, PF + yi(k)), R = pub(1, PF + yi(k));
                T v = fmaT(ey(k) > 0 ? cp : cm, R - L, L);
                if constexpr (ex(k) != 0) {
                    const T a = pub(0, PT + di(k)), b = pub(1, PT + di(k));
                    const T t = NU ? fmaT(wyp, b - a, a) : T(0.5) * (a + b);
                    v = fmaT(ex(k) > 0 ? -tx : tx, t, v);
                }
                Fy[yi(k)] = v;
            }
        });
        auto moment = [&](int v, int n, int t) __attribute__((always_inline)) -> T {
            const T L = pub(0, PM + v), R = pub(1, PM + v), a = pub(0, PT + t), b = pub(1, PT + t);
            const T tt = NU ? fmaT(wyp, b - a, a) : T(0.5) * (a + b);
            return fmaT(-tx, tt, fmaT(-nyp, pub(1, PM + n) - pub(0, PM + n), fmaT(wyp, R - L, L)));
        };
        my[0] = moment(0, 2, 4);
        my[1] = moment(2, 4, 5);
        my[2] = moment(1, 5, 6);
        Gy[0] = face_G(1, field(0, 1), field(1, 1), wyp);  // (n, t)
        Gy[1] = face_G(0, field(0, 0), field(1, 0), wyp);
#pragma unroll
        for (int i = 0; i < 6; i++) pub(0, PFY + i) = Fy[i];
#pragma unroll
        for (int i = 0; i < 3; i++) pub(0, PMY + i) = my[i];
    }
    if (ywalls) {
        __syncthreads();  // x_c's values and moments, from the row next to the wall's
        if (yface && (gy == -1 || gy == ny - 1)) {
            const bool low = gy == -1;
            const int dr = low ? 1 : -1;  // the row that owns x_c
            T Fi[3], Fo[3], Fc[3], cm[3], Gc[2];
            sfor<3>([&](auto ic) {  // t = e_x = i - 1; incoming e_y = +1 (low) or -1 (high)
                constexpr int i = ic, kp = 3 * i + 2, km = 3 * i;
                Fi[i] = low ? Fy[yi(kp)] : Fy[yi(km)];
                Fo[i] = low ? Fy[yi(8 - kp)] : Fy[yi(8 - km)];
                Fc[i] = low ? pub(dr, PFY + yi(kp)) : pub(dr, PFY + yi(km));
                cm[i] = pub(dr, PMY + i);
            });
            // x_c lies between rows 0 and 1 (low) or ny - 2 and ny - 1 (high)
            const T wc = NU ? (T)__ldg(p.metric[1] + (low ? 1 : ny - 1)) : T(0.5);
            Gc[0] = low ? face_G(1, field(1, 1), field(2, 1), wc) : face_G(1, field(-1, 1), field(0, 1), wc);
            Gc[1] = low ? face_G(0, field(1, 0), field(2, 0), wc) : face_G(0, field(-1, 0), field(0, 0), wc);
            wall_face<T, FORCE, 1>(p, cf, low ? 2 : 3, low ? T(1) : T(-1), Fo, Fc, cm, Gc[0], Gc[1], Fi, my);
            sfor<3>([&](auto ic) {
                constexpr int i = ic, kp = 3 * i + 2, km = 3 * i;
                if (low) Fy[yi(kp)] = Fi[i];
                else Fy[yi(km)] = Fi[i];
            });
        }
        __syncthreads();  // everyone has read the unchanged values
        if (yface && (gy == -1 || gy == ny - 1)) {
#pragma unroll
            for (int i = 0; i < 6; i++) pub(0, PFY + i) = Fy[i];
        }
    }
    T vy[6];
    if (yface) {
        face_numbers<T, FORCE>(cf, my, Gy[0], Gy[1], vy);
#pragma unroll
        for (int i = 0; i < NN; i++) pub(0, PN + i) = vy[i];
    }
    // ---- the +x interface ----
    T Fx[6], vx[6];
    if (upd) {
        auto tang_y = [&](T v, T n, T sv) __attribute__((always_inline)) -> T {
            return NU ? fmaT(wyp, n - v, (T(1) - wym) * (v - sv)) : T(0.5) * (n - sv);
        };
        const T cp = wxp - nxp, cm = wxp + nxp;
        auto mid = [&](T a, T b) __attribute__((always_inline)) -> T { return NU ? fmaT(wxp, b - a, a) : T(0.5) * (a + b); };
        sfor<9>([&](auto kc) {
            constexpr int k = kc;
            if constexpr (ex(k) != 0) {
                T v = fmaT(ex(k) > 0 ? cp : cm, down1(f[k]) - f[k], f[k]);
                if constexpr (ey(k) != 0) {
                    const T t = tang_y(f[k], pub(1, PF + yi(k)), pub(-1, PF + yi(k)));
                    v = fmaT(ey(k) > 0 ? -ty : ty, mid(t, down1(t)), v);
                }
                Fx[xi(k)] = v;
            }
        });
        auto moment = [&](int v, int n, int t) __attribute__((always_inline)) -> T {  // t: slot of the tangential moment
            const T tt = tang_y(m[t], pub(1, PM + t), pub(-1, PM + t));
            return fmaT(-ty, mid(tt, down1(tt)), fmaT(-nxp, down1(m[n]) - m[n], fmaT(wxp, down1(m[v]) - m[v], m[v])));
        };
        T mx[3];
        mx[0] = moment(0, 1, 2);
        mx[1] = moment(1, 3, 5);
        mx[2] = moment(2, 5, 4);
        T Gx[2] = {T(0), T(0)};
        if constexpr (FORCE) {
            Gx[0] = face_G(0, fld[0], down1(fld[0]), wxp);
            Gx[1] = face_G(1, fld[1], down1(fld[1]), wxp);
        }
        if (xlo || xhi) {
            // step 5: x_c is the interface that the next lane inward owns
            T Fu[6], Fd[6], mu[3], md[3], Gu[2], Gd[2];
#pragma unroll
            for (int i = 0; i < 6; i++) {
                Fu[i] = up1(Fx[i]);
                Fd[i] = down1(Fx[i]);
            }
#pragma unroll
            for (int i = 0; i < 3; i++) {
                mu[i] = up1(mx[i]);
                md[i] = down1(mx[i]);
            }
#pragma unroll
            for (int c = 0; c < 2; c++) {
                Gu[c] = up1(Gx[c]);
                Gd[c] = down1(Gx[c]);
            }
            const bool low = gx == -1;
            if (!perx && (low || gx == nx - 1)) {
                T Fi[3], Fo[3], Fc[3], cmm[3];
#pragma unroll
                for (int i = 0; i < 3; i++) {  // incoming e_x = +1 (slots 3 + i) at the low wall, -1 (slots i) at the high
                    Fi[i] = low ? Fx[3 + i] : Fx[i];
                    Fo[i] = low ? Fx[2 - i] : Fx[5 - i];
                    Fc[i] = low ? Fd[3 + i] : Fu[i];
                    cmm[i] = low ? md[i] : mu[i];
                }
                wall_face<T, FORCE, 0>(p, cf, low ? 0 : 1, low ? T(1) : T(-1), Fo, Fc, cmm, low ? Gd[0] : Gu[0],
                                       low ? Gd[1] : Gu[1], Fi, mx);
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    if (low) Fx[3 + i] = Fi[i];
                    else Fx[i] = Fi[i];
                }
            }
        }
        face_numbers<T, FORCE>(cf, mx, Gx[0], Gx[1], vx);
    }
    __syncthreads();
    if (!upd) return;

    // ---- steps 7-9: f~(t+dt) = f~+ - sum over axes of dt c / width e_d (f(+d) - f(-d)) ----
    T X[6], Y[6];
#pragma unroll
    for (int i = 0; i < NN; i++) {
        X[i] = dcx * (vx[i] - up1(vx[i]));
        Y[i] = dcy * (vy[i] - pub(-1, PN + i));
    }
    T N[9];
    if constexpr (FORCE) {
        N[7] = X[0];
        N[1] = -X[1];
        N[5] = Y[0];
        N[3] = -Y[1];
        N[8] = X[2] + Y[2];
        N[0] = -X[3] - Y[3];
        N[6] = X[4] - Y[5];
        N[2] = Y[4] - X[5];
    } else {
        const T x3 = T(3) * X[3], y3 = T(3) * Y[3], e2 = T(3) * (X[4] + Y[4]);
        N[7] = x3 + X[0];
        N[1] = x3 - X[0];
        N[5] = y3 + Y[0];
        N[3] = y3 - Y[0];
        const T o1 = X[1] + Y[2], o2 = X[2] + Y[1], e1 = x3 + y3;
        const T op = o1 + o2, om = o1 - o2, ep = e1 + e2, em = e1 - e2;
        N[8] = ep + op;
        N[0] = ep - op;
        N[6] = em + om;
        N[2] = em - om;
    }
    const T a7 = T(1) - cf.b7, dxa = dcx * a7, dya = dcy * a7;
    const T w1 = (FORCE ? T(1) : cf.b7) * Lat<9>::wt<T>(1), w2 = (FORCE ? T(1) : cf.b7) * Lat<9>::wt<T>(0);
    const bool mine = lane >= 1 && lane <= TXI && gx < nx;
    const int64_t off = (int64_t)gy * p.px + gx;
    sfor<9>([&](auto kc) {
        constexpr int k = kc;
        T v = u0[k];
        if constexpr (k != 4) {
            T t = (ex(k) != 0 && ey(k) != 0 ? w2 : w1) * N[k];
            if constexpr (ex(k) != 0) t = fmaT(ex(k) > 0 ? dxa : -dxa, Fx[xi(k)] - up1(Fx[xi(k)]), t);
            if constexpr (ey(k) != 0) t = fmaT(ey(k) > 0 ? dya : -dya, Fy[yi(k)] - pub(-1, PFY + yi(k)), t);
            v -= t;
        }
        if (mine) Store<S>::st(dst + k * p.dstride + off, v);
    });
}

}  // namespace lean

}  // namespace dugks
