// dugks_step2d.cuh -- throughput kernel of the fused DUGKS time step for the D2Q9 velocity
// set on sm_103a, FP32 arithmetic, F32 and F16 storage (BF16, and meshes whose step is the latency of a
// block: dugks_step2d_cell.cuh; the rule stands in step2d_q9.cu).
//
// Same scheme and readings as the reference kernel in dugks_step.cuh (Appendix steps 1-10
// of arXiv 1411.6121). What bounds a 2D step is instruction issue, so the work is arranged to
// need few instructions per cell:
//
//  * A block is 32 x RY threads, one warp per row of 64 columns, two neighbouring columns per
//    lane; the inner 60 x (RY - 2) cells are updated, the rest is halo. The two cells of a lane are
//    the halves of a float2 and all arithmetic uses the packed FP32 instructions (two FP32
//    operations each, rounded as the scalar ones). Neighbours along x come by shuffles; along
//    y each row publishes what its neighbours read in shared memory, behind the only barrier
//    of a tile without y walls.
//  * The update of a cell is split into a part linear in fbar+ and the equilibrium (and force)
//    part of the interface values. With phi = fbar+ and, at an interface, f = (1 - b7) F + W Y
//    (step 7; F the step-4 value, Y the bracket of b7 f_eq + c7 S), the microflux divergence of
//    velocity k is (1 - b7) La + W N with
//      La = sum_d e_d [F(+d) - F(-d)]
//         = e_x (phi_E - phi_W)/2 - kappa (phi_E - 2 phi + phi_W) + (the same along y)
//           - kappa/2 e_x e_y [(phi_NE - phi_NW) - (phi_SE - phi_SW)]      (steps 3-4, 8)
//    formed per velocity from differences of neighbouring cells, and N = sum_d e_d [Y(+d) - Y(-d)].
//    No step-4 value is formed at an inner interface.
//  * Y needs the interface moments only (step 6), which are formed in moment space from the cells'
//    moments: A(L) + B(R) with A, B = M/2 +- kappa M_d - kappa/4 dt M_t. Without a force the
//    brackets of all six crossing velocities are polynomials of five numbers per interface,
//      P = base + 4.5 m_n^2/rho0, R = P + 4.5 m_t^2/rho0, S = 9 m_n m_t/rho0, m_n, m_t,
//    (n the normal, t the tangential axis), so a cell takes the differences of those five
//    across its two pairs of interfaces and combines them. With a force the six brackets
//    themselves are differenced. Both cells of an interface use the same numbers, so the
//    equilibrium flux telescopes exactly.
//  * At a wall interface step 5 replaces the incoming velocities' F: the interface moments get
//    the sum of the changes, and the cell's La the changes themselves.
//  * The update adds (1 - b7) La + b7 W N with both coefficients rounded on their own. Error of the state / of u
//    against FP64 over that of the one-cell kernel (dugks_step2d_cell.cuh), geometric means over 64 random
//    meshes (8 to 200 cells a side, six kinds of flow): 20 steps 0.94 / 0.93, 200 0.98 / 0.95, 1000 0.92 / 0.88. The
//    increment form with split weights of dugks_step3d_ws27.cuh gave 0.92 / 0.91, 0.95 / 0.95, 0.91 / 0.88 for 1% of a
//    batch's time.
// Measured (us per step, one instance, before / now; before: one cell per thread, 32 x 8 threads, 30
// warp instructions per cell, 56% issue): 1024^2 cavity 40.0 / 27.2, 2048^2 155 / 102 (15.4 instructions
// per cell, 54% issue, 24 warps per SM), 512 x 256 channel 8.8 / 6.8, 8 x 32 channel 3.45 / 3.2 (the
// latency of one block).
#pragma once

#include "dugks_step.cuh"

namespace dugks {

namespace m2 {

constexpr int TXI = 60;  // columns a tile updates
// What a row publishes, in float2 per lane: fbar+ of the six velocities with e_y != 0, the x
// differences of the four diagonals, M_y, M_xy, M_yy, the parts A and B of its y interfaces
// (drho, j_y, j_x); all linear in fbar+. Then what only the row itself reads: the other
// fbar+ with e_x != 0 (x walls) and u0 of its update; and, with a force, the acceleration field.
constexpr int PF = 0, PDX = 6, PM = 10, PA = 13, PB = 16, PX = 19, PU = 21, PFLD = 30;
template <bool FORCE>
constexpr int slots() { return FORCE ? PFLD + 2 : PFLD; }
template <bool FORCE>
constexpr size_t smem_bytes(int ry) { return sizeof(float2) * 32 * slots<FORCE>() * ry; }
constexpr int MAX_RY = 16;
// 80 registers per thread: three blocks of 256 threads (ry 8) or two of 384 (ry 12) per SM
constexpr int REG_THREADS = 768;

using V = float2;
__device__ __forceinline__ V bc(float x) { return make_float2(x, x); }
__device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ V sub(V a, V b) {
    V r;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; sub.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
// values of the next and the previous column
__device__ __forceinline__ V east(V v) { return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1)); }
__device__ __forceinline__ V west(V v) { return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x); }
// east - west
__device__ __forceinline__ V cdx(V v) {
    return make_float2(__fsub_rn(v.y, __shfl_up_sync(0xffffffffu, v.y, 1)),
                       __fsub_rn(__shfl_down_sync(0xffffffffu, v.x, 1), v.x));
}

__host__ __device__ constexpr int ex(int k) { return Lat<9>::e(k, 0); }
__host__ __device__ constexpr int ey(int k) { return Lat<9>::e(k, 1); }
// position of the diagonal k among 0, 2, 6, 8
__host__ __device__ constexpr int di(int k) { return k < 3 ? k / 2 : k / 2 - 1; }
// position of k among the six with e_y != 0 (0, 2, 3, 5, 6, 8)
__host__ __device__ constexpr int yi(int k) { return k - k / 3 - (k % 3 == 2); }

// Moment slots: 0 M0, 1 M_x, 2 M_y, 3 M_xx, 4 M_yy, 5 M_xy.
struct Row {
    V f[9], m[6], fld[2];  // fbar+, its moments, the cells' acceleration field
};

// What a lane knows of its strip: its first column gx0 (the second is gx0 + 1), the columns it
// loads (wrapped on a periodic axis, the nearest cell beyond a wall) and where x ghosts lie.
struct Strip {
    int lane, gx0, ca, cb;
    bool vec;       // every lane's two columns load as one aligned pair (the same in all lanes)
    bool xlo, xhi;  // the strip holds the ghost column below / above an x wall
};

__device__ __forceinline__ int column(int gx, int nx, bool per) {
    if (gx >= 0 && gx < nx) return gx;
    if (per) {
        const int r = gx % nx;
        return r < 0 ? r + nx : r;
    }
    return gx < 0 ? 0 : nx - 1;
}

__device__ __forceinline__ Strip make_strip(const StepParams &p, int x0) {
    Strip s;
    const bool per = p.bc[0] == 0;
    s.lane = threadIdx.x & 31;
    s.gx0 = x0 - 2 + 2 * s.lane;
    s.ca = column(s.gx0, p.nx, per);
    s.cb = column(s.gx0 + 1, p.nx, per);
    s.vec = __all_sync(0xffffffffu, s.cb == s.ca + 1 && (s.ca & 1) == 0);
    s.xlo = !per && x0 == 0;
    s.xhi = !per && x0 + TXI >= p.nx;
    return s;
}

__device__ __forceinline__ V unpack2(uint32_t w) {  // two F16 values
    return mul(__half22float2(*reinterpret_cast<const __half2 *>(&w)), bc(F16_UNSCALE));
}

// The two values as stored, each rounded as store_state rounds it (the low 13 bits of its random bits
// r added below the kept significand, then truncated), the first in the low half.
__device__ __forceinline__ uint32_t f16_pair(V v, uint32_t r0, uint32_t r1) {
    const V t = mul(v, bc(F16_SCALE));
    uint32_t d;
    asm("cvt.rz.f16x2.f32 %0, %1, %2;"
        : "=r"(d)
        : "f"(__uint_as_float(__float_as_uint(t.y) + (r1 & 0x1fffu))), "f"(__uint_as_float(__float_as_uint(t.x) + (r0 & 0x1fffu))));
    return d;
}

// The lane's stored values of row y (a real row).
template <class S>
__device__ __forceinline__ void load_row(const StepParams &p, const Strip &s, int y, V g[9]) {
    const S *row = reinterpret_cast<const S *>(p.src) + (int64_t)y * p.px;
    if (s.vec) {
#pragma unroll
        for (int k = 0; k < 9; k++) {
            if constexpr (sizeof(S) == 4) g[k] = ld_chained(reinterpret_cast<const float2 *>(row + k * p.dstride + s.ca));
            else g[k] = unpack2(ld_chained(reinterpret_cast<const uint32_t *>(row + k * p.dstride + s.ca)));
        }
    } else {
#pragma unroll
        for (int k = 0; k < 9; k++)
            g[k] = make_float2(Store<S>::ldc(row + k * p.dstride + s.ca), Store<S>::ldc(row + k * p.dstride + s.cb));
    }
}

// The ghost columns beyond x walls (step 2, reading R3: 2 f0 - f1).
__device__ __forceinline__ V x_ghost(V v, const Strip &s, int nx) {
    if (s.xlo) {
        const float a = __shfl_down_sync(0xffffffffu, v.x, 1), b = __shfl_down_sync(0xffffffffu, v.y, 1);
        if (s.gx0 == -2) v.y = ghost_value(a, b);
    }
    if (s.xhi) {
        const float a = __shfl_up_sync(0xffffffffu, v.y, 1), b = __shfl_up_sync(0xffffffffu, v.x, 1);
        if (s.gx0 == nx) v.x = ghost_value(a, b);
        if (s.gx0 == nx - 1) v.y = ghost_value(v.x, a);
    }
    return v;
}

// Row y (a real row) from its stored values g: step 1 (eq. (24)) with the rounding of
// moments<9, float, true> and relax, the moments of fbar+, and x ghosts. With d = fbar+ - g~,
// u0 = g~ + 4/3 d (eq. (25): 4/3 fbar+ - 1/3 g~).
template <bool FORCE>
__device__ __forceinline__ void make_row(const StepParams &p, const Coef<float> &cf, const Strip &s, int y,
                                         const V g[9], Row &r, V u0[9]) {
    V G[2] = {bc(0.0f), bc(0.0f)};
    r.fld[0] = r.fld[1] = bc(0.0f);
    if constexpr (FORCE) {
        if (p.field) {
            const float *fr = p.field + (int64_t)p.nx * y;
            const int64_t ncell = (int64_t)p.nx * p.ny;
#pragma unroll
            for (int a = 0; a < 2; a++) r.fld[a] = make_float2(__ldg(fr + a * ncell + s.ca), __ldg(fr + a * ncell + s.cb));
        }
#pragma unroll
        for (int a = 0; a < 2; a++) G[a] = mul(add(bc(p.fg[a]), r.fld[a]), bc(cf.ct));
    }
    V drho = g[0];
#pragma unroll
    for (int k = 1; k < 9; k++) drho = add(drho, g[k]);
    float ax = 0.0f, ay = 0.0f;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        if (k == 4) continue;
        ax = fmaxf(ax, fabsf(g[k].x));
        ay = fmaxf(ay, fabsf(g[k].y));
    }
    const V sp = make_float2(__uint_as_float((__float_as_uint(ax) & 0x7f800000u) + 0x02c00000u),
                             __uint_as_float((__float_as_uint(ay) & 0x7f800000u) + 0x02c00000u));
    V hi[2] = {bc(0.0f), bc(0.0f)}, lo[2] = {bc(0.0f), bc(0.0f)};
#pragma unroll
    for (int k = 0; k < 9; k++) {
        if (k == 4) continue;
        const V h = sub(add(g[k], sp), sp), l = sub(g[k], h);
        if (ex(k) > 0) { hi[0] = add(hi[0], h); lo[0] = add(lo[0], l); }
        if (ex(k) < 0) { hi[0] = sub(hi[0], h); lo[0] = sub(lo[0], l); }
        if (ey(k) > 0) { hi[1] = add(hi[1], h); lo[1] = add(lo[1], l); }
        if (ey(k) < 0) { hi[1] = sub(hi[1], h); lo[1] = sub(lo[1], l); }
    }
    V m[2];
#pragma unroll
    for (int a = 0; a < 2; a++) m[a] = add(hi[a], FORCE ? fma(G[a], bc(cf.wcell * cf.rho0), lo[a]) : lo[a]);
    const V mm = fma(m[0], m[0], mul(m[1], m[1]));
    V gm = bc(0.0f);
    if constexpr (FORCE) gm = mul(fma(G[0], m[0], mul(G[1], m[1])), bc(cf.inv_rho0));
    const V base = fma(bc(-1.5f * cf.inv_rho0), mm, drho), c45 = bc(4.5f * cf.inv_rho0);
    const V b1 = bc(cf.b1), b43 = bc(cf.b1 * (4.0f / 3.0f)), t43 = bc(4.0f / 3.0f);
    // The weights are 1/9 times 4, 1 and 1/4, so the axes' weight and its split serve all, with e.m and
    // q of the diagonals a quarter and of the rest velocity four times (exact): four constants in
    // registers instead of ten.
    constexpr double W = 1.0 / 9.0;
    constexpr float wh = (float)W, wl = (float)(W - (double)wh);
    constexpr float w3h = (float)(3.0 * W), w3l = (float)(3.0 * W - (double)w3h);
    const V qt = bc(0.25f), mq[2] = {mul(qt, m[0]), mul(qt, m[1])}, base4 = mul(qt, base), c45d = bc(18.0f * cf.inv_rho0);
    sfor<4>([&](auto jc) {
        constexpr int k = 5 + jc;  // (0, 1), (1, -1), (1, 0), (1, 1) and the opposite of each
        constexpr bool diag = ex(k) != 0 && ey(k) != 0;
        const V em = diag ? (ey(k) > 0 ? add(mq[0], mq[1]) : sub(mq[0], mq[1])) : (ex(k) == 0 ? m[1] : m[0]);
        const V q = diag ? fma(mul(c45d, em), em, base4) : fma(mul(c45, em), em, base);
        const V wq = fma(bc(wl), q, mul(bc(wh), q));
        const V en = sub(bc(0.0f), em);
        const V gp = fma(bc(w3h), em, fma(bc(w3l), em, wq)), gn = fma(bc(w3h), en, fma(bc(w3l), en, wq));
        const V dp = sub(gp, g[k]), dn = sub(gn, g[8 - k]);
        if constexpr (!FORCE) {
            r.f[k] = fma(b1, dp, g[k]);
            r.f[8 - k] = fma(b1, dn, g[8 - k]);
            u0[k] = fma(b43, dp, g[k]);
            u0[8 - k] = fma(b43, dn, g[8 - k]);
        } else {
            const V ge = ex(k) == 0 ? G[1] : (ey(k) == 0 ? G[0] : (ey(k) > 0 ? add(G[0], G[1]) : sub(G[0], G[1])));
            const V r0 = bc(diag ? 0.25f * cf.rho0 : cf.rho0);
            const V fqp = fma(bc(wh), r0, gp), fqn = fma(bc(wh), r0, gn);
            const V c3 = bc(3.0f * cf.c1), n3 = bc(-3.0f * cf.c1);
            const V ip = fma(mul(c3, sub(ge, gm)), fqp, mul(b1, dp)), in = fma(mul(n3, add(ge, gm)), fqn, mul(b1, dn));
            r.f[k] = add(g[k], ip);
            r.f[8 - k] = add(g[8 - k], in);
            u0[k] = fma(t43, ip, g[k]);
            u0[8 - k] = fma(t43, in, g[8 - k]);
        }
    });
    {
        const V b4 = mul(bc(4.0f), base), gq = fma(bc(wl), b4, mul(bc(wh), b4));
        V in = mul(b1, sub(gq, g[4]));
        if constexpr (FORCE) in = fma(mul(bc(-3.0f * cf.c1), gm), fma(bc(wh), bc(4.0f * cf.rho0), gq), in);
        r.f[4] = add(g[4], in);
        u0[4] = fma(t43, in, g[4]);
    }
    const V xp = add(add(r.f[6], r.f[7]), r.f[8]), xn = add(add(r.f[0], r.f[1]), r.f[2]);
    const V yp = add(add(r.f[2], r.f[5]), r.f[8]), yn = add(add(r.f[0], r.f[3]), r.f[6]);
    r.m[0] = add(add(add(r.f[3], r.f[4]), r.f[5]), add(xp, xn));
    r.m[1] = sub(xp, xn);
    r.m[2] = sub(yp, yn);
    r.m[3] = add(xp, xn);
    r.m[4] = add(yp, yn);
    r.m[5] = add(sub(sub(r.f[0], r.f[2]), r.f[6]), r.f[8]);
    if (s.xlo || s.xhi) {  // warp-uniform; only the columns' values that x neighbours read
#pragma unroll
        for (int k = 0; k < 9; k++)
            if (ex(k) != 0) r.f[k] = x_ghost(r.f[k], s, p.nx);
#pragma unroll
        for (int i = 0; i < 6; i++) r.m[i] = x_ghost(r.m[i], s, p.nx);
    }
}

// Per-cell parts of the moments at the interface normal to n (mn, mt: slots of M_n, M_t; mnn,
// mnt: of M_nn, M_nt), in the order drho, j_n, j_t; D: differences along t of (M_t, M_nt, M_tt).
template <int SIGN>
__device__ __forceinline__ void moment_parts(float kappa, V m0, V mn, V mt, V mnn, V mnt, const V D[3], V out[3]) {
    const V h = bc(0.5f), k = bc(SIGN > 0 ? kappa : -kappa), q = bc(-0.25f * kappa);
    out[0] = fma(h, m0, fma(k, mn, mul(q, D[0])));
    out[1] = fma(h, mn, fma(k, mnn, mul(q, D[1])));
    out[2] = fma(h, mt, fma(k, mnt, mul(q, D[2])));
}
__device__ __forceinline__ void x_diffs(const V m[6], V D[3]) {  // of (M_x, M_xy, M_xx)
    D[0] = cdx(m[1]);
    D[1] = cdx(m[5]);
    D[2] = cdx(m[3]);
}

// The numbers of an interface that its two cells difference (header): without a force P, R, S,
// m_n, m_t; with one the brackets Y of the six crossing velocities (n, t) = (1, 0), (-1, 0),
// (1, 1), (-1, -1), (1, -1), (-1, 1). fm: drho, j_n, j_t; Gn, Gt: the acceleration / c there.
template <bool FORCE>
__device__ __forceinline__ void face_numbers(const Coef<float> &cf, const V fm[3], V Gn, V Gt, V out[6]) {
    const float c45 = 4.5f * cf.inv_rho0;
    V mn = fm[1], mt = fm[2];
    if constexpr (FORCE) {
        const V w = bc(cf.wface * cf.rho0);
        mn = fma(Gn, w, mn);
        mt = fma(Gt, w, mt);
    }
    const V base = fma(bc(-1.5f * cf.inv_rho0), fma(mn, mn, mul(mt, mt)), fm[0]);
    const V P = fma(mul(bc(c45), mn), mn, base);
    const V R = fma(mul(bc(c45), mt), mt, P);
    const V S = mul(mul(bc(2.0f * c45), mn), mt);
    if constexpr (!FORCE) {
        out[0] = P;
        out[1] = R;
        out[2] = S;
        out[3] = mn;
        out[4] = mt;
    } else {
        // Y = b7 X + t (rho0 + X), X = f_eq / W - rho0 the velocity's even part q +- 3 e.m,
        // t = 3 c7 (G.e - G.m/rho0)
        const V c73 = bc(3.0f * cf.c7), b7 = bc(cf.b7), r0 = bc(cf.rho0);
        const V gm = mul(c73, mul(fma(Gn, mn, mul(Gt, mt)), bc(cf.inv_rho0)));
        auto pair = [&](V q, V em, V ge, V &yp, V &yn) __attribute__((always_inline)) {
            const V e3 = mul(bc(3.0f), em), g3 = mul(c73, ge);
            const V Xp = add(q, e3), Xn = sub(q, e3);
            const V tp = sub(g3, gm), tn = mul(bc(-1.0f), add(g3, gm));
            yp = fma(tp, add(r0, Xp), mul(b7, Xp));
            yn = fma(tn, add(r0, Xn), mul(b7, Xn));
        };
        pair(P, mn, Gn, out[0], out[1]);
        pair(add(R, S), add(mn, mt), add(Gn, Gt), out[2], out[3]);
        pair(sub(R, S), sub(mn, mt), sub(Gn, Gt), out[4], out[5]);
    }
}

// f_eq deviation of velocity k over the cells (geq_k).
template <int k>
__device__ __forceinline__ V geq2(const Coef<float> &cf, V dr, V mx, V my) {
    const float ir = cf.inv_rho0;
    const V mm = fma(mx, mx, mul(my, my));
    V em = bc(0.0f);
    if (ex(k) > 0) em = mx;
    if (ex(k) < 0) em = mul(bc(-1.0f), mx);
    if (ey(k) > 0) em = ex(k) ? add(em, my) : my;
    if (ey(k) < 0) em = ex(k) ? sub(em, my) : mul(bc(-1.0f), my);
    const V x = fma(em, bc(3.0f), fma(mul(bc(ir), em), mul(bc(4.5f), em), fma(bc(-1.5f * ir), mm, dr)));
    constexpr double W = Lat<9>::wt<double>(k);
    constexpr float wh = (float)W, wl = (float)(W - (double)wh);
    return fma(bc(wl), x, mul(bc(wh), x));
}

// Step 5 for the incoming velocities (e_x -1, 0, 1) of a y wall: their new values minus the step-4 ones.
// Fi, Fo: step-4 values of the incoming velocities and of their opposites at the wall; Fc at x_c; cm:
// drho, j_y, j_x at x_c; Gcy, Gcx: acceleration / c there. Adds the change to the wall's moments wm
// (drho, j_y, j_x).
template <int side, bool FORCE>
__device__ __forceinline__ void wall_change(const StepParams &p, const Coef<float> &cf, const V Fi[3], const V Fo[3],
                                            const V Fc[3], const V cm[3], V Gcy, V Gcx, V wm[3], V dF[3]) {
    constexpr int wid = 2 + side, sg = side == 0 ? 1 : -1;  // sg: the incoming velocities' e_y
    const float *mw = p.fwm[wid];
    V my = cm[1], mx = cm[2];
    if constexpr (FORCE) {
        const V w = bc(cf.wface * cf.rho0);
        my = fma(Gcy, w, my);
        mx = fma(Gcx, w, mx);
    }
    const int type = p.bc[wid];
    const bool vel = type == 1;
    const V dra = vel ? cm[0] : bc(wall_drho<float>(p, cf, wid));
    const V m_ay = vel ? bc(mw[1]) : my, m_ax = vel ? bc(mw[0]) : mx;
    sfor<3>([&](auto ic) {
        constexpr int i = ic, t = i - 1, k = 3 * (t + 1) + sg + 1;
        V v;
        if (type == 3) {
            const float em = (float)sg * mw[1] + (float)t * mw[0];
            v = add(Fo[i], bc(wmul<9, float>(k, 6.0f * em)));
        } else {
            v = add(geq2<k>(cf, dra, m_ax, m_ay), sub(Fc[i], geq2<k>(cf, cm[0], mx, my)));
        }
        dF[i] = sub(v, Fi[i]);
    });
    const V s = add(add(dF[0], dF[1]), dF[2]);
    wm[0] = add(wm[0], s);
    wm[1] = sg > 0 ? add(wm[1], s) : sub(wm[1], s);
    wm[2] = add(wm[2], sub(dF[2], dF[0]));
}

// Step 5 of a y wall (side 0: y = 0, 1: y = ny), done by the warp of the ghost row beyond it, which
// has nothing else to do while the tile's rows form their x interfaces. own: the lane's slots of
// the ghost row. Into its u0 slots go the wall interface's moments (drho, j_y, j_x) and the changes of
// the incoming velocities (e_x = -1, 0, 1).
template <int side, bool FORCE>
__device__ __forceinline__ void y_wall(const StepParams &p, const Coef<float> &cf, V *own) {
    constexpr int NS = slots<FORCE>(), dw = side == 0 ? 0 : -1, dc = side == 0 ? 1 : -2;  // low rows of the wall, of x_c
    const float kap = cf.kappa;
    auto pub = [&](int dr, int i) __attribute__((always_inline)) -> V & { return own[(dr * NS + i) * 32]; };
    auto value = [&](int dr, auto kc) __attribute__((always_inline)) -> V {  // step 4, rows dr and dr + 1
        constexpr int k = decltype(kc)::value;
        const V l = pub(dr, PF + yi(k)), r = pub(dr + 1, PF + yi(k));
        V v = fma(bc(-kap * (float)ey(k)), sub(r, l), mul(bc(0.5f), add(l, r)));
        if constexpr (ex(k) != 0)
            v = fma(bc(-0.25f * kap * (float)ex(k)), add(pub(dr, PDX + di(k)), pub(dr + 1, PDX + di(k))), v);
        return v;
    };
    V Fi[3], Fo[3], Fc[3], wm[3], cm[3], dF[3], Gc[2] = {bc(0.0f), bc(0.0f)};
    sfor<3>([&](auto ic) {
        constexpr int i = ic, k = 3 * i + (side == 0 ? 2 : 0);
        Fi[i] = value(dw, std::integral_constant<int, k>{});
        Fo[i] = value(dw, std::integral_constant<int, 8 - k>{});
        Fc[i] = value(dc, std::integral_constant<int, k>{});
        wm[i] = add(pub(dw, PA + i), pub(dw + 1, PB + i));
        cm[i] = add(pub(dc, PA + i), pub(dc + 1, PB + i));
    });
    if constexpr (FORCE) {
#pragma unroll
        for (int c = 0; c < 2; c++)
            Gc[c] = mul(add(bc(p.fg[c]), mul(bc(0.5f), add(pub(dc, PFLD + c), pub(dc + 1, PFLD + c)))), bc(cf.cth));
    }
    wall_change<side, FORCE>(p, cf, Fi, Fo, Fc, cm, Gc[1], Gc[0], wm, dF);
#pragma unroll
    for (int i = 0; i < 3; i++) {
        pub(0, PU + i) = wm[i];
        pub(0, PU + 3 + i) = dF[i];
    }
}

// Step 5 for the columns at x walls (own: the lane's slots of its row): column 0's -x and column
// nx - 1's +x interface. Both walls' lanes run the same code at once, with the side (sg: the incoming
// velocities' e_x) as data.
struct XWall {
    V fe[3], fw[3], Ge[2], Gw[2];  // in/out: moments at the columns' x interfaces; in: G there (n, t)
    V lo[3], hi[3];                // out: changes at column 0's -x and column nx - 1's +x interface
};
template <bool FORCE>
__device__ __forceinline__ void x_wall(const StepParams &p, const Coef<float> &cf, const Strip &s, const V *own, XWall &w) {
    constexpr int NS = slots<FORCE>();
    const float kap = cf.kappa, ir = cf.inv_rho0;
    auto pub = [&](int dr, int i) __attribute__((always_inline)) -> const V & { return own[(dr * NS + i) * 32]; };
    // step-4 values of the six crossing velocities at the +x interface of every column
    V F[9];
    sfor<9>([&](auto kc) {
        constexpr int k = kc;
        if constexpr (ex(k) != 0) {
            const V l = pub(0, ey(k) != 0 ? PF + yi(k) : PX + k / 7), r = east(l);
            V v = fma(bc(-kap * (float)ex(k)), sub(r, l), mul(bc(0.5f), add(l, r)));
            if constexpr (ey(k) != 0) {
                const V C = sub(pub(1, PF + yi(k)), pub(-1, PF + yi(k)));
                v = fma(bc(-0.25f * kap * (float)ey(k)), add(C, east(C)), v);
            }
            F[k] = v;
        }
    });
#pragma unroll
    for (int i = 0; i < 3; i++) w.lo[i] = w.hi[i] = bc(0.0f);
    const bool at0 = s.gx0 == p.nx - 1, at1 = s.gx0 + 1 == p.nx - 1;
    bool lo = s.xlo && s.gx0 == 0, hi = s.xhi && (at0 || at1);
    // a lane with both walls (nx = 2) takes a second pass
    for (bool both = __any_sync(0xffffffffu, lo && hi);; both = false) {
        const bool l = lo;
        const float sg = l ? 1.0f : -1.0f;
        const int wid = l ? 0 : 1, type = p.bc[wid];
        // the wall's and x_c's values: column 0's -x and +x interfaces, column nx - 1's +x and -x ones
        auto pick = [&](V e, V we, bool wall) __attribute__((always_inline)) {
            const V v = wall == l ? we : e;
            return l || at0 ? v.x : v.y;
        };
        float Fi[3], Fo[3], Fc[3], cm[3], wm[3], Gc[2];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const V a = F[i], b = F[6 + i], wa = west(a), wb = west(b);  // e_x = -1, +1 with e_y = i - 1
            Fi[i] = l ? pick(b, wb, true) : pick(a, wa, true);
            Fc[i] = l ? pick(b, wb, false) : pick(a, wa, false);
            const V oa = F[2 - i], ob = F[8 - i], woa = west(oa), wob = west(ob);  // the opposites
            Fo[i] = l ? pick(oa, woa, true) : pick(ob, wob, true);
            wm[i] = pick(w.fe[i], w.fw[i], true);
            cm[i] = pick(w.fe[i], w.fw[i], false);
        }
#pragma unroll
        for (int c = 0; c < 2; c++) Gc[c] = pick(w.Ge[c], w.Gw[c], false);
        if (lo || hi) {
            const float *mw = p.fwm[wid];
            float mc[2] = {cm[1], cm[2]};
            if constexpr (FORCE) {
                mc[0] = fmaf(Gc[0], cf.wface * cf.rho0, mc[0]);
                mc[1] = fmaf(Gc[1], cf.wface * cf.rho0, mc[1]);
            }
            const bool vel = type == 1;
            const float dra = vel ? cm[0] : wall_drho<float>(p, cf, wid);
            const float ma[2] = {vel ? mw[0] : mc[0], vel ? mw[1] : mc[1]};
            const float ba = fmaf(-1.5f * ir, fmaf(ma[0], ma[0], ma[1] * ma[1]), dra);
            const float bcc = fmaf(-1.5f * ir, fmaf(mc[0], mc[0], mc[1] * mc[1]), cm[0]);
            float d[3], sum = 0.0f;
            sfor<3>([&](auto ic) {
                constexpr int i = ic, t = i - 1;
                constexpr double W = t == 0 ? 1.0 / 9.0 : 1.0 / 36.0;
                constexpr float wh = (float)W, wl = (float)(W - (double)wh);
                auto geq = [&](const float *m, float b) __attribute__((always_inline)) {
                    const float em = fmaf((float)t, m[1], sg * m[0]);
                    const float x = fmaf(em, 3.0f, fmaf(ir * em, 4.5f * em, b));
                    return fmaf(wl, x, wh * x);
                };
                const float em6 = 6.0f * (sg * mw[0] + (float)t * mw[1]);
                const float v = type == 3 ? Fo[i] + fmaf(wl, em6, wh * em6) : geq(ma, ba) + (Fc[i] - geq(mc, bcc));
                d[i] = v - Fi[i];
                sum += d[i];
            });
            wm[0] += sum;
            wm[1] = fmaf(sg, sum, wm[1]);
            wm[2] += d[2] - d[0];
#pragma unroll
            for (int i = 0; i < 3; i++) {
                if (l) { w.fw[i].x = wm[i]; w.lo[i].x = d[i]; }
                else if (at0) { w.fe[i].x = wm[i]; w.hi[i].x = d[i]; }
                else { w.fe[i].y = wm[i]; w.hi[i].y = d[i]; }
            }
        }
        if (!both) break;
        hi = lo && hi;  // the second pass: the lanes whose other wall is left
        lo = false;
    }
}

// With a force it is kept out of line: inlined, the tile spills at 80 registers.
template <bool FORCE>
__device__ __noinline__ void x_wall_call(const StepParams &p, const Strip s, const V *own, XWall &w) {
    const Coef<float> cf(p);
    x_wall<FORCE>(p, cf, s, own, w);
}

// One tile: columns [x0, x0 + 60) x rows [y0, y0 + RY - 2) of the instance p, by a block of 32 x RY
// threads; sm: smem_bytes(RY). Called by every thread of the block.
template <class S, bool FORCE>
__device__ __forceinline__ void tile(const StepParams &p, V *sm, int x0, int y0) {
    constexpr int NN = FORCE ? 6 : 5, NS = slots<FORCE>();
    const Coef<float> cf(p);
    const Strip s = make_strip(p, x0);
    const int ny = p.ny, ry = blockDim.y, row = threadIdx.y, gy = y0 - 1 + row;
    const bool pery = p.bc[2] == 0;
    const float kap = cf.kappa;
    V *own = sm + row * NS * 32 + s.lane;  // this row's published values
    auto pub = [&](int dr, int i) __attribute__((always_inline)) -> V & { return own[(dr * NS + i) * 32]; };
    const bool real = (gy >= 0 && gy < ny) || (pery && gy >= -1 && gy <= ny);
    const bool upd = row >= 1 && row <= ry - 2 && gy < ny;
    const V ca = bc(0.5f - kap), cb = bc(0.5f + kap), ch = bc(0.5f * kap), cn = bc(-0.5f * kap);

    uint32_t seed = 0;  // stochastic rounding of F16 stores
    if constexpr (sizeof(S) == 2) seed = store_seed(*p.step_ctr + p.step_off);

    // ---- step 1 and what needs the own row only: La's x part, the y interfaces' parts ----
    Row n;
    V La[9];
    if (real) {
        const int y = wrap_idx(gy, ny);
        {
            V g[9], u0[9];
            load_row<S>(p, s, y, g);
            make_row<FORCE>(p, cf, s, y, g, n, u0);
#pragma unroll
            for (int k = 0; k < 9; k++) pub(0, PU + k) = u0[k];
        }
        sfor<9>([&](auto kc) {
            constexpr int k = kc;
            if constexpr (ex(k) != 0) {
                const V e = east(n.f[k]), w = west(n.f[k]);
                const V dE = ex(k) > 0 ? sub(e, n.f[k]) : sub(n.f[k], e);
                const V dW = ex(k) > 0 ? sub(n.f[k], w) : sub(w, n.f[k]);
                La[k] = fma(ex(k) > 0 ? ca : cb, dE, mul(ex(k) > 0 ? cb : ca, dW));
                if constexpr (ey(k) != 0) pub(0, PDX + di(k)) = sub(e, w);
            }
            if constexpr (ey(k) != 0) pub(0, PF + yi(k)) = n.f[k];
            else if constexpr (k != 4) pub(0, PX + k / 7) = n.f[k];
        });
        V Dx[3], A[3];
        x_diffs(n.m, Dx);
        moment_parts<1>(kap, n.m[0], n.m[2], n.m[1], n.m[4], n.m[5], Dx, A);
#pragma unroll
        for (int i = 0; i < 3; i++) pub(0, PA + i) = A[i];
        moment_parts<-1>(kap, n.m[0], n.m[2], n.m[1], n.m[4], n.m[5], Dx, A);
#pragma unroll
        for (int i = 0; i < 3; i++) pub(0, PB + i) = A[i];
        pub(0, PM) = n.m[2];
        pub(0, PM + 1) = n.m[5];
        pub(0, PM + 2) = n.m[4];
        if constexpr (FORCE) {
            pub(0, PFLD) = n.fld[0];
            pub(0, PFLD + 1) = n.fld[1];
        }
    }
    const bool ywalls = !pery && (y0 == 0 || y0 + ry - 2 >= ny);  // the tile holds a ghost row
    const bool ghost = ywalls && (gy == -1 || gy == ny);
    if (ywalls) {
        __syncthreads();
        if (ghost) {  // step 2: 2 f0 - f1
            const int d = gy < 0 ? 1 : -1;
            for (int i = 0; i < PX; i++) {
                const V a = pub(d, i);
                pub(0, i) = sub(add(a, a), pub(2 * d, i));
            }
            if constexpr (FORCE) {  // a wall interface takes the one adjacent cell's acceleration
                pub(0, PFLD) = pub(d, PFLD);
                pub(0, PFLD + 1) = pub(d, PFLD + 1);
            }
        }
    }
    __syncthreads();

    // from here on the row's own fbar+ is read back where it is needed: the registers hold La and M0,
    // M_x, M_xx
    // acceleration / c at an interface: mean of the two cells (reading R2)
    auto mean = [&](int c, V a, V b) __attribute__((always_inline)) -> V {
        if constexpr (FORCE) return mul(add(bc(p.fg[c]), mul(bc(0.5f), add(a, b))), bc(cf.cth));
        else return bc(0.0f);
    };
    auto fld = [&](int dr, int c) __attribute__((always_inline)) -> V {
        if constexpr (FORCE) return pub(dr, PFLD + c);
        else return bc(0.0f);
    };
    V X[6], Y[6];  // differences of the interfaces' numbers: x (E - W), y (N - S)
    if (upd) {  // warp-uniform
        // ---- x interfaces (E, W): parts exchanged by shuffles ----
        V fe[3], fw[3], Ge[2], Gw[2];
        {
            V D[3], A[3], B[3];
            D[0] = sub(pub(1, PM), pub(-1, PM));
            D[1] = sub(pub(1, PM + 1), pub(-1, PM + 1));
            D[2] = sub(pub(1, PM + 2), pub(-1, PM + 2));
            const V my = pub(0, PM), mxy = pub(0, PM + 1);
            moment_parts<1>(kap, n.m[0], n.m[1], my, n.m[3], mxy, D, A);
            moment_parts<-1>(kap, n.m[0], n.m[1], my, n.m[3], mxy, D, B);
#pragma unroll
            for (int i = 0; i < 3; i++) {
                fe[i] = add(A[i], east(B[i]));
                fw[i] = add(west(A[i]), B[i]);
            }
        }
#pragma unroll
        for (int c = 0; c < 2; c++) {
            Ge[c] = mean(c, fld(0, c), FORCE ? east(fld(0, c)) : fld(0, c));
            Gw[c] = mean(c, FORCE ? west(fld(0, c)) : fld(0, c), fld(0, c));
        }
        if (s.xlo || s.xhi) {  // step 5 at x walls
            XWall w;
#pragma unroll
            for (int i = 0; i < 3; i++) {
                w.fe[i] = fe[i];
                w.fw[i] = fw[i];
            }
#pragma unroll
            for (int c = 0; c < 2; c++) {
                w.Ge[c] = Ge[c];
                w.Gw[c] = Gw[c];
            }
            if constexpr (FORCE) x_wall_call<FORCE>(p, s, own, w);
            else x_wall<FORCE>(p, cf, s, own, w);
#pragma unroll
            for (int i = 0; i < 3; i++) {
                fe[i] = w.fe[i];
                fw[i] = w.fw[i];
                La[i] = sub(La[i], w.hi[i]);
                La[6 + i] = sub(La[6 + i], w.lo[i]);
            }
        }
        {
            V a[6], b[6];
            face_numbers<FORCE>(cf, fe, Ge[0], Ge[1], a);
            face_numbers<FORCE>(cf, fw, Gw[0], Gw[1], b);
#pragma unroll
            for (int i = 0; i < NN; i++) X[i] = sub(a[i], b[i]);
        }
    } else if (ghost) {
        if (gy < 0) y_wall<0, FORCE>(p, cf, own);
        else y_wall<1, FORCE>(p, cf, own);
    }
    if (ywalls) __syncthreads();
    if (!upd) return;
    // ---- y interfaces (N, S): moments from the parts of the two rows ----
    V fn[3], fs[3], Gn[2], Gs[2];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        fn[i] = add(pub(0, PA + i), pub(1, PB + i));
        fs[i] = add(pub(-1, PA + i), pub(0, PB + i));
    }
#pragma unroll
    for (int c = 0; c < 2; c++) {
        Gn[c] = mean(c, fld(0, c), fld(1, c));
        Gs[c] = mean(c, fld(-1, c), fld(0, c));
    }
    // La's y part and the mixed differences
    sfor<9>([&](auto kc) {
        constexpr int k = kc;
        if constexpr (ey(k) != 0) {
            const V f = pub(0, PF + yi(k)), N = pub(1, PF + yi(k)), Sv = pub(-1, PF + yi(k));
            const V dN = ey(k) > 0 ? sub(N, f) : sub(f, N), dS = ey(k) > 0 ? sub(f, Sv) : sub(Sv, f);
            V l = mul(ey(k) > 0 ? cb : ca, dS);
            if constexpr (ex(k) != 0) {
                l = add(La[k], l);
                l = fma(ex(k) * ey(k) > 0 ? ch : cn, sub(pub(-1, PDX + di(k)), pub(1, PDX + di(k))), l);
            }
            La[k] = fma(ey(k) > 0 ? ca : cb, dN, l);
        }
    });
    // step 5 at y walls: the changes of the incoming velocities enter La and the moments
    if (ywalls && gy == 0) {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            fs[i] = pub(-1, PU + i);
            La[3 * i + 2] = sub(La[3 * i + 2], pub(-1, PU + 3 + i));
        }
    }
    if (ywalls && gy == ny - 1) {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            fn[i] = pub(1, PU + i);
            La[3 * i] = sub(La[3 * i], pub(1, PU + 3 + i));
        }
    }
    {
        V a[6], b[6];
        face_numbers<FORCE>(cf, fn, Gn[1], Gn[0], a);
        face_numbers<FORCE>(cf, fs, Gs[1], Gs[0], b);
#pragma unroll
        for (int i = 0; i < NN; i++) Y[i] = sub(a[i], b[i]);
    }
    // ---- step 8 ----
    V N[9];
    const V zero = bc(0.0f);
    if constexpr (FORCE) {
        N[7] = X[0];
        N[1] = sub(zero, X[1]);
        N[5] = Y[0];
        N[3] = sub(zero, Y[1]);
        N[8] = add(X[2], Y[2]);
        N[0] = sub(zero, add(X[3], Y[3]));
        N[6] = sub(X[4], Y[5]);
        N[2] = sub(Y[4], X[5]);
    } else {
        const V t3 = bc(3.0f), x3 = mul(t3, X[3]), y3 = mul(t3, Y[3]);
        N[7] = add(x3, X[0]);
        N[1] = sub(x3, X[0]);
        N[5] = add(y3, Y[0]);
        N[3] = sub(y3, Y[0]);
        const V o1 = add(X[1], Y[2]), o2 = add(X[2], Y[1]);
        const V e1 = add(x3, y3), e2 = mul(t3, add(X[4], Y[4]));
        const V op = add(o1, o2), om = sub(o1, o2), ep = add(e1, e2), em = sub(e1, e2);
        N[8] = add(ep, op);
        N[0] = sub(ep, op);
        N[6] = add(em, om);
        N[2] = sub(em, om);
    }
    // ---- step 9, eq. (16) ----
    const float tk = -cf.two_kappa * (FORCE ? 1.0f : cf.b7);
    const V cL = bc(-cf.two_kappa * (1.0f - cf.b7)), w1 = bc(tk * (1.0f / 9.0f)), w2 = bc(tk * (1.0f / 36.0f));
    V u0[9];
#pragma unroll
    for (int k = 0; k < 9; k++) {
        u0[k] = pub(0, PU + k);
        if (k != 4) u0[k] = add(u0[k], fma(ex(k) != 0 && ey(k) != 0 ? w2 : w1, N[k], mul(cL, La[k])));
    }
    const bool mine = s.lane >= 1 && s.lane <= TXI / 2;
    const bool upd0 = mine && s.gx0 < p.nx, upd1 = mine && s.gx0 + 1 < p.nx;
    const int64_t off = (int64_t)gy * p.px + s.gx0;
    S *o = reinterpret_cast<S *>(p.dst) + off;
    if constexpr (sizeof(S) == 4) {
        if (upd1) {
#pragma unroll
            for (int k = 0; k < 9; k++) *reinterpret_cast<float2 *>(o + k * p.dstride) = u0[k];
        } else if (upd0) {
#pragma unroll
            for (int k = 0; k < 9; k++) o[k * p.dstride] = u0[k].x;
        }
    } else {
        // F16: each value takes the random bits that it has in every kernel (CellRandom), so the noise of a
        // run does not depend on the kernel; one conversion truncates the lane's two cells
        const CellRandom rnd0(seed, off), rnd1(seed, off + 1);
        sfor<9>([&](auto kc) {
            constexpr int k = kc;
            const uint32_t w = f16_pair(u0[k], rnd0.template bits<k>(), rnd1.template bits<k>());
            if (upd1) *reinterpret_cast<uint32_t *>(o + k * p.dstride) = w;
            else if (upd0) o[k * p.dstride] = __ushort_as_half((unsigned short)(w & 0xffffu));
        });
    }
}

}  // namespace m2

// One instance on a grid of tiles.
template <class S, bool FORCE>
__global__ void __launch_bounds__(m2::REG_THREADS) fused_step2d(const __grid_constant__ StepParams p) {
    extern __shared__ __align__(16) float2 smem2[];
    chain_wait();
    m2::tile<S, FORCE>(p, smem2, blockIdx.x * m2::TXI, blockIdx.y * (blockDim.y - 2));
}

// Batched form: params holds two descriptors per instance (source/destination swapped:
// index 2 i + parity); items is the work list of (instance, x0, y0, -) tiles, largest
// instances first, one per block. Each instance takes the path with or without the force term that it
// would take alone: FORCE 0 none of them has a force, 1 all have (both with the registers of their one
// path), 2 some.
// One tile per block and the parameters read through the cache: a loop over tiles in a persistent block
// and a copy of the parameters in shared memory kept both their addresses and what the compiler hoists out
// of the loop in registers, and the tile spilled 140 bytes per thread (now 52). 64 instances of 32 x 16 to
// 512 x 256 cells, 30 x 6 tiles, us per step before / now: 155 / 134 with a field, 126 / 103 without. (Tiles of
// 14 rows, one block per SM, lose 2 to 6%; 6 rows are the default.)
template <class S, int FORCE>
__global__ void __launch_bounds__(m2::REG_THREADS) fused_step2d_batch(const StepParams *__restrict__ params,
                                                                    const int4 *__restrict__ items, int parity) {
    extern __shared__ __align__(16) float2 smem2[];
    chain_wait();
    const int4 w = __ldg(items + blockIdx.x);
    const StepParams &p = params[2 * w.x + parity];
    if constexpr (FORCE != 2) {
        m2::tile<S, FORCE != 0>(p, smem2, w.y, w.z);
    } else {
        if (p.field != nullptr || p.g[0] != 0.0 || p.g[1] != 0.0) m2::tile<S, true>(p, smem2, w.y, w.z);
        else m2::tile<S, false>(p, smem2, w.y, w.z);
    }
}

}  // namespace dugks
