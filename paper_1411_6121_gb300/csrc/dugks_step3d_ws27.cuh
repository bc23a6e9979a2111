// dugks_step3d_ws27.cuh -- warp-specialised throughput kernel of the fused DUGKS time step for
// D3Q27 on sm_103a (FP32 arithmetic, F32/BF16/F16 storage): the scheme and readings of
// dugks_step3d.cuh, with the z march split between two groups of warps that run concurrently,
// and the arithmetic done on pairs of opposite velocities.
//
//  * Producer warps (8, one cell column each) make step 1: the state of the tile's plane arrives by
//    TMA into one shared-memory stage, each column forms fbar+ and its moments, then the ghost columns
//    and rows (step 2) and, beyond non-periodic z walls, the ghost planes.
//  * Consumer warps (8, one cell column each) do the rest for plane kz.
//  * The planes pass through a ring of four slots (fbar+ and moments). u0 = 4/3 fbar+ - 1/3 g~ of the update
//    has no room beside them: the consumers read g~ a second time. Each ring slot has a "full" mbarrier (every producer thread arrives after its last write of the
//    plane) and an "empty" one (every consumer thread arrives after its last read), so neither
//    group waits on a CTA-wide barrier: the producer runs up to two planes ahead. The consumers'
//    y exchange and the producers' ghost passes use named barriers of their own group.
//
// What bounds the kernel is instruction issue and its latency, so the consumers' part is arranged to
// need few instructions. At an interface f = (1 - b7) F + W Y (step 7; F the step-4 value, Y the
// bracket of b7 f_eq + c7 S), so the microflux divergence of velocity k is (1 - b7) La + W N:
//   La = sum_d e_d [F(+d) - F(-d)]
//      = sum_d [e_d (phi_+d - phi_-d)/2 - kappa (phi_+d - 2 phi + phi_-d)]
//        - kappa/2 sum_{a<b} e_a e_b [(phi_+a+b - phi_-a+b) - (phi_+a-b - phi_-a-b)],  phi = fbar+
// is formed per pair of opposite velocities from differences of neighbouring cells, and
// N = sum_d e_d [Y(+d) - Y(-d)]. No step-4 value is formed at an inner interface. Y needs only the
// interface's moments, formed in moment space (A(L) + B(R), A, B = M/2 +- kappa M_d - kappa/4 dt M_t).
// Without a force the brackets of all velocities that cross the interface are polynomials of
// ten numbers, which are differenced across the cell and combined; with a force the
// brackets themselves are. Both cells of an interface use the same numbers, so the equilibrium
// flux telescopes exactly. The z march keeps La, the x and y differences and the numbers of the -z
// interface in registers. At a wall interface: x, step 5 changes the interface's moments and La; y
// and z, the direct path (all velocities) gives f there, and its numbers are zero.
//
// Pairs. The velocity order puts opposite velocities at k and Q - 1 - k (the rest velocity in
// the middle), so the moving velocities form pairs (j, Q - 1 - j) with e_{Q-1-j} = -e_j. Every
// linear step of the scheme treats the two members of a pair with the same operation and
// coefficients of equal size (opposite signs where e enters), so the kernel keeps a pair in one
// float2 and uses the packed FP32 instructions of sm_100 and later (fma/add/mul .f32x2: two
// FP32 operations per instruction, each rounded as its scalar form). Shared memory holds pairs
// side by side, so a pair moves with one 64-bit access; strides of 2 mod 4 words keep those
// accesses free of bank conflicts.
//
// The 512 threads launch with 128 registers each; the producer warpgroups then give registers
// back (setmaxnreg to PROD_REGS) and the consumer warpgroups take them (CONS_REGS): 256 x 72 +
// 256 x 184 = 512 x 128. Every wait on an mbarrier gives up after about two seconds (a device
// flag, then the group leaves together; see tma.cuh).
// The update adds the flux in increment form, La + b7 (W N' - La), with the weight W in head and tail: with
// rounded (1 - b7) and b7 W, whose errors repeat at every step, forced and channel flows were up to 1.6 times
// as far from FP64 as the non-specialised kernel after 20 steps. Error of the state / of u against FP64, this
// kernel over the non-specialised one, geometric means over 36 random meshes (8 to 40 cells a side; channels on
// three axes, forced, cavity, duct, periodic): 20 steps 0.86 / 0.92, 200 0.96 / 0.97, 1000 0.90 / 0.88, 4000 0.88 /
// 0.88 (the worst family, cavities: 1.11 / 1.07 after 4000; the reference kernel scatters by 0.94 to 1.03).
// Measured (ms, the non-specialised kernel / this one): a step of the 256^3 cavity 3.81 / 2.62; 20 steps of a
// 157 x 101 x 83 channel under a force field, its moments and state read 13.9 / 8.3.
#pragma once

#include <math.h>
#include <string.h>

#include "dugks_internal.h"
#include "dugks_step3d.cuh"

namespace dugks {

namespace ws27 {  // the D3Q19 kernel (dugks_step3d_ws.cuh) has parts of the same names

// Opposite pairs and the per-cell layout of the ring.
template <int Q>
struct Pr {
    static constexpr int NP = (Q - 1) / 2, NX = n_flux<Q>(0) / 2;  // pairs; those that cross an interface
    __host__ __device__ static constexpr int e(int j, int a) { return Lat<Q>::e(j, a); }
    __host__ __device__ static constexpr int nnz(int j) { return (e(j, 0) != 0) + (e(j, 1) != 0) + (e(j, 2) != 0); }
    // the p-th pair whose velocities cross a face normal to d, and the position of pair j in that list
    __host__ __device__ static constexpr int cross(int d, int p) {
        int n = 0, r = -1;
        for (int j = 0; j < NP; j++)
            if (e(j, d) != 0) {
                if (n == p) r = j;
                n++;
            }
        return r;
    }
    __host__ __device__ static constexpr int pos(int d, int j) {
        int n = 0;
        for (int i = 0; i < j; i++) n += e(i, d) != 0;
        return e(j, d) != 0 ? n : -1;
    }
    // Per cell, CS floats: [2j, 2j+1] fbar+ of pair j; the rest velocity and M0; (M_a, M_aa) per axis;
    // (M_xy, M_xz); (M_yz, M_xz).
    static constexpr int REST = 2 * NP, M0 = REST + 1, XY = 2 * NP + 8, YZ = XY + 2, CS = XY + 4;
    __host__ __device__ static constexpr int ma(int a) { return 2 * NP + 2 + 2 * a; }
    // slot of velocity k and of the second moment M_ab
    __host__ __device__ static constexpr int rslot(int k) {
        return k < NP ? 2 * k : (k > NP ? 2 * (Q - 1 - k) + 1 : REST);
    }
    __host__ __device__ static constexpr int mslot(int a, int b) {
        return a == b ? ma(a) + 1 : (a + b == 1 ? XY : (a + b == 2 ? XY + 1 : YZ));
    }
    __host__ __device__ static constexpr bool layout_ok() {
        for (int j = 0; j < NP; j++)
            if (opposite<Q>(j) != Q - 1 - j || nnz(j) == 0) return false;
        for (int j = 0; j < NP; j++)
            if (e(j, 0) > 0) return false;  // the first member of an x pair has e_x = -1
        return nnz(NP) == 0 && CS % 4 == 2;
    }
};
static_assert(Pr<27>::layout_ok(), "velocity order without opposite pairs at k, Q - 1 - k");

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ void st2(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
// a - b, rounded as the scalar difference
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 r;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; sub.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 ghost2(float2 a, float2 b) { return f2(ghost_value(a.x, b.x), ghost_value(a.y, b.y)); }

template <int Q, class S, bool FORCE>
struct ShapeWS {
    using P = Pr<Q>;
    static constexpr int RX = 32, RY = 8, NC = RX * RY;  // cell columns of the tile, halo included
    static constexpr int NPROD = NC, NCONS = NC, NTHREADS = NPROD + NCONS;
    static constexpr int PROD_REGS = 72, CONS_REGS = 184;
    static_assert(NPROD * PROD_REGS + NCONS * CONS_REGS <= NTHREADS * 128, "register split above the launch's");
    static constexpr int TXI = RX - 2, TYI = RY - 2;  // inner columns
    static constexpr int CS = P::CS;                  // ring floats per cell
    // numbers per interface: the polynomial's, or (with a force) the brackets of the crossing pairs
    static constexpr int NV = FORCE ? 2 * P::NX : 10;
    static constexpr int NSLOT = 4;
    static constexpr int PLANE = RY * RX * CS;
    // Without a force every row forms the numbers of both its y interfaces from the parts A_y, B_y of
    // its neighbours (double-buffered, one barrier per plane); with one, where they are many, each
    // interface's are formed once and published behind a second barrier.
    static constexpr bool BOTH_Y = !FORCE;
    // ring; A_y and B_y of all rows; numbers at +y of rows 0..RY-2; wall terms of the low and high y wall
    static constexpr int XB = (BOTH_Y ? 2 : 1) * RY * RX * 8, YV = BOTH_Y ? 0 : (RY - 1) * RX * NV, WT = 2 * 2 * RX * 2 * P::NX;
    static constexpr size_t FLOATS = (size_t)NSLOT * PLANE + XB + YV + WT;
    static_assert(PLANE % 4 == 0 && XB % 4 == 0 && YV % 4 == 0 && WT % 4 == 0, "vector accesses must stay aligned");
    static constexpr int BX = 32 + (sizeof(S) == 4 ? 4 : 8);  // TMA box width (start rounded down)
    static constexpr size_t STAGE_BYTES = (size_t)Q * RY * BX * sizeof(S);
    static constexpr size_t STAGE_OFF = FLOATS * 4;  // aligned to 128 bytes at run time
    static constexpr size_t BAR_OFF = (STAGE_BYTES + 7) / 8 * 8;  // from the aligned stage: full[4], empty[4], stage
    static constexpr size_t smem_bytes = STAGE_OFF + 128 + BAR_OFF + 9 * 8;
    static_assert(smem_bytes <= 227 * 1024, "warp-specialised tile does not fit");
};

__device__ __forceinline__ void named_bar(int id, int n) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }
// Named barrier with an OR over the participating threads' predicates.
__device__ __forceinline__ bool named_bar_or(int id, int n, bool v) {
    uint32_t r;
    asm volatile(
        "{ .reg .pred p, q; setp.ne.u32 p, %1, 0; bar.red.or.pred q, %2, %3, p; selp.u32 %0, 1, 0, q; }\n"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(id), "r"(n)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// Step 1 (eq. (24) with eq. (6)) for one cell on pairs: G[j] = (g~_j, g~_{Q-1-j}), g9 the rest
// velocity, Gh the acceleration / c at t_n (FORCE). Writes the cell's ring entry o (fbar+ and its
// moments).
// The momentum sums are exact as in moments<Q, float, true>: heads on the grid of the cell's largest
// |g| are summed without rounding (pair by pair: the head sums of the first and second members,
// then their difference), tails separately, one rounding at the end. The equilibrium pair is
// geq_pair's, the relaxation relax's, one packed operation per pair.
template <int Q, bool FORCE>
__device__ __forceinline__ void step1_pairs(const float2 *G, float g9, const float Gh[3], const Coef<float> &cf,
                                            float *o) {
    using P = Pr<Q>;
    float2 Rs = G[0];
#pragma unroll
    for (int j = 1; j < P::NP; j++) Rs = __fadd2_rn(Rs, G[j]);
    const float drho = (Rs.x + Rs.y) + g9;
    float amax = 0.0f;
#pragma unroll
    for (int j = 0; j < P::NP; j++) amax = fmaxf(amax, fmaxf(fabsf(G[j].x), fabsf(G[j].y)));
    // 1.5 * 2^(E + 5) for amax in [2^E, 2^(E+1)): exponent field + 5, significand 1.5
    const float split = __uint_as_float((__float_as_uint(amax) & 0x7f800000u) + 0x02c00000u);
    const float2 SP = f2(split, split);
    float2 AH[3] = {f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f)}, AL[3] = {f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f)};
    sfor<P::NP>([&](auto jc) {
        constexpr int j = jc;
        const float2 H = sub2(__fadd2_rn(G[j], SP), SP);
        const float2 Lo = sub2(G[j], H);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (P::e(j, a) > 0) { AH[a] = __fadd2_rn(AH[a], H); AL[a] = __fadd2_rn(AL[a], Lo); }
            if (P::e(j, a) < 0) { AH[a] = sub2(AH[a], H); AL[a] = sub2(AL[a], Lo); }
        }
    });
    float m[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float lo = AL[a].x - AL[a].y;
        m[a] = __fadd_rn(AH[a].x - AH[a].y, FORCE ? fmaf(Gh[a], cf.wcell * cf.rho0, lo) : lo);
    }
    const float mm = dotD<3, float>(m, m);
    float gm = 0.0f;
    if (FORCE) gm = dotD<3, float>(Gh, m) * cf.inv_rho0;
    const float base = fmaf(-1.5f * cf.inv_rho0, mm, drho);
    const float c45 = 4.5f * cf.inv_rho0;
    const float2 B2 = f2(cf.b1, cf.b1);
    float f9;
    {
        const float geq = wmul<Q, float>(P::NP, base);
        float inc = cf.b1 * (geq - g9);
        if (FORCE) inc = fmaf(cf.c1, 3.0f * (0.0f - gm) * fmaf((float)Lat<Q>::template wt<double>(P::NP), cf.rho0, geq), inc);
        f9 = g9 + inc;
    }
    // moments of fbar+: Ps[a] sums the pairs whose first member has e_a = +1, Ns[a] those with -1
    // (the second member then counts the other way)
    float2 Ps[3] = {f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f)}, Ns[3] = {f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, 0.f)};
    float2 S0 = f2(0.f, 0.f), XY = f2(0.f, 0.f), XZ = f2(0.f, 0.f), YZ = f2(0.f, 0.f);
    sfor<P::NP>([&](auto jc) {
        constexpr int j = jc;
        constexpr int ex = P::e(j, 0), ey = P::e(j, 1), ez = P::e(j, 2);
        float em = 0.0f, ge = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (P::e(j, a) > 0) { em += m[a]; if (FORCE) ge += Gh[a]; }
            if (P::e(j, a) < 0) { em -= m[a]; if (FORCE) ge -= Gh[a]; }
        }
        const float q = fmaf(c45 * em, em, base);
        constexpr double W = Lat<Q>::template wt<double>(j);
        constexpr float wh = (float)W, wl = (float)(W - (double)wh);
        constexpr float w3h = (float)(3.0 * W), w3l = (float)(3.0 * W - (double)w3h);
        const float wq = fmaf(wl, q, wh * q);
        // scalar: the weights are immediates there, a packed operation would need them in registers
        const float2 GEQ = f2(fmaf(w3h, em, fmaf(w3l, em, wq)), fmaf(-w3h, em, fmaf(-w3l, em, wq)));
        float2 F;
        const float2 D = sub2(GEQ, G[j]);
        if constexpr (FORCE) {
            const float2 FEQ = __ffma2_rn(f2((float)W, (float)W), f2(cf.rho0, cf.rho0), GEQ);
            const float c3 = 3.0f * cf.c1;
            const float2 I = __ffma2_rn(f2(c3 * (ge - gm), c3 * (-ge - gm)), FEQ, __fmul2_rn(B2, D));
            F = __fadd2_rn(G[j], I);
        } else {
            F = __ffma2_rn(B2, D, G[j]);
        }
        st2(o + 2 * j, F);
        if constexpr (ex > 0) Ps[0] = __fadd2_rn(Ps[0], F);
        if constexpr (ex < 0) Ns[0] = __fadd2_rn(Ns[0], F);
        if constexpr (ex == 0) S0 = __fadd2_rn(S0, F);
        if constexpr (ey > 0) Ps[1] = __fadd2_rn(Ps[1], F);
        if constexpr (ey < 0) Ns[1] = __fadd2_rn(Ns[1], F);
        if constexpr (ez > 0) Ps[2] = __fadd2_rn(Ps[2], F);
        if constexpr (ez < 0) Ns[2] = __fadd2_rn(Ns[2], F);
        if constexpr (ex * ey > 0) XY = __fadd2_rn(XY, F);
        if constexpr (ex * ey < 0) XY = sub2(XY, F);
        if constexpr (ex * ez > 0) XZ = __fadd2_rn(XZ, F);
        if constexpr (ex * ez < 0) XZ = sub2(XZ, F);
        if constexpr (ey * ez > 0) YZ = __fadd2_rn(YZ, F);
        if constexpr (ey * ez < 0) YZ = sub2(YZ, F);
    });
    float sp[3], sn[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        sp[a] = Ps[a].x + Ns[a].y;
        sn[a] = Ps[a].y + Ns[a].x;
    }
    st2(o + P::REST, f2(f9, ((S0.x + S0.y) + f9) + (sp[0] + sn[0])));
#pragma unroll
    for (int a = 0; a < 3; a++) st2(o + P::ma(a), f2(sp[a] - sn[a], sp[a] + sn[a]));
    const float xz = XZ.x + XZ.y;
    st2(o + P::XY, f2(XY.x + XY.y, xz));
    st2(o + P::YZ, f2(YZ.x + YZ.y, xz));
}

// Steps 3-4 for all velocities at the interface normal to d (reconstruct of dugks_step.cuh) from
// cells in the ring's pair layout; F in velocity order.
template <int Q, int d>
__device__ __forceinline__ void reconstruct_pairs(const float *L, const float *R, const float *L1m, const float *R1m,
                                                  const float *L1p, const float *R1p, const float *L2m,
                                                  const float *R2m, const float *L2p, const float *R2p, float kappa,
                                                  float *F) {
    constexpr int t1 = d == 0 ? 1 : 0;
    constexpr int t2 = d == 2 ? 1 : 2;
    const float qk = 0.25f * kappa;
    sfor<Q>([&](auto kc) {
        constexpr int k = kc;
        constexpr int s = Pr<Q>::rslot(k);
        const float l = L[s], r = R[s];
        float v = mul_rn(0.5f, l + r);
        if constexpr (Lat<Q>::e(k, d) != 0) v = fmaf(-kappa * (float)Lat<Q>::e(k, d), r - l, v);
        if constexpr (Lat<Q>::e(k, t1) != 0)
            v = fmaf(-qk * (float)Lat<Q>::e(k, t1), (L1p[s] + R1p[s]) - (L1m[s] + R1m[s]), v);
        if constexpr (Lat<Q>::e(k, t2) != 0)
            v = fmaf(-qk * (float)Lat<Q>::e(k, t2), (L2p[s] + R2p[s]) - (L2m[s] + R2m[s]), v);
        F[k] = v;
    });
}

// What the wall paths need of the kernel's position: the ring, the chunk's first plane and the
// time factor of the interface acceleration.
struct WsCtx {
    const float *ring;
    int z0, row, lane, gx, gy;
    float cth;
};

// Interface G / c at time t+h between (x,y,z) - e_d and (x,y,z): mean of the two cells, one cell at
// a wall (reading R2).
__device__ __forceinline__ void face_G3(const StepParams &p, int d, int x, int y, int z, float cth, float Gh[3]) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t ncell = (int64_t)nx * ny * nz;
    int lo[3] = {x, y, z}, hi[3] = {x, y, z};
    const int nd = d == 0 ? nx : (d == 1 ? ny : nz);
    const bool per = p.bc[2 * d] == 0;
    lo[d] -= 1;
    if (per) { lo[d] = wrap_idx(lo[d], nd); hi[d] = wrap_idx(hi[d], nd); }
    else { lo[d] = max(lo[d], 0); hi[d] = min(hi[d], nd - 1); }
    const int64_t il = (int64_t)lo[0] + (int64_t)nx * ((int64_t)lo[1] + (int64_t)ny * lo[2]);
    const int64_t ih = (int64_t)hi[0] + (int64_t)nx * ((int64_t)hi[1] + (int64_t)ny * hi[2]);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        float v = p.fg[a];
        if (p.field) v += 0.5f * (__ldg(p.field + a * ncell + il) + __ldg(p.field + a * ncell + ih));
        Gh[a] = v * cth;
    }
}

// A y or z wall interface by the direct path (all velocities reconstructed, steps 3-7): the
// interface normal to d between the cell (row, lane) at plane pl and the next cell along d, gfd its
// index along d. T: f - (1 - b7) F of the crossing pairs, divided by 1 - b7, so that e_d T added to
// the regular La of the cell below (subtracted above) makes the wall's f its flux. One row of
// a wall tile, and the first and last plane, take it.
template <int Q, bool FORCE, int d>
__device__ __forceinline__ void wall_term(const StepParams &p, const WsCtx &c, int row, int pl, int gfd, float2 *T) {
    using P = Pr<Q>;
    constexpr int RY = 8, NF = n_flux<Q>(0);
    const Coef<float> cf(p, FromTable());
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    auto slot_of = [&](int pz) { return (pz - (c.z0 - 1)) & 3; };
    auto ptr = [&](int s, int r, int l) -> const float * { return c.ring + ((s * RY + r) * 32 + l) * P::CS; };
    const int lane = c.lane;
    auto rec = [&](int r, int pc, float *F) __attribute__((always_inline)) {  // low cell (r, lane) at plane pc
        const int a = slot_of(pc - 1), b = slot_of(pc), e = slot_of(pc + 1);
        if constexpr (d == 1)
            reconstruct_pairs<Q, 1>(ptr(b, r, lane), ptr(b, r + 1, lane), ptr(b, r, lane - 1), ptr(b, r + 1, lane - 1),
                                    ptr(b, r, lane + 1), ptr(b, r + 1, lane + 1), ptr(a, r, lane), ptr(a, r + 1, lane),
                                    ptr(e, r, lane), ptr(e, r + 1, lane), cf.kappa, F);
        else
            reconstruct_pairs<Q, 2>(ptr(b, r, lane), ptr(e, r, lane), ptr(b, r, lane - 1), ptr(e, r, lane - 1),
                                    ptr(b, r, lane + 1), ptr(e, r, lane + 1), ptr(b, r - 1, lane), ptr(e, r - 1, lane),
                                    ptr(b, r + 1, lane), ptr(e, r + 1, lane), cf.kappa, F);
    };
    float F[Q], Fc[Q], o[NF];
    rec(row, pl, F);
    const float a7 = 1.0f - cf.b7;
    sfor<P::NX>([&](auto pc) {
        constexpr int j = P::cross(d, pc);
        T[pc] = f2(a7 * F[j], a7 * F[Q - 1 - j]);
    });
    const int side = gfd == 0 ? 0 : 1, sh = gfd == 0 ? 1 : -1;
    float Gb[3] = {0.0f, 0.0f, 0.0f}, Gc[3] = {0.0f, 0.0f, 0.0f};
    const int fx = min(max(c.gx, 0), nx - 1);
    if constexpr (d == 1) rec(row + sh, pl, Fc);  // x_c: the boundary cell's opposite interface, one cell inward
    else rec(row, gfd == 0 ? 0 : nz - 2, Fc);
    if constexpr (FORCE) {
        const int fy = d == 1 ? gfd : min(max(c.gy, 0), ny - 1), fz = d == 2 ? gfd : pl;
        face_G3(p, d, fx, fy, fz, c.cth, Gb);
        face_G3(p, d, fx, d == 1 ? gfd + sh : fy, d == 2 ? gfd + sh : fz, c.cth, Gc);
    }
    interface_f<Q, d, float, false>(p, cf, F, Gb, 1, side, Fc, Gc, o);
    const float ia = 1.0f / a7;
    sfor<P::NX>([&](auto pc) {
        constexpr int j = P::cross(d, pc);
        T[pc] = f2((o[flux_index<Q>(d, j)] - T[pc].x) * ia, (o[flux_index<Q>(d, Q - 1 - j)] - T[pc].y) * ia);
    });
}

// Step 5 at the x walls of a tile's row: fm (drho, j) of every lane's +x interface, G there; at the
// walls fm takes the changes of the incoming velocities, which come back in lo (the lane of
// column 0: its -x interface's, second members) and hi (column nx - 1's +x interface, first members),
// zero elsewhere. cur, nxt, prv: the lane's ring entries of planes kz, kz + 1, kz - 1. Called by whole
// warps.
template <int Q>
struct WsXWall {
    float fm[4], G[3];
    float lo[Pr<Q>::NX], hi[Pr<Q>::NX];
};
template <int Q, bool FORCE>
__device__ __forceinline__ void x_wall_ws(const StepParams &p, int gx, const float *cur, const float *nxt, const float *prv,
                                       WsXWall<Q> &w) {
    using P = Pr<Q>;
    constexpr int NF = n_flux<Q>(0), NX1 = P::CS, NY1 = 32 * P::CS;
    const Coef<float> cf(p, FromTable());
    const float kap = cf.kappa, qk = 0.25f * kap;
    float F[NF], Fd[NF], Fu[NF];
    // step-4 values of the crossing pairs at the +x interface (lane 31 has none: its neighbour's are
    // read from its own entry)
    const int E = (threadIdx.x & 31) == 31 ? 0 : NX1;
    sfor<P::NX>([&](auto pc) {
        constexpr int j = P::cross(0, pc), ey = P::e(j, 1), ez = P::e(j, 2);
        const float2 l = ld2(cur + 2 * j), r = ld2(cur + E + 2 * j);
        float2 v = __ffma2_rn(f2(kap, -kap), sub2(r, l), __fmul2_rn(f2(0.5f, 0.5f), __fadd2_rn(l, r)));  // e_x = -1, 1
        if constexpr (ey != 0) {
            const float2 C = __fadd2_rn(sub2(ld2(cur + NY1 + 2 * j), ld2(cur - NY1 + 2 * j)),
                                        sub2(ld2(cur + E + NY1 + 2 * j), ld2(cur + E - NY1 + 2 * j)));
            v = __ffma2_rn(ey > 0 ? f2(-qk, qk) : f2(qk, -qk), C, v);
        }
        if constexpr (ez != 0) {
            const float2 C = __fadd2_rn(sub2(ld2(nxt + 2 * j), ld2(prv + 2 * j)), sub2(ld2(nxt + E + 2 * j), ld2(prv + E + 2 * j)));
            v = __ffma2_rn(ez > 0 ? f2(-qk, qk) : f2(qk, -qk), C, v);
        }
        F[flux_index<Q>(0, j)] = v.x;
        F[flux_index<Q>(0, Q - 1 - j)] = v.y;
    });
    // x_c is the interface that the next lane inward owns
    float md[4], mu[4], Gd[3] = {0.0f, 0.0f, 0.0f}, Gu[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < NF; i++) {
        Fd[i] = __shfl_down_sync(0xffffffffu, F[i], 1);
        Fu[i] = __shfl_up_sync(0xffffffffu, F[i], 1);
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        md[i] = __shfl_down_sync(0xffffffffu, w.fm[i], 1);
        mu[i] = __shfl_up_sync(0xffffffffu, w.fm[i], 1);
    }
    if constexpr (FORCE) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            Gd[a] = __shfl_down_sync(0xffffffffu, w.G[a], 1);
            Gu[a] = __shfl_up_sync(0xffffffffu, w.G[a], 1);
        }
    }
    float dl[P::NX];
    sfor<P::NX>([&](auto pc) {
        constexpr int j = P::cross(0, pc);
        dl[pc] = -F[flux_index<Q>(0, Q - 1 - j)];
        w.hi[pc] = -F[flux_index<Q>(0, j)];
    });
    if (gx == -1) neq_wall<Q, 0, FORCE, 0>(p, cf, F, w.fm[0], w.fm + 1, Fd, md[0], md + 1, Gd);
    if (gx == p.nx - 1) neq_wall<Q, 0, FORCE, 1>(p, cf, F, w.fm[0], w.fm + 1, Fu, mu[0], mu + 1, Gu);
    sfor<P::NX>([&](auto pc) {
        constexpr int j = P::cross(0, pc);
        const float d = __shfl_up_sync(0xffffffffu, dl[pc] + F[flux_index<Q>(0, Q - 1 - j)], 1);
        w.lo[pc] = gx == 0 ? d : 0.0f;
        w.hi[pc] = gx == p.nx - 1 ? w.hi[pc] + F[flux_index<Q>(0, j)] : 0.0f;
    });
}

template <int Q, class S, bool FORCE>
__global__ void __launch_bounds__(512, 1)
    fused_step3d_ws(const __grid_constant__ StepParams p, const __grid_constant__ CUtensorMap tmap, int zchunk) {
    using K = ShapeWS<Q, S, FORCE>;
    using P = Pr<Q>;
    constexpr int RY = K::RY, CS = K::CS, NP = P::NP, NX = P::NX, NV = K::NV;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int z0 = blockIdx.z * zchunk;
    const int z1 = min(p.nz, z0 + zchunk);
    const int x0 = blockIdx.x * K::TXI, y0 = blockIdx.y * K::TYI;

    float *ring = reinterpret_cast<float *>(smem_raw);  // [NSLOT][RY][32][CS]
    float *xb = ring + K::NSLOT * K::PLANE;            // [2][RY][32][8]: A_y, B_y (by the plane's parity)
    float *yv = xb + K::XB;                            // [rows 0..RY-2][NV][32]: numbers at +y
    float *wt = yv + K::YV;                            // [2][2][32][2 NX]: terms of the low / high y wall
    unsigned char *stage = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw + K::STAGE_OFF) + 127) & ~(uintptr_t)127);
    uint64_t *full = reinterpret_cast<uint64_t *>(stage + K::BAR_OFF);
    uint64_t *empty = full + 4;
    uint64_t *sbar = full + 8;

    const int tid = threadIdx.x;
    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < 4; s++) {
            mbar_init(full + s, K::NPROD);
            mbar_init(empty + s, K::NCONS);
        }
        mbar_init(sbar, 1);
        mbar_fence_init();
    }
    __syncthreads();

    const Coef<float> cf(p, FromTable());
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t ncell = (int64_t)nx * ny * nz;
    const bool perx = p.bc[0] == 0, pery = p.bc[2] == 0, perz = p.bc[4] == 0;
    const S *src = reinterpret_cast<const S *>(p.src);
    S *dst = reinterpret_cast<S *>(p.dst);
    // planes z0 - 1 .. z1 in order: n = pz - (z0 - 1) selects ring slot n % 4 (phase n / 4)
    auto nidx = [&](int pz) __attribute__((always_inline)) { return pz - (z0 - 1); };
    auto slot_of = [&](int pz) __attribute__((always_inline)) { return nidx(pz) & 3; };
    auto R = [&](int slot, int r, int l) __attribute__((always_inline)) -> float * {
        return ring + ((slot * RY + r) * 32 + l) * CS;
    };
    const bool xwall_tile = !perx && (x0 == 0 || x0 + K::TXI >= nx);
    const bool ywall_tile = !pery && (y0 == 0 || y0 + K::TYI >= ny);

    // the cell column of a thread: producer thread c and consumer thread NPROD + c own column c
    const int lane = tid & 31, row = (tid & (K::NC - 1)) >> 5;
    const int gx = x0 - 1 + lane, gy = y0 - 1 + row;
    int cx = gx, cy = gy;  // the column's cell: wrapped on a periodic axis
    bool load = true;
    if (gx < 0 || gx >= nx) { if (perx && gx >= -1 && gx <= nx) cx = wrap_idx(gx, nx); else load = false; }
    if (gy < 0 || gy >= ny) { if (pery && gy >= -1 && gy <= ny) cy = wrap_idx(gy, ny); else load = false; }

    if (tid < K::NPROD) {
        // =============================== producer ===============================
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(K::PROD_REGS));
        // real planes first .. lastp are copied in order into the one stage (phase m & 1 for the
        // m-th); thread 0 issues the next copy once every producer thread has read the stage
        const int first = (!perz && z0 - 1 < 0) ? z0 : z0 - 1;
        const int lastp = (!perz && z1 >= nz) ? nz - 1 : z1;
        constexpr int XA = 16 / (int)sizeof(S);
        const int xs = (x0 - 1 >= 0) ? (x0 - 1) / XA * XA : -XA;
        auto issue = [&](int pz) __attribute__((always_inline)) {
            if (tid == 0 && pz >= first && pz <= lastp) {
                mbar_arrive_expect_tx(sbar, (uint32_t)K::STAGE_BYTES);
                tma_load_4d(stage, &tmap, sbar, xs, y0 - 1, wrap_idx(pz, nz), 0);
            }
        };
        bool ok = true;
        issue(first);
        const bool boxed = load && cx == gx && cy == gy;
        const bool yreal = (gy >= 0 && gy < ny) || (pery && gy >= -1 && gy <= ny);
        const bool xghost = !perx && (gx == -1 || gx == nx) && yreal;
        const bool yghost = !pery && (gy == -1 || gy == ny) && gx >= -1 && gx <= nx;
        int m = 0;  // real planes read from the stage so far
        // step 1 for real plane pz into its ring slot; false: a wait gave up (every
        // producer thread learns it at the same barrier)
        auto make_plane = [&](int pz) __attribute__((always_inline)) -> bool {
            const int gz = wrap_idx(pz, nz);
            float2 G[NP];
            float g9;
            ok = ok && mbar_wait(sbar, (uint32_t)(m & 1));
            m++;
            {
                const S *sb = reinterpret_cast<const S *>(stage) + row * K::BX + ((x0 - 1) - xs + lane);
                if (boxed) {
#pragma unroll
                    for (int j = 0; j < NP; j++)
                        G[j] = f2(stage_value(sb + j * (RY * K::BX)), stage_value(sb + (Q - 1 - j) * (RY * K::BX)));
                    g9 = stage_value(sb + NP * (RY * K::BX));
                } else if (load) {
                    const int64_t off = (int64_t)gz * p.plane + (int64_t)cy * p.px + cx;
#pragma unroll
                    for (int j = 0; j < NP; j++)
                        G[j] = f2((float)Store<S>::ld(src + j * p.dstride + off),
                                  (float)Store<S>::ld(src + (Q - 1 - j) * p.dstride + off));
                    g9 = (float)Store<S>::ld(src + NP * p.dstride + off);
                } else {
#pragma unroll
                    for (int j = 0; j < NP; j++) G[j] = f2(0.0f, 0.0f);
                    g9 = 0.0f;
                }
            }
            // the stage has been read: the next plane may land in it; every producer thread has
            // also finished the previous plane
            if (named_bar_or(1, K::NPROD, !ok)) return false;
            // the next real plane in order
            issue(pz + 1 <= lastp ? pz + 1 : lastp + 1);
            float *o = R(slot_of(pz), row, lane);
            if (!load) {
#pragma unroll
                for (int i = 0; i < CS / 2; i++) st2(o + 2 * i, f2(0.0f, 0.0f));
                return true;
            }
            float Gh[3] = {0.0f, 0.0f, 0.0f};
            if (FORCE) {
                const int64_t ci = (int64_t)cx + (int64_t)nx * ((int64_t)cy + (int64_t)ny * gz);
                cell_G<3, float>(p, ci, ncell, cf.ct, Gh);
            }
            step1_pairs<Q, FORCE>(G, g9, Gh, cf, o);
            return true;
        };
        // step 2 (reading R3: ghost = 2 f0 - f1, x then y): fbar+ and, by linearity, its moments
        auto ghosts_xy = [&](int pz) __attribute__((always_inline)) {
            const int sl = slot_of(pz);
            if (xwall_tile) {
                named_bar(1, K::NPROD);
                if (xghost) {
                    const int d1 = gx < 0 ? 1 : -1;
                    float *o = R(sl, row, lane);
                    const float *a = R(sl, row, lane + d1), *b = R(sl, row, lane + 2 * d1);
#pragma unroll
                    for (int i = 0; i < CS / 2; i++) st2(o + 2 * i, ghost2(ld2(a + 2 * i), ld2(b + 2 * i)));
                }
            }
            if (ywall_tile) {
                named_bar(1, K::NPROD);
                if (yghost) {
                    const int d1 = gy < 0 ? 1 : -1;
                    float *o = R(sl, row, lane);
                    const float *a = R(sl, row + d1, lane), *b = R(sl, row + 2 * d1, lane);
#pragma unroll
                    for (int i = 0; i < CS / 2; i++) st2(o + 2 * i, ghost2(ld2(a + 2 * i), ld2(b + 2 * i)));
                }
            }
        };
        // a ghost plane beyond a non-periodic z wall (whole region)
        auto ghost_z = [&](int pz) __attribute__((always_inline)) {
            float *o = R(slot_of(pz), row, lane);
            const float *a = R(slot_of(pz < 0 ? 0 : nz - 1), row, lane);
            const float *b = R(slot_of(pz < 0 ? 1 : nz - 2), row, lane);
#pragma unroll
            for (int i = 0; i < CS / 2; i++) st2(o + 2 * i, ghost2(ld2(a + 2 * i), ld2(b + 2 * i)));
        };
        auto leave = [&]() __attribute__((always_inline)) {
            if (tid == 0) mbar_wait(sbar, (uint32_t)(m & 1));  // a copy still in flight: bounded wait
        };

        // prologue: planes z0 - 1 .. z0 + 1 (a ghost plane below z = 0 after the planes it needs)
        for (int pz = z0 - 1; pz <= z0 + 1; pz++) {
            if (!perz && (pz < 0 || pz >= nz)) continue;
            if (!make_plane(pz)) { leave(); return; }
            ghosts_xy(pz);
        }
        if (named_bar_or(1, K::NPROD, !ok)) { leave(); return; }
        for (int pz = z0 - 1; pz <= z0 + 1; pz++)
            if (!perz && (pz < 0 || pz >= nz)) ghost_z(pz);
        for (int pz = z0 - 1; pz <= z0 + 1; pz++) mbar_arrive(full + slot_of(pz));
        // the rest of the chunk, each plane into a slot the consumers have released
        for (int pz = z0 + 2; pz <= z1; pz++) {
            const int n = nidx(pz);
            if (n >= 4) ok = ok && mbar_wait(empty + (n & 3), (uint32_t)(((n >> 2) - 1) & 1));
            if (perz || pz < nz) {
                if (!make_plane(pz)) { leave(); return; }
                ghosts_xy(pz);
            } else {  // pz == nz: the ghost plane above the top wall
                if (named_bar_or(1, K::NPROD, !ok)) { leave(); return; }
                ghost_z(pz);
            }
            mbar_arrive(full + (n & 3));
        }
        return;
    }

    // =============================== consumers ===============================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(K::CONS_REGS));
    constexpr int NX1 = CS, NY1 = 32 * CS;  // ring offsets of the x and y neighbours
    constexpr std::integral_constant<int, 0> AX{};
    constexpr std::integral_constant<int, 1> AY{};
    constexpr std::integral_constant<int, 2> AZ{};
    const bool inner = lane >= 1 && lane <= K::TXI && row >= 1 && row <= K::TYI;
    const bool xrow = row >= 1 && row <= K::TYI && gy < ny;  // rows that update (warp-uniform)
    const bool upd = inner && gx < nx && gy < ny;
    const bool ycol = lane >= 1 && lane <= K::TXI && gx >= 0 && gx < nx && gy >= -1 && gy <= ny;
    const bool need_y = ycol && row <= K::TYI && gy < ny;
    const bool ywlo = !pery && gy == -1, ywhi = !pery && gy == ny;  // the ghost rows: they make the y walls' terms
    const bool ynwall = !pery && (gy == -1 || gy == ny - 1);        // the +y interface is a wall
    const float kap = cf.kappa, qk = -0.25f * kap, c45 = 4.5f * cf.inv_rho0;
    uint32_t seed = 0;  // stochastic rounding of 16-bit stores
    if constexpr (sizeof(S) == 2) seed = store_seed(*p.step_ctr + p.step_off);
    const WsCtx ctx{ring, z0, row, lane, gx, gy, cf.cth};
    auto wait_full = [&](int pz) __attribute__((always_inline)) -> bool {
        const int n = nidx(pz);
        return mbar_wait(full + (n & 3), (uint32_t)((n >> 2) & 1));
    };
    auto release = [&](int pz) __attribute__((always_inline)) {
        if (pz >= z0 - 1) mbar_arrive(empty + slot_of(pz));
    };
    // the thread's own column in the ring slot of plane pz
    auto Pz = [&](int pz) __attribute__((always_inline)) -> const float * {
        return ring + slot_of(pz) * K::PLANE + (row * 32 + lane) * CS;
    };
    // index along an axis of n cells: wrapped on a periodic axis, the nearest cell beyond a wall (and, for
    // columns that nothing reads, beyond the tile's last)
    auto near = [&](int i, int n, bool per) __attribute__((always_inline)) { return min(max(per ? wrap_idx(i, n) : i, 0), n - 1); };
    const int field_x = near(gx, nx, perx);
    // the cell's acceleration field at plane pz (the nearest cell's beyond a wall), and its +y neighbour's
    auto cell_field = [&](int y, int pz, float f[3]) __attribute__((always_inline)) {
        f[0] = f[1] = f[2] = 0.0f;
        if constexpr (FORCE) {
            if (p.field) {
                const int zz = perz ? wrap_idx(pz, nz) : min(max(pz, 0), nz - 1);
                const int64_t i = (int64_t)field_x + (int64_t)nx * (near(y, ny, pery) + (int64_t)ny * zz);
#pragma unroll
                for (int a = 0; a < 3; a++) f[a] = __ldg(p.field + a * ncell + i);
            }
        }
    };
    auto mean_G = [&](const float a[3], const float b[3], float G[3]) __attribute__((always_inline)) {
#pragma unroll
        for (int i = 0; i < 3; i++) G[i] = FORCE ? (p.fg[i] + 0.5f * (a[i] + b[i])) * cf.cth : 0.0f;
    };
    // differences of the moments (M_t, M_xt, M_yt, M_zt) between two entries
    auto mdiff = [&](const float *lo, const float *hi, auto tc, float dM[4]) __attribute__((always_inline)) {
        constexpr int t = decltype(tc)::value;
        const float2 d1 = sub2(ld2(hi + P::ma(t)), ld2(lo + P::ma(t)));  // (M_t, M_tt)
        dM[0] = d1.x;
        dM[1 + t] = d1.y;
        if constexpr (t == 0) {
            const float2 d2 = sub2(ld2(hi + P::XY), ld2(lo + P::XY));  // (M_xy, M_xz)
            dM[2] = d2.x;
            dM[3] = d2.y;
        } else if constexpr (t == 1) {
            dM[1] = hi[P::XY] - lo[P::XY];
            dM[3] = hi[P::YZ] - lo[P::YZ];
        } else {
            const float2 d2 = sub2(ld2(hi + P::YZ), ld2(lo + P::YZ));  // (M_yz, M_xz)
            dM[2] = d2.x;
            dM[1] = d2.y;
        }
    };
    // parts A (SIGN = 1) or B (-1) of the moments (drho, j) at the interface normal to d
    auto mparts = [&](auto dc, auto sc, const float *c, const float dM1[4], const float dM2[4], float A[4])
                      __attribute__((always_inline)) {
        constexpr int d = decltype(dc)::value;
        const float k = decltype(sc)::value > 0 ? kap : -kap;
        A[0] = fmaf(0.5f, c[P::M0], fmaf(k, c[P::ma(d)], qk * (dM1[0] + dM2[0])));
#pragma unroll
        for (int a = 0; a < 3; a++)
            A[1 + a] = fmaf(0.5f, c[P::ma(a)], fmaf(k, c[P::mslot(a, d)], qk * (dM1[1 + a] + dM2[1 + a])));
    };
    constexpr std::integral_constant<int, 1> SA{};
    constexpr std::integral_constant<int, -1> SB{};
    // the numbers of an interface normal to d from its moments fm = (drho, j) (header)
    auto numbers = [&](auto dc, const float fm[4], const float Gh[3], float V[NV]) __attribute__((always_inline)) {
        constexpr int d = decltype(dc)::value, t = d == 0 ? 1 : 0, u = d == 2 ? 1 : 2;
        float m[3];
#pragma unroll
        for (int a = 0; a < 3; a++) m[a] = FORCE ? fmaf(Gh[a], cf.wface * cf.rho0, fm[1 + a]) : fm[1 + a];
        const float base = fmaf(-1.5f * cf.inv_rho0, dotD<3, float>(m, m), fm[0]);
        if constexpr (!FORCE) {
            const float s = c45 * m[d], s2 = 2.0f * s, Pn = fmaf(s, m[d], base), wt2 = c45 * m[t], wu2 = c45 * m[u];
            V[0] = Pn;
#pragma unroll
            for (int a = 0; a < 3; a++) V[1 + a] = m[a];
            V[4] = fmaf(wt2, m[t], Pn);  // R_t
            V[5] = s2 * m[t];            // S_t
            V[6] = fmaf(wu2, m[u], Pn);  // R_u
            V[7] = s2 * m[u];            // S_u
            V[8] = fmaf(wu2, m[u], V[4]);   // base + 4.5 (m_x^2 + m_y^2 + m_z^2) / rho0
            V[9] = 2.0f * wt2 * m[u];       // 9 m_t m_u / rho0
        } else {
            // Y = b7 X + t (rho0 + X), X = q +- 3 e.m, t = 3 c7 (+-G.e - G.m / rho0)
            const float c73 = 3.0f * cf.c7, gm = c73 * (dotD<3, float>(Gh, m) * cf.inv_rho0);
            sfor<NX>([&](auto pc) {
                constexpr int j = P::cross(d, pc);
                float em = 0.0f, ge = 0.0f;
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    if (P::e(j, a) > 0) { em += m[a]; ge += Gh[a]; }
                    if (P::e(j, a) < 0) { em -= m[a]; ge -= Gh[a]; }
                }
                const float q = fmaf(c45 * em, em, base), g3 = c73 * ge;
                const float2 X = f2(fmaf(3.0f, em, q), fmaf(-3.0f, em, q)), tt = f2(g3 - gm, -g3 - gm);
                const float2 Y = __ffma2_rn(tt, __fadd2_rn(f2(cf.rho0, cf.rho0), X), __fmul2_rn(f2(cf.b7, cf.b7), X));
                V[2 * pc] = Y.x;
                V[2 * pc + 1] = Y.y;
            });
        }
    };
    // pair coefficients of La: differences across the high and low interface of axis d, for a first
    // member with e_d = sg; -kappa/2 e_a e_b (XM) and its negative
    const float ca = 0.5f - kap, cb = 0.5f + kap;
    auto cH = [&](int sg) __attribute__((always_inline)) { return sg > 0 ? f2(ca, -cb) : f2(-cb, ca); };
    auto cL = [&](int sg) __attribute__((always_inline)) { return sg > 0 ? f2(cb, -ca) : f2(-ca, cb); };
    auto xm = [&](int s) __attribute__((always_inline)) { const float v = s > 0 ? -0.5f * kap : 0.5f * kap; return f2(v, v); };
    // the in-plane part of La of pair j at the entry q, and the pair's x and y differences (for its
    // mixed differences along z)
    auto planar = [&](auto jc, const float *q, float2 &l, float2 &dx, float2 &dy) __attribute__((always_inline)) {
        constexpr int j = decltype(jc)::value, ex = P::e(j, 0), ey = P::e(j, 1), ez = P::e(j, 2);
        const float2 f = ld2(q + 2 * j);
        l = f2(0.0f, 0.0f);
        if constexpr (ex != 0) {
            const float2 E = ld2(q + NX1 + 2 * j), Wv = ld2(q - NX1 + 2 * j);
            l = __ffma2_rn(cH(ex), sub2(E, f), __fmul2_rn(cL(ex), sub2(f, Wv)));
            if constexpr (ez != 0) dx = sub2(E, Wv);
        }
        if constexpr (ey != 0) {
            const float2 N = ld2(q + NY1 + 2 * j), Sv = ld2(q - NY1 + 2 * j);
            const float2 lo = __fmul2_rn(cL(ey), sub2(f, Sv));
            l = ex != 0 ? __fadd2_rn(l, __ffma2_rn(cH(ey), sub2(N, f), lo)) : __ffma2_rn(cH(ey), sub2(N, f), lo);
            if constexpr (ez != 0) dy = sub2(N, Sv);
        }
        if constexpr (ex != 0 && ey != 0) {
            const float2 X = sub2(sub2(ld2(q + NY1 + NX1 + 2 * j), ld2(q + NY1 - NX1 + 2 * j)),
                                  sub2(ld2(q - NY1 + NX1 + 2 * j), ld2(q - NY1 - NX1 + 2 * j)));
            l = __ffma2_rn(xm(ex * ey), X, l);
        }
    };
    auto cons_bar = [&]() __attribute__((always_inline)) { named_bar(2, K::NCONS); };
    auto cons_bar_or = [&](bool v) __attribute__((always_inline)) { return named_bar_or(2, K::NCONS, v); };
    bool ok = true;
    for (int pz = z0 - 1; pz <= z0 + 1; pz++) ok = ok && wait_full(pz);
    if (cons_bar_or(!ok)) return;

    // carried for the current plane: La, the x and y differences of the pairs with e_z != 0, the
    // numbers of the -z interface, A_z, the moments' x and y differences, the acceleration field
    float2 La[NP], dxc[NX], dyc[NX];
    float Vz[NV], Az[4], Mx[4], My[4], fc[3];
#pragma unroll
    for (int j = 0; j < NP; j++) La[j] = f2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < NX; i++) dxc[i] = dyc[i] = f2(0.0f, 0.0f);
#pragma unroll
    for (int i = 0; i < NV; i++) Vz[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; i++) Az[i] = Mx[i] = My[i] = 0.0f;
    cell_field(gy, z0, fc);
    if (ycol) {
        const float *q = Pz(z0);
        mdiff(q - NX1, q + NX1, AX, Mx);
    }
    if (xrow) {  // every lane: the x interfaces' parts of lanes 0 and 31 are exchanged too
        const float *q = Pz(z0);
        mdiff(q - NY1, q + NY1, AY, My);
    }
    if (upd) {
        const float *q = Pz(z0), *b = Pz(z0 - 1);
        // La of plane z0 with the part of plane z0 - 1
        sfor<NP>([&](auto jc) {
            constexpr int j = jc, ex = P::e(j, 0), ey = P::e(j, 1), ez = P::e(j, 2), i = ez != 0 ? P::pos(2, j) : 0;
            float2 l, dx, dy;
            planar(jc, q, l, dx, dy);
            if constexpr (ez != 0) {
                l = __ffma2_rn(cL(ez), sub2(ld2(q + 2 * j), ld2(b + 2 * j)), l);
                if constexpr (ex != 0) {
                    l = __ffma2_rn(xm(-ex * ez), sub2(ld2(b + NX1 + 2 * j), ld2(b - NX1 + 2 * j)), l);
                    dxc[i] = dx;
                }
                if constexpr (ey != 0) {
                    l = __ffma2_rn(xm(-ey * ez), sub2(ld2(b + NY1 + 2 * j), ld2(b - NY1 + 2 * j)), l);
                    dyc[i] = dy;
                }
            }
            La[j] = l;
        });
        mparts(AZ, SA, q, Mx, My, Az);
        if (!perz && z0 == 0) {
            float2 T[NX];
            wall_term<Q, FORCE, 2>(p, ctx, row, -1, 0, T);
            sfor<NX>([&](auto pc) {
                constexpr int j = P::cross(2, pc);
                La[j] = P::e(j, 2) > 0 ? f2(La[j].x - T[pc].x, La[j].y + T[pc].y) : f2(La[j].x + T[pc].x, La[j].y - T[pc].y);
            });
        } else {
            float dx[4], dy[4], A[4], B[4], fb[3], Gb[3];
            mdiff(b - NX1, b + NX1, AX, dx);
            mdiff(b - NY1, b + NY1, AY, dy);
            mparts(AZ, SA, b, dx, dy, A);
            mparts(AZ, SB, q, Mx, My, B);
#pragma unroll
            for (int i = 0; i < 4; i++) A[i] += B[i];
            cell_field(gy, z0 - 1, fb);
            mean_G(fb, fc, Gb);
            numbers(AZ, A, Gb, Vz);
        }
    }

    for (int kz = z0; kz < z1; kz++) {
        // ---- plane kz+1 (fbar+, moments, ghosts) from the producer warps; planes z0 - 1 .. z0 + 1
        //      were awaited before the loop ----
        if (kz > z0) ok = ok && wait_full(kz + 1);
        const float *cur = Pz(kz), *prv = Pz(kz - 1), *nxt = Pz(kz + 1);
        if (ywlo || ywhi) {  // warp-uniform: the ghost row's warp makes the wall's term
            if (lane >= 1 && lane <= K::TXI && gx < nx) {
                float2 T[NX];
                wall_term<Q, FORCE, 1>(p, ctx, ywlo ? row : row - 1, kz, ywlo ? 0 : ny, T);
                float *o = wt + (((kz & 1) * 2 + (ywlo ? 0 : 1)) * 32 + lane) * 2 * NX;
#pragma unroll
                for (int i = 0; i < NX; i++) st2(o + 2 * i, T[i]);
            }
        }
        const bool zwall = !perz && kz + 1 == nz;
        if (upd && zwall) {
            float2 T[NX];
            wall_term<Q, FORCE, 2>(p, ctx, row, kz, kz + 1, T);
            sfor<NX>([&](auto pc) {
                constexpr int j = P::cross(2, pc);
                La[j] = P::e(j, 2) > 0 ? f2(La[j].x + T[pc].x, La[j].y - T[pc].y) : f2(La[j].x - T[pc].x, La[j].y + T[pc].y);
            });
        }
        // ---- y parts of plane kz: publish B_y ----
        float dz[4], Ay[4], By[4];
        float *xp = xb + ((K::BOTH_Y ? (kz & 1) * RY * 32 : 0) + row * 32 + lane) * 8;
        mdiff(prv, nxt, AZ, dz);
        if (ycol) {
            float B[4];
            mparts(AY, SA, cur, Mx, dz, Ay);
            mparts(AY, SB, cur, Mx, dz, B);
            float4 *o = reinterpret_cast<float4 *>(xp);
            if (K::BOTH_Y) o[0] = make_float4(Ay[0], Ay[1], Ay[2], Ay[3]);
            o[1] = make_float4(B[0], B[1], B[2], B[3]);
#pragma unroll
            for (int i = 0; i < 4; i++) By[i] = B[i];
        }
        // ---- differences of the interfaces' numbers, or (FORCE) N: x by shuffles, z carried ----
        float DX[NV], DZ[NV];
        float2 N[NP];
        float fn[3], Mxn[4], Myn[4];
        if constexpr (FORCE) {
#pragma unroll
            for (int j = 0; j < NP; j++) N[j] = f2(0.0f, 0.0f);
        }
        // N of the crossing pairs: + e_d (hi - lo)
        auto add_N = [&](auto dc, const float *D) __attribute__((always_inline)) {
            constexpr int d = decltype(dc)::value;
            sfor<NX>([&](auto pc) {
                constexpr int j = P::cross(d, pc);
                N[j] = P::e(j, d) > 0 ? f2(N[j].x + D[2 * pc], N[j].y - D[2 * pc + 1]) : f2(N[j].x - D[2 * pc], N[j].y + D[2 * pc + 1]);
            });
        };
        cell_field(gy, kz + 1, fn);
        if (xrow) {
            float A[4], B[4], Gb[3], V[NV], fe[3];
            mparts(AX, SA, cur, My, dz, A);
            mparts(AX, SB, cur, My, dz, B);
#pragma unroll
            for (int i = 0; i < 4; i++) A[i] += __shfl_down_sync(0xffffffffu, B[i], 1);
#pragma unroll
            for (int i = 0; i < 3; i++) fe[i] = FORCE ? __shfl_down_sync(0xffffffffu, fc[i], 1) : 0.0f;
            mean_G(fc, fe, Gb);
            if (xwall_tile) {
                WsXWall<Q> w;
#pragma unroll
                for (int i = 0; i < 4; i++) w.fm[i] = A[i];
#pragma unroll
                for (int i = 0; i < 3; i++) w.G[i] = Gb[i];
                x_wall_ws<Q, FORCE>(p, gx, cur, nxt, prv, w);
#pragma unroll
                for (int i = 0; i < 4; i++) A[i] = w.fm[i];
                sfor<NX>([&](auto pc) {
                    constexpr int j = P::cross(0, pc);
                    La[j].x -= w.hi[pc];
                    La[j].y -= w.lo[pc];
                });
            }
            numbers(AX, A, Gb, V);
#pragma unroll
            for (int i = 0; i < NV; i++) DX[i] = V[i] - __shfl_up_sync(0xffffffffu, V[i], 1);
            if constexpr (FORCE) add_N(AX, DX);
            mdiff(nxt - NY1, nxt + NY1, AY, Myn);
        }
        if (ycol) mdiff(nxt - NX1, nxt + NX1, AX, Mxn);
        if (upd) {
            float B[4], Gb[3], V[NV];
            if (zwall) {
#pragma unroll
                for (int i = 0; i < NV; i++) V[i] = 0.0f;
            } else {
                mparts(AZ, SB, nxt, Mxn, Myn, B);
#pragma unroll
                for (int i = 0; i < 4; i++) B[i] += Az[i];
                mean_G(fc, fn, Gb);
                numbers(AZ, B, Gb, V);
            }
#pragma unroll
            for (int i = 0; i < NV; i++) {
                DZ[i] = V[i] - Vz[i];
                Vz[i] = V[i];
            }
            if constexpr (FORCE) add_N(AZ, DZ);
            mparts(AZ, SA, nxt, Mxn, Myn, Az);
        }

        // consumer barrier; a wait that gave up makes every consumer leave together
        if (cons_bar_or(!ok)) {
            release(kz - 1);
            return;
        }
        if (upd) {  // the y walls' terms (their warps overwrite them after the next barrier)
            if (!pery && (gy == 0 || gy == ny - 1)) {
                auto wall = [&](const float *t, float s) __attribute__((always_inline)) {
                    sfor<NX>([&](auto pc) {
                        constexpr int j = P::cross(1, pc);
                        const float2 T = ld2(t + 2 * pc);
                        const float g = P::e(j, 1) > 0 ? s : -s;
                        La[j] = f2(fmaf(g, T.x, La[j].x), fmaf(-g, T.y, La[j].y));
                    });
                };
                const float *w = wt + ((kz & 1) * 64 + lane) * 2 * NX;
                if (gy == 0) wall(w, -1.0f);
                if (gy == ny - 1) wall(w + 64 * NX, 1.0f);
            }
        }
        float DY[NV];
        if constexpr (K::BOTH_Y) {
            if (upd) {
                const float G0[3] = {0.0f, 0.0f, 0.0f};
                const float4 hb = *reinterpret_cast<const float4 *>(xp + 32 * 8 + 4), la = *reinterpret_cast<const float4 *>(xp - 32 * 8);
                float V[NV];
                const float fn4[4] = {Ay[0] + hb.x, Ay[1] + hb.y, Ay[2] + hb.z, Ay[3] + hb.w};
                const float fs4[4] = {la.x + By[0], la.y + By[1], la.z + By[2], la.w + By[3]};
                numbers(AY, fn4, G0, DY);
                numbers(AY, fs4, G0, V);
                const bool wn = !pery && gy == ny - 1, ws = !pery && gy == 0;  // warp-uniform
#pragma unroll
                for (int i = 0; i < NV; i++) DY[i] = (wn ? 0.0f : DY[i]) - (ws ? 0.0f : V[i]);
            }
        } else {
            if (need_y) {
                if (ynwall) {
#pragma unroll
                    for (int i = 0; i < NV; i++) DY[i] = 0.0f;
                } else {
                    const float4 nb = *reinterpret_cast<const float4 *>(xp + 32 * 8 + 4);  // row + 1's B
                    const float fm[4] = {Ay[0] + nb.x, Ay[1] + nb.y, Ay[2] + nb.z, Ay[3] + nb.w};
                    float Gb[3], fy[3];
                    cell_field(gy + 1, kz, fy);
                    mean_G(fc, fy, Gb);
                    numbers(AY, fm, Gb, DY);
                }
#pragma unroll
                for (int i = 0; i < NV; i++) yv[(row * NV + i) * 32 + lane] = DY[i];
            }
            cons_bar();
        }

        // ---- steps 8-9, update of cell (gx, gy, kz) ----
        if (upd) {
            if constexpr (!K::BOTH_Y) {
#pragma unroll
                for (int i = 0; i < NV; i++) DY[i] -= yv[((row - 1) * NV + i) * 32 + lane];
            }
            if constexpr (FORCE) add_N(AY, DY);
            // sums that the pairs of a coordinate plane, and the corners, share
            float o1[3], o2[3], e1[3], e2[3];  // planes xy, xz, yz
            if constexpr (!FORCE) {
                const float *D[3] = {DX, DY, DZ};
                sfor<3>([&](auto ic) {
                    constexpr int i = ic, a = i == 2 ? 1 : 0, b = i == 0 ? 1 : 2;  // axes a < b
                    // slots of R, S for the tangential axis: first (4, 5) or second (6, 7)
                    constexpr int ab = b == (a == 0 ? 1 : 0) ? 4 : 6, ba = a == (b == 0 ? 1 : 0) ? 4 : 6;
                    o1[i] = D[a][ab] + D[b][ba + 1];
                    o2[i] = D[a][ab + 1] + D[b][ba];
                    e1[i] = 3.0f * (D[a][1 + a] + D[b][1 + b]);
                    e2[i] = 3.0f * (D[a][1 + b] + D[b][1 + a]);
                });
            }
            const float mk = -cf.two_kappa, b7 = cf.b7;
            const int64_t off = (int64_t)kz * p.plane + (int64_t)gy * p.px + gx;
            const CellRandom rnd(seed, off);
            sfor<NP>([&](auto jc) {
                constexpr int j = jc, ex = P::e(j, 0), ey = P::e(j, 1), ez = P::e(j, 2), nn = P::nnz(j);
                constexpr int i = ez != 0 ? P::pos(2, j) : 0;
                const float2 f = ld2(cur + 2 * j);
                // eq. (25): 4/3 fbar+ - 1/3 g~
                const float2 g = f2((float)Store<S>::ld(src + j * p.dstride + off),
                                    (float)Store<S>::ld(src + (Q - 1 - j) * p.dstride + off));
                const float2 u = __ffma2_rn(f2(1.0f / 3.0f, 1.0f / 3.0f), sub2(f, g), f);
                // La: the part of plane kz + 1; then the next plane's, with the part of this one
                float2 l = La[j], ln, dx, dy;
                planar(jc, nxt, ln, dx, dy);
                if constexpr (ez != 0) {
                    const float2 dzv = sub2(ld2(nxt + 2 * j), f);
                    l = __ffma2_rn(cH(ez), dzv, l);
                    ln = __ffma2_rn(cL(ez), dzv, ln);
                    if constexpr (ex != 0) {
                        l = __ffma2_rn(xm(ex * ez), dx, l);
                        ln = __ffma2_rn(xm(-ex * ez), dxc[i], ln);
                        dxc[i] = dx;
                    }
                    if constexpr (ey != 0) {
                        l = __ffma2_rn(xm(ey * ez), dy, l);
                        ln = __ffma2_rn(xm(-ey * ez), dyc[i], ln);
                        dyc[i] = dy;
                    }
                }
                La[j] = ln;
                constexpr double W = Lat<Q>::template wt<double>(j);
                constexpr float wh = (float)W, wl = (float)(W - (double)wh);
                float2 n;
                if constexpr (FORCE) {
                    n = N[j];
                } else {
                    float O, E;
                    if constexpr (nn == 1) {
                        constexpr int d = ex != 0 ? 0 : (ey != 0 ? 1 : 2);
                        const float *D = d == 0 ? DX : (d == 1 ? DY : DZ);
                        O = P::e(j, d) > 0 ? D[0] : -D[0];
                        E = 3.0f * D[1 + d];
                    } else if constexpr (nn == 2) {
                        constexpr int pl = ex == 0 ? 2 : (ey == 0 ? 1 : 0), ea = ex != 0 ? ex : ey, eb = ez != 0 ? ez : ey;
                        O = ea * eb > 0 ? o1[pl] + o2[pl] : o1[pl] - o2[pl];
                        O = ea > 0 ? O : -O;
                        E = ea * eb > 0 ? e1[pl] + e2[pl] : e1[pl] - e2[pl];
                    } else {
                        // even part at the face normal to d: Q + sum e_a e_b c_ab, c_ab = 9 m_a m_b / rho0
                        auto even = [&](const float *D, int st, int su, int stu) __attribute__((always_inline)) {
                            float v = D[8];
                            v = st > 0 ? v + D[5] : v - D[5];
                            v = su > 0 ? v + D[7] : v - D[7];
                            return stu > 0 ? v + D[9] : v - D[9];
                        };
                        const float vx = even(DX, ex * ey, ex * ez, ey * ez), vy = even(DY, ey * ex, ey * ez, ex * ez),
                                    vz = even(DZ, ez * ex, ez * ey, ex * ey);
                        O = ex > 0 ? vx : -vx;
                        O = ey > 0 ? O + vy : O - vy;
                        O = ez > 0 ? O + vz : O - vz;
                        E = 3.0f * (DX[1] + DY[2] + DZ[3]);
                        E = ex * ey > 0 ? E + e2[0] : E - e2[0];
                        E = ex * ez > 0 ? E + e2[1] : E - e2[1];
                        E = ey * ez > 0 ? E + e2[2] : E - e2[2];
                    }
                    n = f2(E + O, E - O);
                }
                // eq. (16): f~(t+dt) = f~+ - dt/|V| flux, the flux in increment form, La + b7 (W N' - La) (with
                // a force N = b7 N'), with the weight in head and tail: see the header
                float2 v;
                if constexpr (FORCE) {
                    const float2 t = __ffma2_rn(f2(wh, wh), n, __ffma2_rn(f2(wl, wl), n, __fmul2_rn(f2(-b7, -b7), l)));
                    v = __ffma2_rn(f2(mk, mk), __fadd2_rn(l, t), u);
                } else {
                    const float2 t = __ffma2_rn(f2(wh, wh), n, sub2(__fmul2_rn(f2(wl, wl), n), l));
                    v = __ffma2_rn(f2(mk, mk), __ffma2_rn(f2(b7, b7), t, l), u);
                }
                // the random bits that each value has in every kernel of the set
                store_state<S>(dst + j * p.dstride + off, v.x, sizeof(S) == 2 ? rnd.template bits<j>() : 0u);
                store_state<S>(dst + (Q - 1 - j) * p.dstride + off, v.y, sizeof(S) == 2 ? rnd.template bits<Q - 1 - j>() : 0u);
            });
            const float f0 = cur[P::REST], ur = fmaf(1.0f / 3.0f, f0 - (float)Store<S>::ld(src + NP * p.dstride + off), f0);
            store_state<S>(dst + NP * p.dstride + off, ur, sizeof(S) == 2 ? rnd.template bits<NP>() : 0u);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) { Mx[i] = Mxn[i]; My[i] = Myn[i]; }
        if constexpr (FORCE) {
#pragma unroll
            for (int i = 0; i < 3; i++) fc[i] = fn[i];
        }
        // this thread has read the ring slot of plane kz - 1 for the last time
        release(kz - 1);
    }
}

// One step by the kernel above: 8 producer + 8 consumer warps, one CTA per SM, 32 x 8 columns per tile.
template <int Q, class S, bool FORCE>
cudaError_t launch_ws(const StepParams &p, cudaStream_t stream) {
    using K = ShapeWS<Q, S, FORCE>;
    static int configured_dev = -1;
    static int sms = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        cudaError_t e = cudaFuncSetAttribute(fused_step3d_ws<Q, S, FORCE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)K::smem_bytes);
        if (e != cudaSuccess) return e;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        configured_dev = dev;
    }
    const int tiles_x = (p.nx + K::TXI - 1) / K::TXI;
    const int tiles_y = (p.ny + K::TYI - 1) / K::TYI;
    const int zchunk = zchunk_for((int64_t)tiles_x * tiles_y, p.nz, sms);
    const int nchunks = (p.nz + zchunk - 1) / zchunk;
    CUtensorMap map;
    memset(&map, 0, sizeof map);
    const cudaError_t e = encode_state_map(&map, p.src, (int)sizeof(S), std::is_same<S, __nv_bfloat16>::value, p.px,
                                           p.ny, p.nz, Q, K::BX, K::RY);
    if (e != cudaSuccess) return e;
    if (p.omega != 0.0 && !p.tfac) return cudaErrorInvalidValue;  // the kernel reads the table
    // Not chained (launch_chained): the update reads the state a second time, between its stores, which
    // costs 13% of a step by ordinary loads (forced 157 x 101 x 83) and nothing by __ldg.
    fused_step3d_ws<Q, S, FORCE><<<dim3(tiles_x, tiles_y, nchunks), K::NTHREADS, K::smem_bytes, stream>>>(p, map, zchunk);
    return cudaGetLastError();
}

}  // namespace ws27

}  // namespace dugks
