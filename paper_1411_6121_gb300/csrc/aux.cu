// aux.cu -- initialisation, moments and FP64 reductions of the DUGKS state (sm_103a).
// The per-cell sums of 32- and 16-bit states run in FP32 as unevaluated pairs; the reductions
// (residual, conservation totals) accumulate such pairs per thread and FP64 beyond.
#include "dugks_internal.h"

namespace dugks {

// Initial state (Sec. 3: the equilibrium is initialised from the given fields):
// g~ = f_eq(rho0 + p/RT, u) - W rho0 of eq. (6) (eq. (5) for the original model: rho in
// place of rho0 in the velocity part), evaluated in double and rounded once.
template <int Q, class S>
__global__ void init_kernel(const StepParams p, const double *pres, const double *vel, double rt, double c) {
    constexpr int D = Lat<Q>::D;
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    S *dst = reinterpret_cast<S *>(p.dst);
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < ncell; n += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(n % p.nx);
        const int y = (int)((n / p.nx) % p.ny);
        const int z = (int)(n / ((int64_t)p.nx * p.ny));
        const double drho = pres ? pres[n] / rt : 0.0;
        double uh[3] = {0.0, 0.0, 0.0};
        for (int a = 0; a < D; a++) uh[a] = vel ? vel[a * ncell + n] / c : 0.0;
        const double uu = uh[0] * uh[0] + uh[1] * uh[1] + uh[2] * uh[2];
        const int64_t off = (int64_t)z * p.plane + (int64_t)y * p.px + x;
#pragma unroll
        for (int k = 0; k < Q; k++) {
            double eu = 0.0;
            for (int a = 0; a < D; a++) eu += Lat<Q>::e(k, a) * uh[a];
            const double rv = p.model == 1 ? (double)p.rho0 + drho : (double)p.rho0;
            const double g = Lat<Q>::template wt<double>(k) * (drho + rv * (3.0 * eu + 4.5 * eu * eu - 1.5 * uu));
            Store<S>::st(dst + k * p.dstride + off, (typename Arith<S>::T)g);
        }
    }
}

// Cell moments in double from the stored state: drho = sum g, u = c/rho0 sum e g + G dt/2.
template <int Q, class S>
__device__ __forceinline__ void cell_moments_d(const StepParams &p, const S *src, int64_t n, int64_t ncell, double ct,
                                               double dtc, double c, double &drho, double u[3]) {
    constexpr int D = Lat<Q>::D;
    const int x = (int)(n % p.nx);
    const int y = (int)((n / p.nx) % p.ny);
    const int z = (int)(n / ((int64_t)p.nx * p.ny));
    const int64_t off = (int64_t)z * p.plane + (int64_t)y * p.px + x;
    double r = 0.0, j[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < Q; k++) {
        const double g = (double)Store<S>::ld(src + k * p.dstride + off);
        r += g;
#pragma unroll
        for (int a = 0; a < D; a++) j[a] += Lat<Q>::e(k, a) * g;
    }
    drho = r;
    // u = c j / rho0 + G dt/2 (eq. (27)); c j / rho + G dt/2 in the original model
    const double rd = p.model == 1 ? (double)p.rho0 + r : (double)p.rho0;
    for (int a = 0; a < 3; a++) {
        double G = a < D ? (double)p.g[a] : 0.0;
        if (p.field && a < D) G += (double)p.field[a * ncell + n];
        u[a] = a < D ? c / rd * j[a] + G * ct * dtc : 0.0;
    }
}

// One or two neighbouring cells (along x) of one thread: V = float or float2, the two components
// of a float2 computed with the packed FP32 instructions (each rounded as its scalar form).
__device__ __forceinline__ float vset(float, float x) { return x; }
__device__ __forceinline__ float2 vset(float2, float x) { return make_float2(x, x); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
template <class V>
__device__ __forceinline__ V vneg(V a) {
    if constexpr (sizeof(V) == 4) return -a;
    else return make_float2(-a.x, -a.y);
}
template <class V>
__device__ __forceinline__ V vsub(V a, V b) { return vfma(vset(b, -1.0f), b, a); }
__device__ __forceinline__ float vmaxabs(float m, float g) { return fmaxf(m, fabsf(g)); }
__device__ __forceinline__ float2 vmaxabs(float2 m, float2 g) {
    return make_float2(fmaxf(m.x, fabsf(g.x)), fmaxf(m.y, fabsf(g.y)));
}
// Splitting constant of a cell whose largest |g_k| is m (2^E <= m < 2^(E+1)): 1.5 * 2^(E+7), or
// zero (no splitting: plain FP32 sums) where that is near the end of the range.
__device__ __forceinline__ float split_of(float m) {
    const uint32_t e = __float_as_uint(m) & 0x7f800000u;
    return e < 0x78000000u ? __uint_as_float(e + 0x03c00000u) : 0.0f;
}
__device__ __forceinline__ float2 split_of(float2 m) { return make_float2(split_of(m.x), split_of(m.y)); }

// The state values of V's cells at element offset off (even, and the row's values 2-aligned, for
// float2).
template <class V, class S>
__device__ __forceinline__ V load_cells(const S *p) {
    if constexpr (sizeof(V) == 4) {
        return (float)Store<S>::ld(p);
    } else if constexpr (sizeof(S) == 4) {
        return __ldg(reinterpret_cast<const float2 *>(p));
    } else {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(p));
        if constexpr (std::is_same<S, __half>::value) {
            const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(&w));
            return make_float2(v.x * F16_UNSCALE, v.y * F16_UNSCALE);
        } else {
            return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
        }
    }
}

// A value as an unevaluated sum hi + lo.
template <class V>
struct Two {
    V hi, lo;
};
// Knuth's TwoSum: hi + lo == a + b exactly.
template <class V>
__device__ __forceinline__ Two<V> two_sum(V a, V b) {
    const V s = vadd(a, b), bb = vsub(s, a);
    return Two<V>{s, vadd(vsub(a, vsub(s, bb)), vsub(b, bb))};
}
// a + b of two such sums, to about 2^-47 of the larger.
template <class V>
__device__ __forceinline__ Two<V> two_add(Two<V> a, Two<V> b) {
    const Two<V> t = two_sum(a.hi, b.hi);
    return two_sum(t.hi, vadd(t.lo, vadd(a.lo, b.lo)));
}
// a b.
template <class V>
__device__ __forceinline__ Two<V> two_mul(Two<V> a, Two<V> b) {
    const V p = vmul(a.hi, b.hi);
    V e = vfma(a.hi, b.hi, vneg(p));
    e = vfma(a.hi, b.lo, e);
    e = vfma(a.lo, b.hi, e);
    const V h = vadd(p, e);
    return Two<V>{h, vsub(e, vsub(h, p))};
}
template <class V>
__device__ __forceinline__ Two<V> two_set(double x) {
    const float h = (float)x;
    return Two<V>{vset(V(), h), vset(V(), (float)(x - (double)h))};
}

// Cell sums of a 32- or 16-bit state in FP32, each as an unevaluated pair: r = sum_k g_k and
// j[a] = sum_k e_ka g_k. Every g_k is split into a head on the grid of 2^(E-16), where 2^E
// bounds the cell's largest |g_k|, and a tail (adding and subtracting 1.5 * 2^(E+7)): the sums of
// heads are exact (at most 27 terms below 2^(E+1)), and so are those of tails unless some
// |g_k| is below 2^-13 of the largest, where they round near 2^(E-40). GB300 runs FP64 at a
// 64th of its FP32 rate, so sums in FP64 would bound these kernels; TwoSum chains, which hold the
// same, took 340 dependent operations per D3Q19 cell against about 140 for the split.
template <int Q, class S, class V>
__device__ __forceinline__ void cell_sums(const StepParams &p, const S *src, int64_t off, Two<V> &r, Two<V> j[3]) {
    constexpr int D = Lat<Q>::D, C = (Q - 1) / 2;  // velocities k and Q - 1 - k are opposite, C is at rest
    V g[Q];
#pragma unroll
    for (int k = 0; k < Q; k++) g[k] = load_cells<V, S>(src + k * p.dstride + off);
    V m = vset(V(), 0.0f);
#pragma unroll
    for (int k = 0; k < Q; k++) m = vmaxabs(m, g[k]);
    const V sp = split_of(m), sn = vneg(sp);
    r.hi = vadd(vadd(g[C], sp), sn);
    r.lo = vsub(g[C], r.hi);
#pragma unroll
    for (int a = 0; a < 3; a++) j[a].hi = j[a].lo = vset(V(), 0.0f);
#pragma unroll
    for (int k = 0; k < C; k++) {
        const V h0 = vadd(vadd(g[k], sp), sn), h1 = vadd(vadd(g[Q - 1 - k], sp), sn);
        const V l0 = vsub(g[k], h0), l1 = vsub(g[Q - 1 - k], h1);
        r.hi = vadd(r.hi, vadd(h0, h1));
        r.lo = vadd(r.lo, vadd(l0, l1));
        const V dh = vsub(h0, h1), dl = vsub(l0, l1);
#pragma unroll
        for (int a = 0; a < D; a++) {
            if (Lat<Q>::e(k, a) > 0) { j[a].hi = vadd(j[a].hi, dh); j[a].lo = vadd(j[a].lo, dl); }
            if (Lat<Q>::e(k, a) < 0) { j[a].hi = vsub(j[a].hi, dh); j[a].lo = vsub(j[a].lo, dl); }
        }
    }
}

// Element offset of cell n (x fastest) in the padded state layout: n itself when the rows carry
// no padding; otherwise by 32-bit divisions where the cells allow it.
__device__ __forceinline__ int64_t cell_offset(const StepParams &p, int64_t n, int64_t ncell) {
    if (p.px == p.nx) return n;
    if (ncell <= 0x7fffffff) {
        const uint32_t row = (uint32_t)n / (uint32_t)p.nx, x = (uint32_t)n - row * (uint32_t)p.nx;
        return (int64_t)row * p.px + x;  // rows are px apart in every plane (plane = px ny)
    }
    const int64_t row = n / p.nx;
    return row * p.px + (n - row * p.nx);
}

// The FP32 output of V's cells.
__device__ __forceinline__ void store_out(float *p, float v) { *p = v; }
__device__ __forceinline__ void store_out(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
__device__ __forceinline__ float load_field(const float *p, float) { return __ldg(p); }
__device__ __forceinline__ float2 load_field(const float *p, float2) { return make_float2(__ldg(p), __ldg(p + 1)); }
__device__ __forceinline__ float model_factor(float cr, float rho0, float dr) { return cr * rho0 / (rho0 + dr); }
__device__ __forceinline__ float2 model_factor(float2 cr, float rho0, float2 dr) {
    return make_float2(cr.x * rho0 / (rho0 + dr.x), cr.y * rho0 / (rho0 + dr.y));
}

// Moments as FP32 output from a 32- or 16-bit state, without FP64 arithmetic.
template <int Q, class S, class V>
__device__ __forceinline__ void cell_moments_out_f(const StepParams &p, const S *src, int64_t n, int64_t ncell,
                                                   float ctdt, float c_over_rho0, float rt, float *out) {
    constexpr int D = Lat<Q>::D;
    Two<V> r, j[3];
    cell_sums<Q, S, V>(p, src, cell_offset(p, n, ncell), r, j);
    const V dr = vadd(r.hi, r.lo);
    store_out(out + n, vmul(dr, vset(V(), rt)));
    // c / rho0, or c / rho in the original model
    V cr = vset(V(), c_over_rho0);
    if (p.model == 1) cr = model_factor(cr, (float)p.rho0, dr);
#pragma unroll
    for (int a = 0; a < D; a++) {
        V G = vset(V(), (float)p.g[a]);
        if (p.field) G = vadd(G, load_field(p.field + a * ncell + n, V()));
        store_out(out + (a + 1) * ncell + n, vfma(cr, vadd(j[a].hi, j[a].lo), vmul(G, vset(V(), ctdt))));
    }
}

// Moments (eq. (27)): out[0] = p = (rho - rho0) RT, out[1+a] = u_a; [dim+1][ncell]. A pass over
// the state bound by its bytes: V = float2 takes two cells per thread (64-bit loads, packed
// arithmetic). 256^3 D3Q19 FP32, 1.54 GB: 536 us before, 268 us now (5.7 TB/s).
template <int Q, class S, class V>
__global__ void __launch_bounds__(256) moments_kernel(const StepParams p, double ct, double rt, double c, float *out) {
    constexpr int D = Lat<Q>::D, NV = sizeof(V) / 4;
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    const S *src = reinterpret_cast<const S *>(p.src);
    const int64_t t0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * NV, stride = (int64_t)gridDim.x * blockDim.x * NV;
    if constexpr (sizeof(S) != 8) {
        const float ctdt = (float)(ct * 0.5 * p.dt), cr = (float)(c / p.rho0), rtf = (float)rt;
        for (int64_t n = t0; n < ncell; n += stride) cell_moments_out_f<Q, S, V>(p, src, n, ncell, ctdt, cr, rtf, out);
    } else {
        for (int64_t n = t0; n < ncell; n += stride) {
            double drho, u[3];
            cell_moments_d<Q, S>(p, src, n, ncell, ct, 0.5 * p.dt, c, drho, u);
            out[n] = (float)(drho * rt);
            for (int a = 0; a < D; a++) out[(a + 1) * ncell + n] = (float)u[a];
        }
    }
}

// Steady-state residual of Sec. 3.1 and conservation totals, in FP64. Per block:
// s[0] = sum |u - u_prev|^2, s[1] = sum |u|^2, s[2] = sum rho, s[3+a] = sum rho0 u_a.
// u_prev is overwritten with u. Deterministic: fixed per-block order, fixed final order.
constexpr int RES_THREADS = 256;
constexpr int RES_SLOTS = 8;

// The block's sums of its threads' s into its row of `partials`.
__device__ __forceinline__ void block_partials(const double s[RES_SLOTS], double *partials) {
    __shared__ double red[RES_THREADS / 32][RES_SLOTS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < RES_SLOTS; i++) {
        double v = s[i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[warp][i] = v;
    }
    __syncthreads();
    if (threadIdx.x < RES_SLOTS) {
        double v = 0.0;
        for (int w = 0; w < RES_THREADS / 32; w++) v += red[w][threadIdx.x];
        partials[blockIdx.x * RES_SLOTS + threadIdx.x] = v;
    }
}

// FP64 states, and the original model (whose velocity divides by the local density).
template <int Q, class S>
__global__ void __launch_bounds__(RES_THREADS) residual_kernel(const StepParams p, double ct, double c, double *uprev,
                                                                int have_prev, double *partials) {
    constexpr int D = Lat<Q>::D;
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    const S *src = reinterpret_cast<const S *>(p.src);
    double s[RES_SLOTS] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < ncell; n += (int64_t)gridDim.x * blockDim.x) {
        double drho, u[3];
        cell_moments_d<Q, S>(p, src, n, ncell, ct, 0.5 * p.dt, c, drho, u);
        for (int a = 0; a < D; a++) {
            const double du = u[a] - (have_prev ? uprev[a * ncell + n] : 0.0);
            s[0] += du * du;
            s[1] += u[a] * u[a];
            s[3 + a] += (p.model == 1 ? (double)p.rho0 + drho : (double)p.rho0) * u[a];  // rho0 u, or rho u
            uprev[a * ncell + n] = u[a];
        }
        s[2] += (double)p.rho0 + drho;
    }
    block_partials(s, partials);
}

// 32- and 16-bit states of the incompressible model. Each cell's velocity u / c = sum e g / rho0 +
// shift is formed, differenced, squared and summed over the thread's cells as an unevaluated
// pair of FP32 values (about 47 bits; the squares are taken of 2^30 u / c, which keeps the low
// parts of slow flows in range), and goes to FP64 once per thread: a pass over the state bound
// by its bytes instead of 37 FP64 instructions per cell at a 64th of the FP32 rate. PAIR: u_prev
// is the handle's own and holds those pairs; otherwise it is the caller's array of doubles.
// 256^3 D3Q19 FP32, 2.08 GB: 2626 us before, 316 us now (6.6 TB/s).
constexpr float SQ_SCALE = 1073741824.0f;  // 2^30
// u_prev / c of V's cells (zero before any).
template <class V, bool PAIR>
__device__ __forceinline__ Two<V> load_prev(const double *up, int have_prev, double c) {
    static_assert(PAIR || sizeof(V) == 4, "the caller's array is taken one cell at a time");
    Two<V> r = {vset(V(), 0.0f), vset(V(), 0.0f)};
    if (!have_prev) return r;
    if constexpr (!PAIR) {
        r = two_set<V>(*up / c);
    } else if constexpr (sizeof(V) == 4) {
        const float2 v = *reinterpret_cast<const float2 *>(up);
        r = Two<V>{v.x, v.y};
    } else {
        const float4 v = *reinterpret_cast<const float4 *>(up);
        r = Two<V>{make_float2(v.x, v.z), make_float2(v.y, v.w)};
    }
    return r;
}
template <int Q, class S, class V, bool PAIR>
__global__ void __launch_bounds__(RES_THREADS) residual_kernel_f(const StepParams p, double ct, double c, double *uprev,
                                                                  int have_prev, double *partials) {
    constexpr int D = Lat<Q>::D, NV = sizeof(V) / 4;
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    const S *src = reinterpret_cast<const S *>(p.src);
    const Two<V> zero = {vset(V(), 0.0f), vset(V(), 0.0f)};
    const Two<V> ir = two_set<V>(1.0 / p.rho0), cs = two_set<V>(ct * 0.5 * p.dt / c);  // shift = (g + field) cs
    Two<V> sh[3];
#pragma unroll
    for (int a = 0; a < 3; a++) sh[a] = two_set<V>(p.g[a] * (ct * 0.5 * p.dt / c));
    const bool shifted = p.g[0] != 0.0 || p.g[1] != 0.0 || p.g[2] != 0.0;
    Two<V> s0 = zero, s1 = zero, s2 = zero, su[3] = {zero, zero, zero};
    int64_t cells = 0;
    for (int64_t n = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * NV; n < ncell;
         n += (int64_t)gridDim.x * blockDim.x * NV) {
        // u_prev first: its loads must not wait behind the stores of u below (which the compiler
        // has to order, axis by axis) or behind the sums
        Two<V> before[3];
#pragma unroll
        for (int a = 0; a < D; a++) before[a] = load_prev<V, PAIR>(uprev + a * ncell + n, have_prev, c);
        Two<V> r, j[3];
        cell_sums<Q, S, V>(p, src, cell_offset(p, n, ncell), r, j);
        s2 = two_add(s2, r);
        cells += NV;
#pragma unroll
        for (int a = 0; a < D; a++) {
            Two<V> u = two_mul(two_sum(j[a].hi, j[a].lo), ir);
            if (shifted) u = two_add(u, sh[a]);
            if (p.field) u = two_add(u, two_mul(Two<V>{load_field(p.field + a * ncell + n, V()), zero.lo}, cs));
            double *up = uprev + a * ncell + n;
            if constexpr (!PAIR) *up = ((double)u.hi + (double)u.lo) * c;
            else if constexpr (NV == 2) *reinterpret_cast<float4 *>(up) = make_float4(u.hi.x, u.lo.x, u.hi.y, u.lo.y);
            else *reinterpret_cast<float2 *>(up) = make_float2(u.hi, u.lo);
            Two<V> du = two_add(u, Two<V>{vneg(before[a].hi), vneg(before[a].lo)});
            du = Two<V>{vmul(du.hi, vset(V(), SQ_SCALE)), vmul(du.lo, vset(V(), SQ_SCALE))};
            const Two<V> us = {vmul(u.hi, vset(V(), SQ_SCALE)), vmul(u.lo, vset(V(), SQ_SCALE))};
            s0 = two_add(s0, two_mul(du, du));
            s1 = two_add(s1, two_mul(us, us));
            su[a] = two_add(su[a], u);
        }
    }
    auto total = [](const Two<V> &t) -> double {
        if constexpr (NV == 2) return ((double)t.hi.x + (double)t.lo.x) + ((double)t.hi.y + (double)t.lo.y);
        else return (double)t.hi + (double)t.lo;
    };
    const double q2 = (c / SQ_SCALE) * (c / SQ_SCALE);
    double s[RES_SLOTS] = {total(s0) * q2, total(s1) * q2, p.rho0 * (double)cells + total(s2), 0, 0, 0, 0, 0};
#pragma unroll
    for (int a = 0; a < D; a++) s[3 + a] = p.rho0 * c * total(su[a]);
    block_partials(s, partials);
}

// One block: warp i sums slot i, lane l the blocks l, l + 32, ... in index order, then a butterfly
// (one thread per slot took 320 us for 4096 blocks, a chain of FP64 additions).
__global__ void __launch_bounds__(32 * RES_SLOTS) residual_final(const double *partials, int nblocks, double *out) {
    const int lane = threadIdx.x & 31, slot = threadIdx.x >> 5;
    double v = 0.0;
    for (int b = lane; b < nblocks; b += 32) v += partials[b * RES_SLOTS + slot];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) out[slot] = v;
}

__global__ void advance_kernel(long long *ctr, long long n) { *ctr += n; }

__global__ void time_factors_kernel(const long long *ctr, int n, double omega, double dt, double inv_c,
                                    TimeFactors *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = eval_time_factors(omega, dt, inv_c, (double)(*ctr) + (double)i);
}

static int grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    return (int)(b < 1 ? 1 : (b > 65535 * 8 ? 65535 * 8 : b));
}

// One block per 256 cells up to 608 (four per SM), which then stride: a mesh of 16,384 cells in
// FP64 took 41 us on the 8 blocks of one per 2048 cells, 11 us on 64.
int residual_blocks(int64_t ncell) {
    const int64_t b = (ncell + RES_THREADS - 1) / RES_THREADS;
    return (int)(b < 1 ? 1 : (b > 608 ? 608 : b));
}

// Two cells per thread: the rows hold whole pairs, and every pair starts on its own size.
static bool pairs_ok(const StepParams &p, int store, const void *out, size_t out_align) {
    const size_t pair = store == 0 ? 8 : 4;
    return p.nx % 2 == 0 && p.px % 2 == 0 && p.dstride % 2 == 0 && (uintptr_t)p.src % pair == 0 &&
           (uintptr_t)out % out_align == 0;
}

template <int Q>
static cudaError_t init_q(int store, const StepParams &p, const double *pres, const double *vel, double rt,
                          cudaStream_t st) {
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    const double c = sqrt(3.0 * rt);
    const int g = grid_for(ncell, 256);
    if (store == 0) init_kernel<Q, float><<<g, 256, 0, st>>>(p, pres, vel, rt, c);
    else if (store == 1) init_kernel<Q, __nv_bfloat16><<<g, 256, 0, st>>>(p, pres, vel, rt, c);
    else if (store == 2) init_kernel<Q, __half><<<g, 256, 0, st>>>(p, pres, vel, rt, c);
    else init_kernel<Q, double><<<g, 256, 0, st>>>(p, pres, vel, rt, c);
    return cudaGetLastError();
}

template <int Q, class S>
static void moments_s(const StepParams &p, int store, double ct, double rt, double c, float *out, cudaStream_t st) {
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    if (pairs_ok(p, store, out, 8))
        moments_kernel<Q, S, float2><<<grid_for(ncell / 2, 256), 256, 0, st>>>(p, ct, rt, c, out);
    else
        moments_kernel<Q, S, float><<<grid_for(ncell, 256), 256, 0, st>>>(p, ct, rt, c, out);
}

template <int Q>
static cudaError_t moments_q(int store, const StepParams &p, double t, double rt, float *out, cudaStream_t st) {
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    const double c = sqrt(3.0 * rt);
    const double ct = cos(p.omega * t);
    if (store == 0) moments_s<Q, float>(p, store, ct, rt, c, out, st);
    else if (store == 1) moments_s<Q, __nv_bfloat16>(p, store, ct, rt, c, out, st);
    else if (store == 2) moments_s<Q, __half>(p, store, ct, rt, c, out, st);
    else moments_kernel<Q, double, float><<<grid_for(ncell, 256), 256, 0, st>>>(p, ct, rt, c, out);
    return cudaGetLastError();
}

template <int Q, class S>
static void residual_s(const StepParams &p, int store, double ct, double c, double *uprev, bool pair, int have_prev,
                       double *partials, int nblocks, cudaStream_t st) {
    if (!pair) residual_kernel_f<Q, S, float, false><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
    else if (pairs_ok(p, store, uprev, 16))
        residual_kernel_f<Q, S, float2, true><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
    else
        residual_kernel_f<Q, S, float, true><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
}

template <int Q>
static cudaError_t residual_q(int store, const StepParams &p, double t, double rt, double *uprev, bool pair,
                              int have_prev, double *partials, int nblocks, double *out, cudaStream_t st) {
    const double c = sqrt(3.0 * rt);
    const double ct = cos(p.omega * t);
    const bool orig = p.model == 1;
    if (store == 0 && !orig) residual_s<Q, float>(p, store, ct, c, uprev, pair, have_prev, partials, nblocks, st);
    else if (store == 1 && !orig)
        residual_s<Q, __nv_bfloat16>(p, store, ct, c, uprev, pair, have_prev, partials, nblocks, st);
    else if (store == 2 && !orig) residual_s<Q, __half>(p, store, ct, c, uprev, pair, have_prev, partials, nblocks, st);
    else if (store == 0) residual_kernel<Q, float><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
    else if (store == 1)
        residual_kernel<Q, __nv_bfloat16><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
    else if (store == 2) residual_kernel<Q, __half><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
    else residual_kernel<Q, double><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    residual_final<<<1, 32 * RES_SLOTS, 0, st>>>(partials, nblocks, out);
    return cudaGetLastError();
}

cudaError_t launch_init(int q, int store, const StepParams &p, const double *pres, const double *vel, double rt,
                        cudaStream_t st) {
    switch (q) {
        case 9: return init_q<9>(store, p, pres, vel, rt, st);
        case 19: return init_q<19>(store, p, pres, vel, rt, st);
        case 27: return init_q<27>(store, p, pres, vel, rt, st);
    }
    return cudaErrorNotSupported;
}

cudaError_t launch_moments(int q, int store, const StepParams &p, double t, double rt, float *out, cudaStream_t st) {
    switch (q) {
        case 9: return moments_q<9>(store, p, t, rt, out, st);
        case 19: return moments_q<19>(store, p, t, rt, out, st);
        case 27: return moments_q<27>(store, p, t, rt, out, st);
    }
    return cudaErrorNotSupported;
}

cudaError_t launch_residual(int q, int store, const StepParams &p, double t, double rt, double *uprev, bool pair,
                            int have_prev, double *partials, int nblocks, double *out, cudaStream_t st) {
    switch (q) {
        case 9: return residual_q<9>(store, p, t, rt, uprev, pair, have_prev, partials, nblocks, out, st);
        case 19: return residual_q<19>(store, p, t, rt, uprev, pair, have_prev, partials, nblocks, out, st);
        case 27: return residual_q<27>(store, p, t, rt, uprev, pair, have_prev, partials, nblocks, out, st);
    }
    return cudaErrorNotSupported;
}

cudaError_t launch_time_factors(const long long *ctr, int n, double omega, double dt, double inv_c, TimeFactors *out,
                                cudaStream_t st) {
    time_factors_kernel<<<(n + 31) / 32, 32, 0, st>>>(ctr, n, omega, dt, inv_c, out);
    return cudaGetLastError();
}

cudaError_t launch_advance(long long *ctr, long long n, cudaStream_t st) {
    advance_kernel<<<1, 1, 0, st>>>(ctr, n);
    return cudaGetLastError();
}

}  // namespace dugks
