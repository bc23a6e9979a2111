// aux.cu -- initialisation, moments and FP64 reductions of the DUGKS state (sm_103a).
// The per-cell sums of 32- and 16-bit states run in FP32 as unevaluated pairs; the reductions
// (residual, conservation totals) go on in FP64.
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
// Cell sums of a 32- or 16-bit state in FP32, each as an unevaluated pair: r = sum_k g_k and
// j[a] = sum_k e_ka g_k. With 2^E <= max |g_k| < 2^(E+1) every g_k is cut into a head on the grid of 2^(E-16)
// (adding and subtracting 1.5 * 2^(E+7)), a middle part on that of 2^(E-33) and a tail: the sums of heads and of
// middle parts are exact (at most 27 terms below 2^(E+1) and 2^(E-17)), the tails' round below 2^(E-50), and
// head + middle is exact as a pair, whose low half takes the tail: 2^-48 of the sum itself. (Compensated
// summation with TwoSum held 2^-48 of sum |g|, in 340 dependent operations per D3Q19 cell; with heads and
// tails only, cells whose large values cancel lost 2^-41.) GB300 runs FP64 at a 64th of its FP32 rate, so
// sums in FP64 would bound these kernels.
template <class V>
struct Three {
    V h, m, t;
    __device__ __forceinline__ void zero() { h = m = t = vset(V(), 0.0f); }
    __device__ __forceinline__ void add(const Three &b) { h = vadd(h, b.h); m = vadd(m, b.m); t = vadd(t, b.t); }
    __device__ __forceinline__ void sub(const Three &b) { h = vsub(h, b.h); m = vsub(m, b.m); t = vsub(t, b.t); }
    __device__ __forceinline__ Two<V> pair() const {
        const Two<V> p = two_sum(h, m);
        return Two<V>{p.hi, vadd(p.lo, t)};
    }
};
template <int Q, class V>
__device__ __forceinline__ void cell_sums(const V g[Q], Two<V> &r, Two<V> j[3]) {
    constexpr int D = Lat<Q>::D, C = (Q - 1) / 2;  // velocities k and Q - 1 - k are opposite, C is at rest
    V big = vset(V(), 0.0f);
#pragma unroll
    for (int k = 0; k < Q; k++) big = vmaxabs(big, g[k]);
    const V sp = split_of(big), sn = vneg(sp), mp = vmul(sp, vset(V(), 0x1p-17f)), mn = vneg(mp);
    auto cut = [&](V v) __attribute__((always_inline)) {
        Three<V> c;
        c.h = vadd(vadd(v, sp), sn);
        const V l = vsub(v, c.h);
        c.m = vadd(vadd(l, mp), mn);
        c.t = vsub(l, c.m);
        return c;
    };
    Three<V> R = cut(g[C]), J[3];
#pragma unroll
    for (int a = 0; a < 3; a++) J[a].zero();
#pragma unroll
    for (int k = 0; k < C; k++) {
        const Three<V> p = cut(g[k]), n = cut(g[Q - 1 - k]);
        Three<V> s = p, d = p;
        s.add(n);
        d.sub(n);
        R.add(s);
#pragma unroll
        for (int a = 0; a < D; a++) {
            if (Lat<Q>::e(k, a) > 0) J[a].add(d);
            if (Lat<Q>::e(k, a) < 0) J[a].sub(d);
        }
    }
    r = R.pair();
#pragma unroll
    for (int a = 0; a < D; a++) j[a] = J[a].pair();
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
    V g[Q];
    const int64_t off = cell_offset(p, n, ncell);
#pragma unroll
    for (int k = 0; k < Q; k++) g[k] = load_cells<V, S>(src + k * p.dstride + off);
    Two<V> r, j[3];
    cell_sums<Q, V>(g, r, j);
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
// arithmetic). 256^3 D3Q19 FP32, 1.54 GB: 536 us before, 294 us now (5.2 TB/s).
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

// FP32 values as doubles by integer operations: a conversion takes the FP64 unit, at a 64th of the FP32 rate.
// Not for subnormal, infinite and NaN values (odd_value).
__device__ __forceinline__ bool odd_value(float x) {
    const uint32_t m = __float_as_uint(x) & 0x7fffffffu;
    return m - 0x00800000u >= 0x7f000000u && m != 0;
}
__device__ __forceinline__ double widen(float x) {
    const uint32_t b = __float_as_uint(x), m = b & 0x7fffffffu, h = m != 0 ? (m >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)((b & 0x80000000u) | h), (int)(b << 29));
}
template <bool ODD>
__device__ __forceinline__ double2 widen(Two<float2> v) {
    if constexpr (ODD) return make_double2((double)v.hi.x + (double)v.lo.x, (double)v.hi.y + (double)v.lo.y);
    else return make_double2(widen(v.hi.x) + widen(v.lo.x), widen(v.hi.y) + widen(v.lo.y));
}
__device__ __forceinline__ bool odd_value(Two<float2> v) {
    return odd_value(v.hi.x) || odd_value(v.hi.y) || odd_value(v.lo.x) || odd_value(v.lo.y);
}

// FP64 states.
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

// 32- and 16-bit states: the cell sums in FP32 (cell_sums), then FP64 per cell: u, its difference, the squares
// and the sums. A thread takes the cells n and n + 1, VEC: by loads of both at once; the order of the sums
// is the same either way. ORIG: the original model, whose velocity divides by the local density.
// 256^3 D3Q19 FP32, 2.08 GB (us): 2626 with one thread per cell, conversions and u_prev behind the stores,
// 670 now: 21 FP64 instructions per cell, the FP64 unit 83% busy. (Pairs of floats all the way took 316, but
// hold 47 bits and the range of FP32.)
template <int Q, class S, bool VEC, bool ORIG>
__global__ void __launch_bounds__(RES_THREADS) residual_kernel_f(const StepParams p, double ct, double c, double *uprev,
                                                                  int have_prev, double *partials) {
    constexpr int D = Lat<Q>::D;
    const int64_t ncell = (int64_t)p.nx * p.ny * p.nz;
    const S *src = reinterpret_cast<const S *>(p.src);
    const double cr0 = c / p.rho0, dtc = 0.5 * p.dt;
    double shift[3];
#pragma unroll
    for (int a = 0; a < 3; a++) shift[a] = p.g[a] * ct * dtc;
    double s[RES_SLOTS] = {0, 0, 0, 0, 0, 0, 0, 0};
    int64_t cells = 0;
    for (int64_t n = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); n < ncell;
         n += 2 * (int64_t)gridDim.x * blockDim.x) {
        const int64_t n1 = VEC || n + 1 < ncell ? n + 1 : n;
        // u_prev first: its loads must not wait behind the stores of u below (which the compiler
        // has to order, axis by axis) or behind the sums
        double2 before[3];
#pragma unroll
        for (int a = 0; a < D; a++) {
            const double *up = uprev + a * ncell;
            if (!have_prev) before[a] = make_double2(0.0, 0.0);
            else if constexpr (VEC) before[a] = *reinterpret_cast<const double2 *>(up + n);
            else before[a] = make_double2(up[n], up[n1]);
        }
        float2 g[Q];
        const int64_t off = cell_offset(p, n, ncell), off1 = VEC ? off : cell_offset(p, n1, ncell);
#pragma unroll
        for (int k = 0; k < Q; k++) {
            const S *q = src + k * p.dstride;
            if constexpr (VEC) g[k] = load_cells<float2, S>(q + off);
            else g[k] = make_float2(Store<S>::ld(q + off), Store<S>::ld(q + off1));
        }
        Two<float2> r, j[3];
        cell_sums<Q, float2>(g, r, j);
        double2 u[3], drho;  // u: the momenta first
        bool odd = odd_value(r);
#pragma unroll
        for (int a = 0; a < D; a++) odd = odd || odd_value(j[a]);
        if (odd) {
            drho = widen<true>(r);
#pragma unroll
            for (int a = 0; a < D; a++) u[a] = widen<true>(j[a]);
        } else {
            drho = widen<false>(r);
#pragma unroll
            for (int a = 0; a < D; a++) u[a] = widen<false>(j[a]);
        }
        double2 cr = make_double2(cr0, cr0);
        if constexpr (ORIG) cr = make_double2(c / (p.rho0 + drho.x), c / (p.rho0 + drho.y));
        double2 sh[3];
#pragma unroll
        for (int a = 0; a < D; a++) sh[a] = make_double2(shift[a], shift[a]);
        if (p.field) {  // one block of all axes: a real branch, not predicated FP64 operations
#pragma unroll
            for (int a = 0; a < D; a++) {
                const float *f = p.field + a * ncell;
                sh[a] = make_double2((p.g[a] + (double)__ldg(f + n)) * ct * dtc, (p.g[a] + (double)__ldg(f + n1)) * ct * dtc);
            }
        }
#pragma unroll
        for (int a = 0; a < D; a++) {
            u[a] = make_double2(fma(cr.x, u[a].x, sh[a].x), fma(cr.y, u[a].y, sh[a].y));
            double *up = uprev + a * ncell;
            if constexpr (VEC) *reinterpret_cast<double2 *>(up + n) = u[a];
            else {
                up[n] = u[a].x;
                if (n1 != n) up[n1] = u[a].y;
            }
        }
        auto take = [&](double dr, const double v[3], const double b[3]) __attribute__((always_inline)) {
            const double rho = ORIG ? p.rho0 + dr : p.rho0;
#pragma unroll
            for (int a = 0; a < D; a++) {
                const double du = v[a] - b[a];
                s[0] = fma(du, du, s[0]);
                s[1] = fma(v[a], v[a], s[1]);
                s[3 + a] = fma(rho, v[a], s[3 + a]);  // rho0 u, or rho u
            }
            s[2] += dr;
            cells++;
        };
        const double ux[3] = {u[0].x, u[1].x, D == 3 ? u[2].x : 0.0}, bx[3] = {before[0].x, before[1].x, D == 3 ? before[2].x : 0.0};
        take(drho.x, ux, bx);
        if (n1 != n) {
            const double uy[3] = {u[0].y, u[1].y, D == 3 ? u[2].y : 0.0}, by[3] = {before[0].y, before[1].y, D == 3 ? before[2].y : 0.0};
            take(drho.y, uy, by);
        }
    }
    s[2] = fma(p.rho0, (double)cells, s[2]);
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

template <int Q, class S, bool ORIG>
static void residual_m(const StepParams &p, int store, double ct, double c, double *uprev, int have_prev, double *partials,
                       int nblocks, cudaStream_t st) {
    if (pairs_ok(p, store, uprev, 16))
        residual_kernel_f<Q, S, true, ORIG><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
    else
        residual_kernel_f<Q, S, false, ORIG><<<nblocks, RES_THREADS, 0, st>>>(p, ct, c, uprev, have_prev, partials);
}

template <int Q, class S>
static void residual_s(const StepParams &p, int store, double ct, double c, double *uprev, int have_prev, double *partials,
                       int nblocks, cudaStream_t st) {
    if (p.model == 1) residual_m<Q, S, true>(p, store, ct, c, uprev, have_prev, partials, nblocks, st);
    else residual_m<Q, S, false>(p, store, ct, c, uprev, have_prev, partials, nblocks, st);
}

template <int Q>
static cudaError_t residual_q(int store, const StepParams &p, double t, double rt, double *uprev, int have_prev,
                              double *partials, int nblocks, double *out, cudaStream_t st) {
    const double c = sqrt(3.0 * rt);
    const double ct = cos(p.omega * t);
    if (store == 0) residual_s<Q, float>(p, store, ct, c, uprev, have_prev, partials, nblocks, st);
    else if (store == 1) residual_s<Q, __nv_bfloat16>(p, store, ct, c, uprev, have_prev, partials, nblocks, st);
    else if (store == 2) residual_s<Q, __half>(p, store, ct, c, uprev, have_prev, partials, nblocks, st);
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

cudaError_t launch_residual(int q, int store, const StepParams &p, double t, double rt, double *uprev,
                            int have_prev, double *partials, int nblocks, double *out, cudaStream_t st) {
    switch (q) {
        case 9: return residual_q<9>(store, p, t, rt, uprev, have_prev, partials, nblocks, out, st);
        case 19: return residual_q<19>(store, p, t, rt, uprev, have_prev, partials, nblocks, out, st);
        case 27: return residual_q<27>(store, p, t, rt, uprev, have_prev, partials, nblocks, out, st);
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
