// step2d_cell.cu -- instantiations and launchers of the one-cell-per-thread D2Q9 kernel
// (dugks_step2d_cell.cuh): BF16 storage, and the F32 and F16 meshes that it is the faster one for.
#include <algorithm>

#include "dugks_internal.h"
#include "dugks_step2d_cell.cuh"

namespace dugks {

namespace {

// Blocks per SM of a kernel of one device, and its SMs.
struct Resident {
    int dev = -1, blocks = 1, sms = 1;
};

template <class S, int RY, bool FORCE, bool BATCH>
cudaError_t configure(const Resident **out) {
    using K = Shape2<RY, S>;
    static Resident r;
    int dev = 0;
    cudaGetDevice(&dev);
    if (r.dev != dev) {
        const void *fn;
        if constexpr (BATCH) fn = (const void *)fused_step2d_cell_batch<S, RY, FORCE>;
        else fn = (const void *)fused_step2d_cell<S, RY, FORCE>;
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::smem_bytes);
        if (e != cudaSuccess) return e;
        int blocks = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, 32 * RY, K::smem_bytes);
        r.blocks = std::max(1, blocks);
        cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev);
        r.dev = dev;
    }
    *out = &r;
    return cudaSuccess;
}

template <class S, int RY, bool FORCE>
cudaError_t launch_one(const StepParams &p, cudaStream_t stream) {
    using K = Shape2<RY, S>;
    const Resident *r;
    const cudaError_t e = configure<S, RY, FORCE, false>(&r);
    if (e != cudaSuccess) return e;
    const dim3 grid((p.nx + K::TXI - 1) / K::TXI, (p.ny + K::TYI - 1) / K::TYI);
    return launch_chained(fused_step2d_cell<S, RY, FORCE>, grid, dim3(32, RY), K::smem_bytes, stream, r->blocks, r->sms, p);
}

template <int RY, bool FORCE>
cudaError_t launch_many(const StepParams *params, const int4 *items, int nitems, int parity, cudaStream_t stream) {
    using S = __nv_bfloat16;
    using K = Shape2<RY, S>;
    const Resident *r;
    const cudaError_t e = configure<S, RY, FORCE, true>(&r);
    if (e != cudaSuccess) return e;
    const int grid = std::min(nitems, r->blocks * r->sms);  // persistent: the resident blocks, at most the items
    if (grid < 1) return cudaSuccess;
    return launch_chained(fused_step2d_cell_batch<S, RY, FORCE>, dim3(grid), dim3(32, RY), K::smem_bytes, stream, r->blocks,
                          r->sms, params, items, nitems, parity);
}

template <bool FORCE>
cudaError_t one(const StepParams &p, int store, int ry, cudaStream_t st) {
    if (ry == 8 && store == 0) return launch_one<float, 8, FORCE>(p, st);
    if (ry == 8 && store == 2) return launch_one<__half, 8, FORCE>(p, st);
    if (store != 1) return cudaErrorNotSupported;
    if (ry == 4) return launch_one<__nv_bfloat16, 4, FORCE>(p, st);
    if (ry == 8) return launch_one<__nv_bfloat16, 8, FORCE>(p, st);
    if (ry == 16) return launch_one<__nv_bfloat16, 16, FORCE>(p, st);
    return cudaErrorNotSupported;
}

template <bool FORCE>
cudaError_t many(const StepParams *params, const int4 *items, int nitems, int parity, int ry, cudaStream_t st) {
    if (ry == 4) return launch_many<4, FORCE>(params, items, nitems, parity, st);
    if (ry == 8) return launch_many<8, FORCE>(params, items, nitems, parity, st);
    if (ry == 16) return launch_many<16, FORCE>(params, items, nitems, parity, st);
    return cudaErrorNotSupported;
}

template <class S>
int warps(const StepParams &p, bool force) {
    using K = Shape2<8, S>;
    const Resident *r;
    if ((force ? configure<S, 8, true, false>(&r) : configure<S, 8, false, false>(&r)) != cudaSuccess) return 0;
    const int64_t blocks = (int64_t)((p.nx + K::TXI - 1) / K::TXI) * ((p.ny + K::TYI - 1) / K::TYI);
    const int64_t per_sm = (blocks + r->sms - 1) / r->sms;
    return per_sm <= r->blocks ? (int)per_sm * 8 : 0;
}

}  // namespace

int step2d_cell_warps(const StepParams &p, int store, bool force) {
    return store == 0 ? warps<float>(p, force) : store == 2 ? warps<__half>(p, force) : 0;
}

cudaError_t launch_step2d_cell(const StepParams &p, int store, int ry, cudaStream_t stream) {
    const bool force = p.field != nullptr || p.g[0] != 0.0 || p.g[1] != 0.0;
    return force ? one<true>(p, store, ry, stream) : one<false>(p, store, ry, stream);
}

cudaError_t launch_step2d_batch_bf16(const StepParams *params, const int4 *items, int nitems, int parity, int ry,
                                     bool force, cudaStream_t stream) {
    return force ? many<true>(params, items, nitems, parity, ry, stream)
                 : many<false>(params, items, nitems, parity, ry, stream);
}

}  // namespace dugks
