// step2d_q9_bf16.cu -- instantiations and launchers of the one-cell-per-thread D2Q9 kernel
// (dugks_step2d_cell.cuh) for BF16 storage.
#include <algorithm>

#include "dugks_internal.h"
#include "dugks_step2d_cell.cuh"

namespace dugks {

namespace {

using S = __nv_bfloat16;

template <int RY, bool FORCE>
cudaError_t launch_one(const StepParams &p, cudaStream_t stream) {
    using K = Shape2<RY, S>;
    static int configured_dev = -1, bps = 1, sms = 1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        cudaError_t e = cudaFuncSetAttribute(fused_step2d_cell<S, RY, FORCE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)K::smem_bytes);
        if (e != cudaSuccess) return e;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fused_step2d_cell<S, RY, FORCE>, 32 * RY, K::smem_bytes);
        bps = std::max(1, bps);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        configured_dev = dev;
    }
    const dim3 grid((p.nx + K::TXI - 1) / K::TXI, (p.ny + K::TYI - 1) / K::TYI);
    return launch_chained(fused_step2d_cell<S, RY, FORCE>, grid, dim3(32, RY), K::smem_bytes, stream, bps, sms, p);
}

template <int RY, bool FORCE>
cudaError_t launch_many(const StepParams *params, const int4 *items, int nitems, int parity, cudaStream_t stream) {
    using K = Shape2<RY, S>;
    static int configured_dev = -1, bps = 1, sms = 1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        cudaError_t e = cudaFuncSetAttribute(fused_step2d_cell_batch<S, RY, FORCE>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::smem_bytes);
        if (e != cudaSuccess) return e;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fused_step2d_cell_batch<S, RY, FORCE>, 32 * RY, K::smem_bytes);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        bps = std::max(1, bps);
        configured_dev = dev;
    }
    const int grid = std::min(nitems, bps * sms);  // persistent: the resident blocks, at most the items
    if (grid < 1) return cudaSuccess;
    return launch_chained(fused_step2d_cell_batch<S, RY, FORCE>, dim3(grid), dim3(32, RY), K::smem_bytes, stream, bps, sms,
                          params, items, nitems, parity);
}

template <bool FORCE>
cudaError_t one(const StepParams &p, int ry, cudaStream_t st) {
    if (ry == 4) return launch_one<4, FORCE>(p, st);
    if (ry == 8) return launch_one<8, FORCE>(p, st);
    if (ry == 16) return launch_one<16, FORCE>(p, st);
    return cudaErrorNotSupported;
}

template <bool FORCE>
cudaError_t many(const StepParams *params, const int4 *items, int nitems, int parity, int ry, cudaStream_t st) {
    if (ry == 4) return launch_many<4, FORCE>(params, items, nitems, parity, st);
    if (ry == 8) return launch_many<8, FORCE>(params, items, nitems, parity, st);
    if (ry == 16) return launch_many<16, FORCE>(params, items, nitems, parity, st);
    return cudaErrorNotSupported;
}

}  // namespace

cudaError_t launch_step2d_q9_bf16(const StepParams &p, int ry, cudaStream_t stream) {
    const bool force = p.field != nullptr || p.g[0] != 0.0 || p.g[1] != 0.0;
    if (ry == 0) ry = 8;
    return force ? one<true>(p, ry, stream) : one<false>(p, ry, stream);
}

cudaError_t launch_step2d_batch_bf16(const StepParams *params, const int4 *items, int nitems, int parity, int ry,
                                     bool force, cudaStream_t stream) {
    return force ? many<true>(params, items, nitems, parity, ry, stream)
                 : many<false>(params, items, nitems, parity, ry, stream);
}

}  // namespace dugks
