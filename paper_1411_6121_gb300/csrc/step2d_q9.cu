// step2d_q9.cu -- instantiations and launchers of the D2Q9 throughput kernel
// (dugks_step2d.cuh): one instance on a grid of tiles, or a batch on a list of them.
#include <algorithm>

#include "dugks_internal.h"
#include "dugks_step2d.cuh"

namespace dugks {

namespace {

// Resident blocks per SM of a kernel at every number of block rows, for one device.
struct Residency {
    int dev = -1, sms = 1, blocks[m2::MAX_RY + 1] = {};
};

// FORCE: as the batch kernel's; the single kernel has 0 and 1.
template <class S, int FORCE, bool BATCH>
cudaError_t configure(const Residency **out) {
    static Residency r;
    int dev = 0;
    cudaGetDevice(&dev);
    if (r.dev != dev) {
        const void *fn;
        if constexpr (BATCH) fn = (const void *)fused_step2d_batch<S, FORCE>;
        else fn = (const void *)fused_step2d<S, FORCE != 0>;
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)m2::smem_bytes<FORCE != 0>(m2::MAX_RY));
        if (e != cudaSuccess) return e;
        for (int ry = 3; ry <= m2::MAX_RY; ry++) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.blocks[ry], fn, 32 * ry, m2::smem_bytes<FORCE != 0>(ry));
            r.blocks[ry] = std::max(1, r.blocks[ry]);
        }
        cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev);
        r.dev = dev;
    }
    *out = &r;
    return cudaSuccess;
}

// Block rows of an nx x ny mesh: the ones that leave the busiest SM the fewest warps to run,
// counted against 24 resident ones where they come in waves (10 and 16 rows fit 20 and 16 per
// SM); the smaller block on a tie. A block updates ry - 2 of its rows, so large meshes take 12 rows
// and small ones, where a step is the latency of one block, few. us per step with 4 / 6 / 8 / 12
// rows: 128 x 64 channel 3.38 / 3.72 / 4.04 / 5.01, 512 x 256 channel 7.64 / 6.70 / 7.05 / 7.04, 2048^2
// cavity 124 / 106 / 103 / 102.
// on_sm: the warps of the busiest SM.
int block_rows(int64_t nx, int64_t ny, const Residency &r, int64_t *on_sm) {
    const int64_t strips = (nx + m2::TXI - 1) / m2::TXI;
    const int cand[] = {3, 4, 6, 8, 12};
    int best = 8;
    double least = 1e300;
    for (int ry : cand) {
        const int64_t blocks = strips * ((ny + ry - 3) / (ry - 2));
        const int64_t mine = (blocks + r.sms - 1) / r.sms * ry;
        const double warps = (double)mine;
        const int cap = std::min(24, r.blocks[ry] * ry);
        const double cost = warps > cap ? warps * 24.0 / cap : warps;
        if (cost < least) {
            least = cost;
            best = ry;
            *on_sm = mine;
        }
    }
    return best;
}

template <class S, bool FORCE>
cudaError_t launch_one(const StepParams &p, int ry, cudaStream_t stream) {
    const Residency *r;
    cudaError_t e = configure<S, FORCE, false>(&r);
    if (e != cudaSuccess) return e;
    if (ry == 0) {
        // Where a step of the one-cell kernel (8 rows of 30 columns) is all resident at once, it is latency that
        // counts and that kernel has the shorter way through a block: it is taken where the pairs would still
        // put two thirds (F16, whose rounding is a longer tail for two cells: half) of its warps on the busiest SM.
        // us per step, F32 cavity / channel, one cell / pairs: 9 x 724 (8 / 8 warps) 3.9 / 4.6, 3.7 / 4.2; 78 x 883
        // (24 / 16) 5.8 / 5.8, 4.9 / 6.2; 119 x 32 (8 / 3) 3.8 / 3.7, 3.7 / 3.3; 1140 x 49 (24 / 12) 5.4 / 4.4, 5.0 / 4.4.
        int64_t pairs = 0;
        ry = block_rows(p.nx, p.ny, *r, &pairs);
        const int store = sizeof(S) == 4 ? 0 : 2, cells = step2d_cell_warps(p, store, FORCE);
        if (cells > 0 && (sizeof(S) == 4 ? 3 * pairs >= 2 * cells : 2 * pairs >= cells))
            return launch_step2d_cell(p, store, 8, stream);
    }
    const dim3 grid((p.nx + m2::TXI - 1) / m2::TXI, (p.ny + ry - 3) / (ry - 2));
    return launch_chained(fused_step2d<S, FORCE>, grid, dim3(32, ry), m2::smem_bytes<FORCE>(ry), stream, r->blocks[ry],
                          r->sms, p);
}

template <class S, int FORCE>
cudaError_t launch_many(const StepParams *params, const int4 *items, int nitems, int parity, int ry,
                        cudaStream_t stream) {
    const Residency *r;
    cudaError_t e = configure<S, FORCE, true>(&r);
    if (e != cudaSuccess) return e;
    if (nitems < 1) return cudaSuccess;
    return launch_chained(fused_step2d_batch<S, FORCE>, dim3(nitems), dim3(32, ry), m2::smem_bytes<FORCE != 0>(ry), stream,
                          r->blocks[ry], r->sms, params, items, parity);
}

template <class S>
cudaError_t many(const StepParams *params, const int4 *items, int nitems, int parity, int ry, int force, cudaStream_t st) {
    if (force == 0) return launch_many<S, 0>(params, items, nitems, parity, ry, st);
    if (force == 1) return launch_many<S, 1>(params, items, nitems, parity, ry, st);
    return launch_many<S, 2>(params, items, nitems, parity, ry, st);
}

}  // namespace

int step2d_tile_columns(int store) { return store == 1 ? 30 : m2::TXI; }

cudaError_t launch_step2d_q9(const StepParams &p, int store, int ry, cudaStream_t stream) {
    const bool force = p.field != nullptr || p.g[0] != 0.0 || p.g[1] != 0.0;
    switch (store) {
        case 0: return force ? launch_one<float, true>(p, ry, stream) : launch_one<float, false>(p, ry, stream);
        case 1: return launch_step2d_cell(p, store, ry == 0 ? 8 : ry, stream);
        case 2: return force ? launch_one<__half, true>(p, ry, stream) : launch_one<__half, false>(p, ry, stream);
    }
    return cudaErrorNotSupported;
}

cudaError_t launch_step2d_batch(const StepParams *params, const int4 *items, int nitems, int parity, int store,
                                int ry, int force, cudaStream_t stream) {
    switch (store) {
        case 0: return many<float>(params, items, nitems, parity, ry, force, stream);
        case 1: return launch_step2d_batch_bf16(params, items, nitems, parity, ry, force != 0, stream);
        case 2: return many<__half>(params, items, nitems, parity, ry, force, stream);
    }
    return cudaErrorNotSupported;
}

}  // namespace dugks
