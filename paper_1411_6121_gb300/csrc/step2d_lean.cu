// step2d_lean.cu -- instantiations and launcher of the D2Q9 kernel with few operations
// (dugks_step2d_lean.cuh): FP64 storage, and non-uniform meshes in F32 and F64.
#include "dugks_internal.h"
#include "dugks_step2d_lean.cuh"

namespace dugks {

namespace {

// Block rows: the ones that leave the busiest SM the least arithmetic, a row's step 1 (84 operations
// per cell) on every row and the rest (290) on the inner ones. 128 x 128 cells on 152 SMs: 7 rows
// (130 blocks, one per SM) instead of 8 (110 blocks).
int block_rows(int64_t nx, int64_t ny, int sms) {
    const int64_t strips = (nx + lean::TXI - 1) / lean::TXI;
    int best = lean::MAX_RY;
    double least = 1e300;
    for (int ry = 3; ry <= lean::MAX_RY; ry++) {
        const int64_t blocks = strips * ((ny + ry - 3) / (ry - 2));
        const double cost = (double)((blocks + sms - 1) / sms) * (84.0 * ry + 290.0 * (ry - 2));
        if (cost < least) {
            least = cost;
            best = ry;
        }
    }
    return best;
}

template <class S, bool NU, bool FORCE>
cudaError_t launch(const StepParams &p, cudaStream_t stream) {
    using T = typename Arith<S>::T;
    static int configured_dev = -1, sms = 1, blocks[lean::MAX_RY + 1];
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        cudaError_t e = cudaFuncSetAttribute(lean::fused_step2d_lean<S, NU, FORCE>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)lean::smem_bytes<T, FORCE>(lean::MAX_RY));
        if (e != cudaSuccess) return e;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        for (int ry = 3; ry <= lean::MAX_RY; ry++) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks[ry], lean::fused_step2d_lean<S, NU, FORCE>, 32 * ry,
                                                          lean::smem_bytes<T, FORCE>(ry));
            blocks[ry] = blocks[ry] < 1 ? 1 : blocks[ry];
        }
        configured_dev = dev;
    }
    const int ry = block_rows(p.nx, p.ny, sms);
    // all tiles along x: a grid's y extent (65,535) would end at 393,210 rows of cells
    const dim3 grid((unsigned)((int64_t)((p.nx + lean::TXI - 1) / lean::TXI) * ((p.ny + ry - 3) / (ry - 2))));
    return launch_chained(lean::fused_step2d_lean<S, NU, FORCE>, grid, dim3(32, ry), lean::smem_bytes<T, FORCE>(ry), stream,
                          blocks[ry], sms, p);
}

template <class S, bool NU>
cudaError_t pick(const StepParams &p, cudaStream_t st) {
    return p.field != nullptr || p.g[0] != 0.0 || p.g[1] != 0.0 ? launch<S, NU, true>(p, st) : launch<S, NU, false>(p, st);
}

}  // namespace

cudaError_t launch_step2d_lean(const StepParams &p, int store, cudaStream_t stream) {
    if (p.metric[0]) {
        if (store == 0) return pick<float, true>(p, stream);
        if (store == 3) return pick<double, true>(p, stream);
    } else if (store == 3) {
        return pick<double, false>(p, stream);
    }
    return cudaErrorNotSupported;
}

}  // namespace dugks
