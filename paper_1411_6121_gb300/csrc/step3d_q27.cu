// step3d_q27.cu -- the 3D throughput kernels instantiated for D3Q27 (the paper's 3D velocity set,
// Sec. 2.3), F32/BF16/F16 storage: the warp-specialised one (dugks_step3d_ws27.cuh, the default) and
// the non-specialised one (dugks_step3d.cuh, 32 x 8 columns per CTA; at 27 velocities its TMA
// stages do not fit beside the ring, so every plane is loaded directly and the tensor map is
// unused).
#include <string.h>

#include "dugks_internal.h"
#include "dugks_step3d.cuh"
#include "dugks_step3d_ws27.cuh"

namespace dugks {

template <class S, bool FORCE>
static cudaError_t launch27(const StepParams &p, cudaStream_t stream) {
    using K = Shape3<27, 8, S>;
    static int configured_dev = -1;
    static int sms = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_dev != dev) {
        cudaError_t e = cudaFuncSetAttribute(fused_step3d<27, S, 8, FORCE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)K::smem_bytes);
        if (e != cudaSuccess) return e;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        configured_dev = dev;
    }
    const int tiles_x = (p.nx + K::TXI - 1) / K::TXI;
    const int tiles_y = (p.ny + K::TYI - 1) / K::TYI;
    const int64_t tiles = (int64_t)tiles_x * tiles_y;
    const int zchunk = zchunk_for(tiles, p.nz, sms);  // one CTA per SM
    const int nchunks = (p.nz + zchunk - 1) / zchunk;
    static_assert(!K::TMA, "D3Q27 loads its planes directly");
    CUtensorMap unused;
    memset(&unused, 0, sizeof unused);
    fused_step3d<27, S, 8, FORCE><<<dim3(tiles_x, tiles_y, nchunks), dim3(32, 8), K::smem_bytes, stream>>>(p, unused,
                                                                                                          zchunk);
    return cudaGetLastError();
}

// Whether a wait of this translation unit's kernels gave up since the last call (and clears it).
int tma_wait_failures_q27() {
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_tma_wait_failed, sizeof v) != cudaSuccess) return -1;
    if (v) {
        const int zero = 0;
        cudaMemcpyToSymbol(g_tma_wait_failed, &zero, sizeof zero);
    }
    return v;
}

template <class S>
static cudaError_t launch_s(const StepParams &p, int ry, cudaStream_t stream) {
    const bool force = p.field != nullptr || p.g[0] != 0.0 || p.g[1] != 0.0 || p.g[2] != 0.0;
    if (ry == 0) return force ? ws27::launch_ws<27, S, true>(p, stream) : ws27::launch_ws<27, S, false>(p, stream);
    return force ? launch27<S, true>(p, stream) : launch27<S, false>(p, stream);
}

cudaError_t launch_step3d_q27(const StepParams &p, int store, int ry, cudaStream_t stream) {
    switch (store) {
        case 0: return launch_s<float>(p, ry, stream);
        case 1: return launch_s<__nv_bfloat16>(p, ry, stream);
        case 2: return launch_s<__half>(p, ry, stream);
    }
    return cudaErrorNotSupported;
}

}  // namespace dugks
