// dugks_internal.h -- host-side declarations shared by the translation units of libdugks.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dugks_device.cuh"

namespace dugks {

// Launches a kernel whose blocks may be set up while the work ahead of it in the stream still runs
// (programmatic stream serialization): the kernel begins with chain_wait(), so it orders after
// that work all the same, and the gap between two steps of a sequence loses the launch itself
// (0.4 of 3.8 us per step of an 8 x 32 channel, 0.5 of 30.4 of a 1024^2 cavity). resident: blocks per SM,
// sms: SMs. Where the blocks of two steps do not fit the GPU together but an SM holds more than a step gives
// it, the waiting blocks would fill the SMs unevenly (two blocks here, three there, and the step takes as long
// as three): there the launch is an ordinary one (2D meshes of 1.5 to 2 blocks per SM where three fit: 5 to
// 17% a step; everywhere else chaining gains 1 to 12%).
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int resident,
                           int sms, A... args) {
    const int64_t blocks = (int64_t)grid.x * grid.y * grid.z;
    const bool uneven = 2 * blocks > (int64_t)resident * sms && blocks <= (int64_t)(resident - 1) * sms;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = uneven ? 0 : 1;
    return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

// Launch one fused step (fused_step<Q, S, TX, TY>) on `stream`. store: DUGKS_STORE_*.
// Returns cudaSuccess or the launch error; cudaErrorNotSupported for a tile that was not
// instantiated.
cudaError_t launch_step_q9(const StepParams &p, int store, int tx, int ty, cudaStream_t stream);
cudaError_t launch_step_q19(const StepParams &p, int store, int tx, int ty, cudaStream_t stream);
cudaError_t launch_step_q27(const StepParams &p, int store, int tx, int ty, cudaStream_t stream);
// Throughput kernels for D3Q19 and D3Q27 with F32/BF16/F16 storage: ry 0 the warp-specialised one
// (dugks_step3d_ws.cuh, dugks_step3d_ws27.cuh), else the non-specialised one (dugks_step3d.cuh) with ry CTA rows (D3Q27: 8).
cudaError_t launch_step3d_q19(const StepParams &p, int store, int ry, cudaStream_t stream);
cudaError_t launch_step3d_q27(const StepParams &p, int store, int ry, cudaStream_t stream);
// Throughput kernel for D2Q9 with F32/BF16/F16 storage (dugks_step2d.cuh; BF16, and small F32 and F16
// meshes with ry 0: dugks_step2d_cell.cuh): ry = block rows, tiles of step2d_tile_columns(store) columns x
// (ry - 2) rows; 0: kernel and rows chosen by the mesh (a kernel's results do not depend on the rows). The
// batch form walks a work list of (instance, x0, y0) tile origins over params[2 i + parity], a block per item
// (BF16: persistent blocks); force: 0 no instance has an acceleration, 1 all have, 2 some.
int step2d_tile_columns(int store);
cudaError_t launch_step2d_q9(const StepParams &p, int store, int ry, cudaStream_t stream);
cudaError_t launch_step2d_batch(const StepParams *params, const int4 *items, int nitems, int parity, int store,
                                int ry, int force, cudaStream_t stream);
// One cell per thread (dugks_step2d_cell.cuh): BF16 with 4, 8 or 16 rows, F32 and F16 with 8.
// step2d_cell_warps: the warps that a step of that kernel (F32, F16) gives the busiest SM, 0 if its blocks are
// not all resident at once.
cudaError_t launch_step2d_cell(const StepParams &p, int store, int ry, cudaStream_t stream);
int step2d_cell_warps(const StepParams &p, int store, bool force);
cudaError_t launch_step2d_batch_bf16(const StepParams *params, const int4 *items, int nitems, int parity, int ry,
                                     bool force, cudaStream_t stream);

// D2Q9 kernel with few operations per cell (dugks_step2d_lean.cuh): F64 storage, and non-uniform meshes
// with F32 or F64 storage; incompressible model.
cudaError_t launch_step2d_lean(const StepParams &p, int store, cudaStream_t stream);

// Whether a TMA wait of the 3D throughput kernel gave up since the last call (the kernel then
// skipped its step); clears the flag. 1: yes, 0: no, -1: the flag could not be read.
int tma_wait_failures();
int tma_wait_failures_q27();

// Auxiliary kernels (aux.cu).
cudaError_t launch_init(int q, int store, const StepParams &p, const double *pres, const double *vel, double rt,
                        cudaStream_t stream);
cudaError_t launch_moments(int q, int store, const StepParams &p, double t, double rt, float *out,
                           cudaStream_t stream);
// FP64 residual and totals: per-block partial sums into `partials` ([nblocks][8] doubles),
// then a fixed-order final sum into `out` (8 doubles on the device).
// uprev: [dim][ncell] u of the call before, overwritten.
cudaError_t launch_residual(int q, int store, const StepParams &p, double t, double rt, double *uprev,
                            int have_prev, double *partials, int nblocks, double *out, cudaStream_t stream);
int residual_blocks(int64_t ncell);
// The time factors of the n steps from the device step counter on into out[0 .. n-1].
cudaError_t launch_time_factors(const long long *ctr, int n, double omega, double dt, double inv_c, TimeFactors *out,
                                cudaStream_t stream);
cudaError_t launch_advance(long long *ctr, long long n, cudaStream_t stream);

// Sets the message that dugks_last_error(NULL) returns in this thread (api.cu).
void set_null_handle_error(const char *msg);

}  // namespace dugks
