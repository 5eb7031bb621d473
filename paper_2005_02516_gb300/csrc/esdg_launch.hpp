// Host-side launch wrappers, one explicit instantiation per degree N (the
// esdg_kernels_nK.cu translation units compile in parallel).
#pragma once

#include <cuda_runtime.h>

#include "esdg_kernels.cuh"
#include "esdg_ensemble.cuh"

namespace esdg {

// Launch geometry of the persistent warp-per-element kernels (k_stage for the
// FP64 right-hand side, k_project for both precisions): CTAs of 8 warps, as
// many CTAs per SM as fit.
struct LaunchGeom {
    int block = 256;
    int grid = 0;
    size_t smem = 0;
    int wide_grid = 0;  // blocks of stage_wide_warps warps that fill the chip
    size_t share = 0;  // shared memory of a block at which grid blocks fill the chip and no more fit
};

// The largest dynamic shared memory of a block of which per_sm fit on an SM (228
// KB, 1 KB of each block's reserved).
constexpr int SMEM_BLOCK_MAX = 232448;
inline size_t smem_share(int per_sm) { return (size_t(SMEM_BLOCK_MAX + 1024) / size_t(per_sm) - 1024) & ~size_t(1023); }

// Launch with programmatic stream serialization (see pdl_wait): the kernel
// starts its prologue while the one before it on the stream drains.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s,
                                    Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(grid));
    cfg.blockDim = dim3(unsigned(block));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// Warps a block and blocks of a batched kernel (one block per SM, one batch a
// warp at a time): the rounds that `most` warps on every SM need, with the
// batches then spread evenly over the SMs and the rounds.  A problem of fewer
// batches than the chip has warps thus puts few warps on every SM instead of
// `most` on a few (the stage is bound by the SM's issue slots and latencies):
// with dependent launches, N = 4 at K = 512 (128 batches) 24.1 -> 9.3 us per
// stage, N = 3 at K = 8192 24.4 -> 14.1 us, K = 31714 in 3 rounds of 18 warps
// instead of 2 of 24 and a remainder 45 -> 36 us.
inline void spread_batches(int batches, int sms, int most, int& warps, int& grid) {
    if (batches < 1) batches = 1;
    const int rounds = (batches + sms * most - 1) / (sms * most);
    warps = (batches + sms * rounds - 1) / (sms * rounds);
    grid = (batches + warps - 1) / warps;
    if (grid > sms) grid = sms;
}

// The same for the warp-per-element kernels (lg.grid blocks of lg.block threads
// fill the chip): problems of at most lg.grid's warps take the warps a block that
// spread the elements over lg.grid blocks (element_of), so that every SM has its
// share; full blocks in part of the places left SMs with half the warps of
// others.  Per stage, FP64: K = 2048, N = 4 33.7 -> 25.4 us, N = 3 31.4 -> 24.2,
// DG-SBP N = 5 141 -> 93; K = 1458, weight-adjusted N = 4 68.5 -> 47.5.  At least 4
// warps a block, because the other warps of a block that holds one element still
// stage the operators (N = 2, K = 128: 27.5 -> 15 us per stage with dependent
// launches).
inline void spread_elements(int K, const LaunchGeom& lg, int& block, int& grid) {
    const int wpb = lg.block / 32, w = (K + lg.grid - 1) / lg.grid;
    block = w >= wpb ? lg.block : 32 * (w > 4 ? w : 4);
    grid = K < lg.grid ? K : lg.grid;
}
// Their shared memory: blocks of more than half the warps take lg.share bytes, as
// more of them would fit on an SM than lg.grid counts on and leave other SMs
// without; smaller ones do not, so that the next stage's blocks fit beside them
// (DG-SBP N = 3, K = 1458, blocks of 4 warps: 16.4 us per stage, 17.5 with the
// share).
inline size_t spread_smem(const LaunchGeom& lg, int block, size_t bytes) {
    return block < lg.block && block > lg.block / 2 && bytes < lg.share ? lg.share : bytes;
}

template <int N, typename real>
cudaError_t stage_geometry(int num_sms, LaunchGeom& lg);
template <int N, typename real>
cudaError_t project_geometry(int num_sms, LaunchGeom& lg);
template <int N, typename real>
cudaError_t launch_project(const StageParams<real>& p, const LaunchGeom& lg, cudaStream_t s);
template <int N, typename real>
cudaError_t launch_stage(const StageParams<real>& p, int mode, const LaunchGeom& lg, cudaStream_t s);
// FP32 batched stage kernel (esdg_stage2.cuh): one block per SM (spread_batches).
template <int N>
cudaError_t stage2_geometry(int num_sms, LaunchGeom& lg);
template <int N>
cudaError_t launch_stage2(const StageParams<float>& p, const float* ops2, int Kpad, int mode, const LaunchGeom& lg,
                          cudaStream_t s);
template <int N>
cudaError_t launch_entropy(int K, double g, const double* u, const double* rhs, const double* Vq, const double* wJq,
                           const double* bq, int bq_stride, double* partial, int nparts, double* out, cudaStream_t s);
// DG-SBP kernels (esdg_sbp.cuh), degree N = 1..5, FP64 and FP32.
template <int N, typename real>
cudaError_t sbp_geometry(int num_sms, LaunchGeom& lg);
template <int N, typename real>
cudaError_t launch_sbp(const StageParams<real>& p, int mode, const LaunchGeom& lg, cudaStream_t s);
// FP32 batched DG-SBP stage kernel (esdg_sbp2.cuh), modes 0 and 1.
template <int N>
cudaError_t sbp2_geometry(int num_sms, LaunchGeom& lg);
template <int N>
cudaError_t launch_sbp2(const StageParams<float>& p, const float* ops2, int Kpad, int mode, const LaunchGeom& lg,
                        cudaStream_t s);
int sbp2_ops_floats(int N);
cudaError_t launch_entropy_nodal(int K, int Nq, double g, const double* u, const double* rhs, const double* wJq,
                                 const double* bq, double* partial, int nparts, double* out, cudaStream_t s);
// FP64 L2 error against given values at the volume points (esdg_diag.cu):
// Vq [Nq][Np] for a modal state, NULL for a nodal one (Np = Nq).
cudaError_t launch_l2_error(int K, int Nq, int Np, const double* u, const double* Vq, const double* wJq,
                            const double* exact, double* partial, int nparts, double* out, cudaStream_t s);

}  // namespace esdg
