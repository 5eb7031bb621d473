// Launch wrappers and instantiations of the DG-SBP kernels for one
// arithmetic type (ESDG_SBP_REAL), degrees 1..5.
#include <type_traits>

#include "esdg_launch.hpp"
#include "esdg_sbp.cuh"

namespace esdg {

// The stage kernel (MODE 0 or 1) of degree N in FP64.
template <int N, int MODE>
static auto sbp_stage_kernel() {
    if constexpr (SbpSched<N>::DIAG)
        return &k_sbp_fx<N, MODE>;
    else
        return &k_sbp<N, double, MODE>;
}
template <int N>
static size_t sbp_stage_bytes(int warps) {
    return SbpSched<N>::DIAG ? sbp_fx_bytes<N>(warps) : SbpSmem<N, double>::bytes(warps);
}

template <int N, typename real>
cudaError_t sbp_geometry(int num_sms, LaunchGeom& lg) {
    lg.block = 256;
    const int warps = lg.block / 32;
    lg.smem = SbpSmem<N, real>::bytes(warps);
    cudaError_t err = cudaFuncSetAttribute(k_sbp<N, real, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lg.smem);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    if constexpr (std::is_same<real, double>::value) {
        const size_t smem = sbp_stage_bytes<N>(warps);
        err = cudaFuncSetAttribute(sbp_stage_kernel<N, 0>(), cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BLOCK_MAX);
        if (err != cudaSuccess) return err;
        err = cudaFuncSetAttribute(sbp_stage_kernel<N, 1>(), cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BLOCK_MAX);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sbp_stage_kernel<N, 1>(), lg.block, smem);
    } else {  // the FP32 path takes the records (MODE 2) only
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sbp<N, real, 2>, lg.block, lg.smem);
    }
    if (err != cudaSuccess) return err;
    if (per_sm < 1) per_sm = 1;
    lg.grid = per_sm * num_sms;
    lg.share = smem_share(per_sm);
    return cudaSuccess;
}

template <int N, typename real>
cudaError_t launch_sbp(const StageParams<real>& p, int mode, const LaunchGeom& lg, cudaStream_t s) {
    int block, grid;
    spread_elements(p.K, lg, block, grid);
    if (mode == 2)
        return launch_dependent(&k_sbp<N, real, 2>, grid, block, SbpSmem<N, real>::bytes(block / 32), s, p);
    if constexpr (std::is_same<real, double>::value) {
        void (*k)(StageParams<double>) = sbp_stage_kernel<N, 1>();
        if (mode == 0) k = sbp_stage_kernel<N, 0>();
        return launch_dependent(k, grid, block, spread_smem(lg, block, sbp_stage_bytes<N>(block / 32)), s, p);
    }
    return cudaErrorInvalidValue;
}

#define ESDG_SBP_INST(n)                                                                                  \
    template cudaError_t sbp_geometry<n, ESDG_SBP_REAL>(int, LaunchGeom&);                               \
    template cudaError_t launch_sbp<n, ESDG_SBP_REAL>(const StageParams<ESDG_SBP_REAL>&, int, const LaunchGeom&, \
                                                      cudaStream_t);
ESDG_SBP_INST(1)
ESDG_SBP_INST(2)
ESDG_SBP_INST(3)
ESDG_SBP_INST(4)
ESDG_SBP_INST(5)
#undef ESDG_SBP_INST

}  // namespace esdg
