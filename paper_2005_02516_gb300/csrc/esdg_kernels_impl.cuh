// Definitions of the launch wrappers for one degree N (ESDG_N).
#include "esdg_launch.hpp"

namespace esdg {

// the stage kernel of degree N (right-hand side, MODE 0, or RK stage, 1) in blocks of 8 warps
template <int N, typename real, int MODE>
static auto stage_kernel() {
    return &k_stage<N, real, MODE, stage_min_blocks<N>(), 8>;
}

template <int N, typename real>
cudaError_t stage_geometry(int num_sms, LaunchGeom& lg) {
    lg.block = 256;
    lg.smem = Smem<N, real>::bytes(lg.block / 32);
    cudaError_t err;
    err = cudaFuncSetAttribute(stage_kernel<N, real, 0>(), cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BLOCK_MAX);
    if (err != cudaSuccess) return err;
    if constexpr (stage_min_blocks<N>() == 3) {
        err = cudaFuncSetAttribute(k_stage<N, real, 0, 1, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BLOCK_MAX);
        if (err != cudaSuccess) return err;
    }
    auto* k1 = stage_kernel<N, real, 1>();
    err = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BLOCK_MAX);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k1, lg.block, lg.smem);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) per_sm = 1;
    lg.grid = per_sm * num_sms;
    lg.share = smem_share(per_sm);
    if constexpr (stage_wide_warps<N>() > 0) {
        constexpr int W = stage_wide_warps<N>();
        err = cudaFuncSetAttribute(k_stage<N, real, 0, 2, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BLOCK_MAX);
        if (err != cudaSuccess) return err;
        auto* kw = &k_stage<N, real, 1, 2, W>;
        err = cudaFuncSetAttribute(kw, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BLOCK_MAX);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kw, 32 * W, Smem<N, real>::bytes(W));
        if (err != cudaSuccess) return err;
        lg.wide_grid = per_sm * num_sms;
    }
    return cudaSuccess;
}

template <int N, typename real>
cudaError_t project_geometry(int num_sms, LaunchGeom& lg) {
    lg.block = 256;
    lg.smem = Smem<N, real>::bytes(lg.block / 32);
    cudaError_t err =
        cudaFuncSetAttribute(k_project<N, real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lg.smem);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_project<N, real>, lg.block, lg.smem);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) per_sm = 1;
    lg.grid = per_sm * num_sms;
    return cudaSuccess;
}

template <int N, typename real>
cudaError_t launch_project(const StageParams<real>& p, const LaunchGeom& lg, cudaStream_t s) {
    int block, grid;
    spread_elements(p.K, lg, block, grid);
    return launch_dependent(&k_project<N, real>, grid, block, Smem<N, real>::bytes(block / 32), s, p);
}

template <int N, typename real>
cudaError_t launch_stage(const StageParams<real>& p, int mode, const LaunchGeom& lg, cudaStream_t s) {
    int block, grid;
    spread_elements(p.K, lg, block, grid);
    if constexpr (stage_wide_warps<N>() > 0) {
        constexpr int W = stage_wide_warps<N>();
        if (p.K > lg.grid * (lg.block / 32) && lg.wide_grid > 0) {
            void (*kw)(StageParams<real>) = &k_stage<N, real, 1, 2, W>;
            if (mode == 0) kw = &k_stage<N, real, 0, 2, W>;
            return launch_dependent(kw, lg.wide_grid, 32 * W, Smem<N, real>::bytes(W), s, p);
        }
    }
    auto* k = mode == 0 ? stage_kernel<N, real, 0>() : stage_kernel<N, real, 1>();
    if constexpr (stage_min_blocks<N>() == 3)
        if (mode == 0 && block <= 32 * FEW_WARPS) k = &k_stage<N, real, 0, 1, 8>;
    return launch_dependent(k, grid, block, spread_smem(lg, block, Smem<N, real>::bytes(block / 32)), s, p);
}

template <int N>
cudaError_t stage2_geometry(int num_sms, LaunchGeom& lg) {
    lg.block = 32 * C2<N>::WARPS;
    lg.smem = C2<N>::bytes();
    cudaError_t err;
    err = cudaFuncSetAttribute(k_stage2<N, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lg.smem);
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(k_stage2<N, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lg.smem);
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(k_stage2<N, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lg.smem);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stage2<N, 1>, lg.block, lg.smem);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    lg.grid = per_sm * num_sms;
    return cudaSuccess;
}

template <int N>
cudaError_t launch_stage2(const StageParams<float>& p, const float* ops2, int Kpad, int mode, const LaunchGeom& lg,
                          cudaStream_t s) {
    typedef C2<N> C;
    const int batches = Kpad / C::EPW;
    auto* k = mode == 0 ? &k_stage2<N, 0> : mode == 1 ? &k_stage2<N, 1> : &k_stage2<N, 2>;
    if constexpr (C::TC) {
        // (tensor memory is allocated per block: no two stages' blocks on one SM)
        const int need = (batches + C::WARPS - 1) / C::WARPS;
        k<<<need < lg.grid ? need : lg.grid, lg.block, lg.smem, s>>>(p, ops2, Kpad);
        return cudaGetLastError();
    }
    int warps, grid;
    spread_batches(batches, lg.grid, C::WARPS, warps, grid);
    return launch_dependent(k, grid, 32 * warps, C::bytes(warps), s, p, ops2, Kpad);
}

template <int N>
cudaError_t launch_entropy(int K, double g, const double* u, const double* rhs, const double* Vq, const double* wJq,
                           const double* bq, int bq_stride, double* partial, int nparts, double* out, cudaStream_t s) {
    k_entropy<N><<<nparts, 256, 0, s>>>(K, g, u, rhs, Vq, wJq, bq, bq_stride, partial);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    k_entropy_finalize<<<1, FINALIZE_THREADS, 0, s>>>(nparts, partial, out);
    return cudaGetLastError();
}

#ifndef ESDG_FP64_ONLY  // the compact forms have the FP64 kernels only
template cudaError_t stage2_geometry<ESDG_N>(int, LaunchGeom&);
template cudaError_t launch_stage2<ESDG_N>(const StageParams<float>&, const float*, int, int, const LaunchGeom&,
                                          cudaStream_t);
#endif
#ifndef ESDG_STAGE2_ONLY  // the tensor-core forms (ESDG_N >= 32) have the FP32 stage kernel only
template cudaError_t stage_geometry<ESDG_N, double>(int, LaunchGeom&);
template cudaError_t project_geometry<ESDG_N, double>(int, LaunchGeom&);
template cudaError_t launch_project<ESDG_N, double>(const StageParams<double>&, const LaunchGeom&, cudaStream_t);
template cudaError_t launch_stage<ESDG_N, double>(const StageParams<double>&, int, const LaunchGeom&, cudaStream_t);
#ifndef ESDG_FP64_ONLY
template cudaError_t launch_entropy<ESDG_N>(int, double, const double*, const double*, const double*, const double*,
                                            const double*, int, double*, int, double*, cudaStream_t);
#endif
#endif

}  // namespace esdg
