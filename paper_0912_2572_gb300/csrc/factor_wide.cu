// The batched persistent kernel for items of more than 64 columns, and with compact-WY FP32
// chains: a translation unit of its own, since each holds every job build (compile time).
#include "batch_job.cuh"
#include "factor_wy.cuh"

namespace tsqr {
namespace {

template <bool CHAINS>
__global__ void __launch_bounds__(kThreads, 2) k_factor_batch_wide(const BatchParams bp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_job, s_go;
  batch_loop<16, CHAINS, false>(bp, smraw, s_job, s_go, [](const FactorParamsT<float> &, const JobDesc &, int) {});
}

// The build that can run mixed chains by compact-WY panels; the others keep their register
// budget for the other job kinds.
__global__ void __launch_bounds__(kThreads, 2) k_factor_batch_wy(const BatchParams bp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_job, s_go;
  batch_loop<16, true, true>(bp, smraw, s_job, s_go, [&](const FactorParamsT<float> &fp, const JobDesc &jd, int n) {
    switch (n <= 32 ? 2 : (n <= 64 ? 4 : 8)) {
      case 2: run_job_f32wy<2>(fp, jd, smraw); break;
      case 4: run_job_f32wy<4>(fp, jd, smraw); break;
      default: run_job_f32wy<8>(fp, jd, smraw); break;
    }
  });
}

}  // namespace

cudaError_t launch_factor_batch_wide(const BatchParams &p, int grid, size_t smem_bytes, cudaStream_t s,
                                     bool fp64_items, bool wy) {
  if (wy) return launch_batch_kernel(k_factor_batch_wy, p, grid, smem_bytes, s);
  if (!fp64_items) return launch_batch_kernel(k_factor_batch_wide<false>, p, grid, smem_bytes, s);
  return launch_batch_kernel(k_factor_batch_wide<true>, p, grid, smem_bytes, s);
}

size_t f32wy_smem_extra_bytes() {
  return sizeof(float) * ((size_t)kWyPanel * kWyLd + (size_t)kF32TileRows * kWyLdT + (size_t)kWyChunk * kWyLd +
                          2 * (size_t)kWyPanel * kWyChunk + (size_t)kWyChunk * kWyLdT +
                          2 * (size_t)kWyPanel * (kWyPanel + 1) + kWyPanel);
}

}  // namespace tsqr
