// The batched persistent kernel up to 64 columns (sm_103a; factor_wide.cu has the wider
// builds) and the sizes of the factorization jobs. The jobs themselves are in batch_job.cuh
// (FP64 items and tree nodes in 64-bit fixed point, factor_fixed.cuh; FP32 chains of mixed
// items, factor_job.cuh); the one-problem launches are in factor_fixed.cu.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "batch_job.cuh"
#include "tsqr_internal.h"
#include "warp_reduce.cuh"

namespace tsqr {
namespace {

// ----------------------------------------------------------- batched persistent kernel

template <int CMAX, bool CHAINS>
__global__ void __launch_bounds__(kThreads, 2) k_factor_batch(const BatchParams bp) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_job, s_go;
  batch_loop<CMAX, CHAINS, false>(bp, smraw, s_job, s_go, [](const FactorParamsT<float> &, const JobDesc &, int) {});
}

__device__ int32_t g_error_word;

}  // namespace

bool cluster_takes(int n, int nc, size_t optin_per_block) {
  const size_t ncp = (size_t)((nc + 7) & ~7);
  return sizeof(double) * ((size_t)nc * n + ncp + (size_t)n * ncp) <= optin_per_block;
}

cudaError_t device_error_word(int32_t **ptr) {
  return cudaGetSymbolAddress(reinterpret_cast<void **>(ptr), g_error_word);
}

size_t factor_smem_bytes(int nc, int ldt, size_t elem) {
  const size_t ncp = (size_t)((nc + 7) & ~7);
  // FP32 register-tile chains: the one-barrier job's two tail buffers and scalar sets, or
  // the compact-WY job's pivot column, Gram row and pivot rows; then the chain's R (the
  // compact-WY job's panel buffers come on top, f32wy_smem_extra_bytes)
  if (elem == sizeof(float))
    return sizeof(float) * (std::max((size_t)2 * kF32TileRows + 8, (size_t)kF32TileRows + 3 * ncp) +
                            (size_t)nc * (ncp + 1));
  return elem * ((size_t)nc * (size_t)ldt + 2 * ncp);
}

int factor_max_rows(int nc, int ctas_per_sm, size_t smem_per_sm, size_t reserved_per_block,
                    size_t optin_per_block, size_t elem) {
  if (ctas_per_sm < 1) return 0;
  size_t per_cta = smem_per_sm / (size_t)ctas_per_sm;
  if (per_cta <= reserved_per_block) return 0;
  per_cta -= reserved_per_block;
  if (per_cta > optin_per_block) per_cta = optin_per_block;
  const size_t extra = factor_smem_bytes(nc, 0, elem);
  if (per_cta <= extra) return 0;
  int rows = (int)((per_cta - extra) / (elem * (size_t)nc));
  return rows >= 16 ? (rows & ~15) : (rows & ~7);  // multiples of 16 keep the half-warps full
}

bool factor_tile_choice(int n, int nc, int leaf_h, size_t smem_per_sm, size_t reserved_per_block,
                        size_t optin_per_block, int max_cps, int &tile_h, int &cps) {
  for (int c = max_cps < 3 ? max_cps : 3; c >= 1; --c) {
    int rows = factor_max_rows(nc, c, smem_per_sm, reserved_per_block, optin_per_block);
    if (rows > 512) rows = 512;  // the apply kernels stage at most 512 rows per tile
    // the one-problem launches factor in fixed point, on register tiles
    if (max_cps >= 3 && factor_fixed_max_rows(nc) > 0) rows = std::min(rows, factor_fixed_max_rows(nc));
    // a third CTA per SM pays only while its tile still holds two triangles' worth of rows
    const int need = (c >= 3) ? 2 * n : n;
    if (rows >= need && rows >= 8) {
      tile_h = rows < (leaf_h > n ? leaf_h : n) ? rows : (leaf_h > n ? leaf_h : n);
      cps = c;
      return true;
    }
  }
  return false;
}

cudaError_t launch_factor_batch(const BatchParams &p, int cmax, int grid, size_t smem_bytes, cudaStream_t s,
                                bool fp64_items, bool wy) {
  if (cmax > 4 || wy) return launch_factor_batch_wide(p, grid, smem_bytes, s, fp64_items, wy);
  if (cmax <= 2) {
    if (!fp64_items) return launch_batch_kernel(k_factor_batch<2, false>, p, grid, smem_bytes, s);
    return launch_batch_kernel(k_factor_batch<2, true>, p, grid, smem_bytes, s);
  }
  if (!fp64_items) return launch_batch_kernel(k_factor_batch<4, false>, p, grid, smem_bytes, s);
  return launch_batch_kernel(k_factor_batch<4, true>, p, grid, smem_bytes, s);
}

size_t batch_job_smem(int n, int nc, bool node) {
  const size_t fx = nc <= 16   ? fx_smem_bytes(n, nc, 1, 16)
                    : nc <= 32 ? fx_smem_bytes(n, nc, 2, 18)
                    : nc <= 64 ? fx_smem_bytes(n, nc, 4, 18)
                    : nc <= 96 ? fx_smem_bytes(n, nc, 4, 12)
                               : fx_smem_bytes(n, nc, 8, nc <= 128 ? 18 : 14);
  return std::max(fx, factor_smem_bytes(nc, batch_job_ldt(n, nc, node)));
}
int batch_job_ldt(int n, int nc, bool node) {
  const int rows = batch_job_rows(nc), pieces = (n + rows - 1) / rows;  // as split_tree_tiles
  return node ? (n + pieces - 1) / pieces : rows;
}

int batch_job_rows(int nc) {
  return nc <= 64 ? factor_fixed_max_rows(nc) : nc <= 96 ? 96 : nc <= 128 ? 72 : 56;
}

}  // namespace tsqr
