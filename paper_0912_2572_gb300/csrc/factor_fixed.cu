// The one-problem factorization launches in 64-bit fixed point
// (factor_fixed.cuh): the chain launch and the tree levels.
#include "cluster_sync.cuh"
#include "factor_fixed.cuh"

namespace tsqr {
namespace {

// A job, or what is left of it once a tile holds an entry the fixed-point form cannot take or
// is light beside its columns, which goes through the FP64 job (written for eight warps).
template <int CPL, int LC, int RPL, int NW>
__device__ __forceinline__ void run_any(const FactorParamsT<double> &p, JobDesc job, unsigned char *smraw) {
  const int done = run_job_fx<CPL, LC, RPL, NW>(p, job, smraw);
  if (done < job.tile_count) {
    job.tile_begin += done;
    job.tile_count -= done;
    if (NW == 8 || threadIdx.x < kThreads)
      run_job<(NW > 8 ? 8 : LC == 1 ? 1 : LC == 2 ? 2 : 4)>(p, job, smraw, NW > 8);
  }
}

// At most 36 entries (72 registers) per thread, so 16 warps fit an SM at 128 registers: two
// CTAs of eight (up to 64 columns), or one of sixteen.
template <int CPL, int LC, int RPL, int NW>
__global__ void __launch_bounds__(32 * NW, 16 / NW) k_factor_fx(const FactorParamsT<double> p) {
  extern __shared__ __align__(16) unsigned char smraw[];
  run_any<CPL, LC, RPL, NW>(p, p.jobs[p.job0 + blockIdx.x], smraw);
}

// Cluster tier: up to three binary levels of the tree in one launch, a level per round, the
// rounds separated by a cluster barrier (a combine takes a third to a tenth of the FP64 job's
// time, so the three levels in sequence cost less than pipelining them did).
template <int CPL, int LC, int RPL, int NW>
__global__ void __launch_bounds__(32 * NW, 16 / NW) k_factor_fx_cluster(const FactorParamsT<double> p,
                                                                        const ClusterSlot *__restrict__ slots) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const ClusterSlot sl = slots[blockIdx.x];
  for (int r = 0; r < 3; ++r) {
    if (sl.job >= 0 && sl.round == r) {
      run_any<CPL, LC, RPL, NW>(p, p.jobs[sl.job], smraw);
      __threadfence();
    }
    if (r < 2) {
      __syncthreads();
      cluster_barrier();
    }
  }
}

size_t cluster_bytes(int n, int nc, int lc, int rpl) {
  const size_t fx = fx_smem_bytes(n, nc, lc, rpl), f64 = factor_smem_bytes(nc, n, sizeof(double));
  return fx > f64 ? fx : f64;
}

template <int CPL, int LC, int RPL, int NW = 8>
cudaError_t launch_fx_cluster(FactorParamsT<double> p, const ClusterSlot *slots, int nclusters, cudaStream_t s) {
  p.ldt = p.n;  // the combines' tiles: what the shared memory below holds for the FP64 job
  const size_t bytes = cluster_bytes(p.n, p.nc, LC, RPL);
  cudaError_t e = cudaFuncSetAttribute(k_factor_fx_cluster<CPL, LC, RPL, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)bytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nclusters * kClusterSize));
  cfg.blockDim = dim3(32 * NW);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kClusterSize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_factor_fx_cluster<CPL, LC, RPL, NW>, p, slots);
}

// Chains of up to 4 and of 9 to 12 columns stay on the FP64 job (half-warps of the CTA own a
// column each): in fixed point such a tile has too few columns for its conversions (2 and 4:
// thin QR of 1.5M rows in 128-row tiles 0.42 and 0.78 ms, 0.53 and 0.91 in fixed point), or
// leaves half of each group empty (1.5M x 12 in 256-row leaves 3.10, 3.31). So do tree nodes of
// up to 8 rows with 9 to 16 columns (200,000 x 8 with one right-hand side 0.43 ms, 0.46). Four
// CTAs per SM fit at 64 registers.
__global__ void __launch_bounds__(kThreads, 4) k_factor_narrow(const FactorParamsT<double> p) {
  extern __shared__ __align__(16) unsigned char smraw[];
  run_job<1>(p, p.jobs[p.job0 + blockIdx.x], smraw);
}

cudaError_t launch_narrow(const FactorParamsT<double> &p, int njobs, cudaStream_t s) {
  const size_t bytes = factor_smem_bytes(p.nc, p.ldt, sizeof(double));
  cudaError_t e = cudaFuncSetAttribute(k_factor_narrow, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  k_factor_narrow<<<njobs, kThreads, bytes, s>>>(p);
  return cudaGetLastError();
}

template <int CPL, int LC, int RPL, int NW = 8>
cudaError_t launch_fx(const FactorParamsT<double> &p, int njobs, cudaStream_t s) {
  const size_t fx = fx_smem_bytes(p.n, p.nc, LC, RPL), f64 = factor_smem_bytes(p.nc, p.ldt, sizeof(double));
  const size_t bytes = fx > f64 ? fx : f64;
  cudaError_t e = cudaFuncSetAttribute(k_factor_fx<CPL, LC, RPL, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  k_factor_fx<CPL, LC, RPL, NW><<<njobs, 32 * NW, bytes, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

int factor_fixed_max_rows(int nc) { return nc <= 16 ? 512 : nc <= 32 ? 288 : nc <= 128 ? 144 : 0; }

cudaError_t launch_factor(const FactorParamsT<double> &p, int njobs, int rows, cudaStream_t s) {
  if (njobs <= 0) return cudaSuccess;
  if (p.nc > 128 || rows > factor_fixed_max_rows(p.nc)) return cudaErrorInvalidValue;
  const bool narrow = rows > 64 ? p.nc <= 4 || (p.nc >= 9 && p.nc <= 12) : p.n <= 8 && p.nc >= 9 && p.nc <= 16;
  if (narrow) return launch_narrow(p, njobs, s);
  if (p.nc <= 8) {
    if (rows <= 64) return launch_fx<1, 1, 2>(p, njobs, s);
    if (rows <= 256) return launch_fx<1, 1, 8>(p, njobs, s);
    return launch_fx<1, 1, 16>(p, njobs, s);
  }
  if (p.nc <= 16) {
    if (rows <= 64) return launch_fx<2, 1, 2>(p, njobs, s);
    if (rows <= 256) return launch_fx<2, 1, 8>(p, njobs, s);
    return launch_fx<2, 1, 16>(p, njobs, s);
  }
  if (p.nc <= 32) {
    if (rows <= 32) return launch_fx<2, 2, 2>(p, njobs, s);
    if (rows <= 160) return launch_fx<2, 2, 10>(p, njobs, s);
    return launch_fx<2, 2, 18>(p, njobs, s);
  }
  if (p.nc <= 64) {
    if (rows <= 64) return launch_fx<2, 4, 8>(p, njobs, s);
    return launch_fx<2, 4, 18>(p, njobs, s);
  }
  return launch_fx<2, 4, 18, 16>(p, njobs, s);
}

size_t cluster_smem_bytes(int n, int nc) {
  if (nc <= 16) return cluster_bytes(n, nc, 1, 2);
  if (nc <= 32) return cluster_bytes(n, nc, 2, 2);
  return cluster_bytes(n, nc, 4, nc <= 64 ? 8 : 18);
}

cudaError_t launch_factor_cluster(const FactorParamsT<double> &p, const ClusterSlot *slots, int nclusters,
                                  cudaStream_t s) {
  if (nclusters <= 0) return cudaSuccess;
  if (p.nc > 128) return cudaErrorInvalidValue;
  if (p.nc <= 8) return launch_fx_cluster<1, 1, 2>(p, slots, nclusters, s);
  if (p.nc <= 16) return launch_fx_cluster<2, 1, 2>(p, slots, nclusters, s);
  if (p.nc <= 32) return launch_fx_cluster<2, 2, 2>(p, slots, nclusters, s);
  if (p.nc <= 64) return launch_fx_cluster<2, 4, 8>(p, slots, nclusters, s);
  return launch_fx_cluster<2, 4, 18, 16>(p, slots, nclusters, s);
}

}  // namespace tsqr
