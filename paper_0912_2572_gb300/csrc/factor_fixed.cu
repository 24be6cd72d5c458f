// The one-problem factorization launches of up to 64 columns in 64-bit fixed point
// (factor_fixed.cuh): the chain launch and the tree levels.
#include "cluster_sync.cuh"
#include "factor_fixed.cuh"

namespace tsqr {
namespace {

// At most 40 entries (80 registers) per thread, so two CTAs of eight warps fit an SM at 128
// registers. A tile the fixed-point form cannot take and the rest of its chain go through
// the FP64 job.
template <int CPL, int LC, int RPL>
__global__ void __launch_bounds__(kThreads, 2) k_factor_fx(const FactorParamsT<double> p) {
  extern __shared__ __align__(16) unsigned char smraw[];
  JobDesc job = p.jobs[p.job0 + blockIdx.x];
  const int done = run_job_fx<CPL, LC, RPL, kThreads / 32>(p, job, smraw);
  if (done < job.tile_count) {
    job.tile_begin += done;
    job.tile_count -= done;
    run_job<(LC == 1 ? 1 : LC == 2 ? 2 : 4), true>(p, job, smraw);
  }
}

// Cluster tier: up to three binary levels of the tree in one launch, a level per round, the
// rounds separated by a cluster barrier (a combine takes a tenth of the FP64 job's time, so
// the three levels in sequence cost less than pipelining them did).
template <int CPL, int LC, int RPL>
__global__ void __launch_bounds__(kThreads, 2) k_factor_fx_cluster(const FactorParamsT<double> p,
                                                                   const ClusterSlot *__restrict__ slots) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const ClusterSlot sl = slots[blockIdx.x];
  for (int r = 0; r < 3; ++r) {
    if (sl.job >= 0 && sl.round == r) {
      const JobDesc job = p.jobs[sl.job];
      if (run_job_fx<CPL, LC, RPL, kThreads / 32>(p, job, smraw) < job.tile_count)
        run_job<(LC == 1 ? 1 : LC == 2 ? 2 : 4), true>(p, job, smraw);
      __threadfence();
    }
    if (r < 2) cluster_barrier();
  }
}

template <int CPL, int LC, int RPL>
cudaError_t launch_fx_cluster(const FactorParamsT<double> &p, const ClusterSlot *slots, int nclusters,
                              cudaStream_t s) {
  const size_t fx = fx_smem_bytes(p.n, p.nc, (32 / LC * RPL + 31) / 32 * 32), f64 = factor_smem_bytes(p.nc, p.n, sizeof(double));
  const size_t bytes = fx > f64 ? fx : f64;
  cudaError_t e = cudaFuncSetAttribute(k_factor_fx_cluster<CPL, LC, RPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)bytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nclusters * kClusterSize));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kClusterSize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_factor_fx_cluster<CPL, LC, RPL>, p, slots);
}

template <int CPL, int LC, int RPL>
cudaError_t launch_fx(const FactorParamsT<double> &p, int njobs, cudaStream_t s) {
  const size_t fx = fx_smem_bytes(p.n, p.nc, (32 / LC * RPL + 31) / 32 * 32), f64 = factor_smem_bytes(p.nc, p.ldt, sizeof(double));
  const size_t bytes = fx > f64 ? fx : f64;
  cudaError_t e = cudaFuncSetAttribute(k_factor_fx<CPL, LC, RPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  k_factor_fx<CPL, LC, RPL><<<njobs, kThreads, bytes, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

int factor_fixed_max_rows(int nc) { return nc <= 16 ? 512 : nc <= 32 ? 288 : nc <= 64 ? 144 : 0; }

cudaError_t launch_factor_fixed(const FactorParamsT<double> &p, int njobs, int rows, cudaStream_t s) {
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
  if (rows <= 64) return launch_fx<2, 4, 8>(p, njobs, s);
  return launch_fx<2, 4, 18>(p, njobs, s);
}

cudaError_t launch_factor_fixed_cluster(const FactorParamsT<double> &p, const ClusterSlot *slots, int nclusters,
                                        cudaStream_t s) {
  if (p.nc <= 8) return launch_fx_cluster<1, 1, 2>(p, slots, nclusters, s);
  if (p.nc <= 16) return launch_fx_cluster<2, 1, 2>(p, slots, nclusters, s);
  if (p.nc <= 32) return launch_fx_cluster<2, 2, 2>(p, slots, nclusters, s);
  return launch_fx_cluster<2, 4, 8>(p, slots, nclusters, s);
}

}  // namespace tsqr
