// FP64 jobs of the batched kernels (factor.cu, factor_wide.cu, resident.cu): the fixed-point
// job without its reflectors (factor_fixed.cuh, KEEP = false), its geometry chosen by the
// width alone, so that a request has the same result in every kernel.
#pragma once
#include "factor_fixed.cuh"

namespace tsqr {
namespace {

// CMAX: the widest item of the launch, in 16 columns. A group per warp: 2, 4, 8, 12, 16 or 24
// columns of up to 36 entries a lane (42 above 128 columns: 56-row tiles; 36-row tiles of 32
// columns a warp took 32 served FP64 requests 76.8 ms, these and the 96-row tiles of 12 columns
// a warp for 65..96 columns 69.4); nodes up to 64 columns wide take builds of their own
// height (a 512-row tile's registers would all be walked for 16 rows). CHAINS: the launch has
// FP64 items; without their builds the kernel's other jobs compile better (16.7M x 32 mixed:
// the factorization 10.4 ms, 11.5 beside them).
//
// What a light tile leaves of a job goes through the FP64 job, out of line: it is rare, and
// inlined it would cost the kernel's other jobs registers.
template <int CMAX, bool COH>
__device__ __noinline__ void run_rest_fp64(const FactorParamsT<double> p, JobDesc job, int done, unsigned char *smraw) {
  job.tile_begin += done;
  job.tile_count -= done;
  run_job<CMAX, COH, false>(p, job, smraw);
}

template <int CMAX, bool CHAINS, bool COH>
__device__ __forceinline__ void run_batch_job(const FactorParamsT<double> &p, const JobDesc job, unsigned char *smraw,
                                              bool node) {
  constexpr int NW = kThreads / 32;
  int done = 0;
  if (p.nc <= 16) {
    if (node) done = run_job_fx<2, 1, 2, NW, false, COH>(p, job, smraw);
    else if constexpr (CHAINS) done = run_job_fx<2, 1, 16, NW, false, COH>(p, job, smraw);
  } else if (p.nc <= 32) {
    if constexpr (CMAX >= 2) {
      if (node) done = run_job_fx<2, 2, 2, NW, false, COH>(p, job, smraw);
      else if constexpr (CHAINS) done = run_job_fx<2, 2, 18, NW, false, COH>(p, job, smraw);
    }
  } else if (p.nc <= 64) {
    if constexpr (CMAX >= 4) {
      if (node) done = run_job_fx<2, 4, 8, NW, false, COH>(p, job, smraw);
      else if constexpr (CHAINS) done = run_job_fx<2, 4, 18, NW, false, COH>(p, job, smraw);
    }
  } else if (p.nc <= 96) {
    if constexpr (CMAX >= 8) done = run_job_fx<3, 4, 12, NW, false, COH>(p, job, smraw);
  } else if (p.nc <= 128) {
    if constexpr (CMAX >= 8) done = run_job_fx<2, 8, 18, NW, false, COH>(p, job, smraw);
  } else {
    if constexpr (CMAX >= 16 && CHAINS) done = run_job_fx<3, 8, 14, NW, false, COH>(p, job, smraw);
  }
  if (done < job.tile_count) run_rest_fp64<CMAX, COH>(p, job, done, smraw);
}

// Items of the batched kernels (bp of k_factor_batch), see factor.cu.
template <int CMAX, bool CHAINS, bool WY, typename WYJOB>
__device__ __forceinline__ void batch_loop(const BatchParams &bp, unsigned char *smraw, int &s_job, int &s_go,
                                           WYJOB wy_job) {
  for (;;) {
    if (threadIdx.x == 0) s_job = atomicAdd(bp.queue, 1);
    __syncthreads();
    int jb = s_job;
    __syncthreads();
    if (jb >= bp.nchains) return;
    for (;;) {
      const BatchJob bj = bp.jobs[jb];
      const BatchInst in = bp.inst[bj.inst];
      const JobDesc jd{bj.piv_row, bj.tile_begin, bj.tile_count};
      const bool chain = jb < bp.nchains;
      if (chain && in.mixed) {
        FactorParamsT<float> fp{};
        fp.A = in.A;
        fp.lda = in.lda;
        fp.V = in.V;
        fp.ldv = in.ldv;
        fp.tiles = bp.tiles;
        fp.tau = in.tau;
        fp.scl = in.scl;
        fp.n = in.n;
        fp.nc = in.n;
        fp.ldt = in.ldt;
        if (WY && in.wy) {  // compact-WY panels, 3xTF32 tensor-core trailing updates
          wy_job(fp, jd, in.n);
        } else {
          switch (in.n <= 16 ? 1 : (in.n <= 32 ? 2 : (in.n <= 64 ? 4 : 8))) {
            case 1: run_job_f32s<1>(fp, jd, smraw); break;
            case 2: if (CMAX >= 2) run_job_f32s<(CMAX >= 2 ? 2 : 1)>(fp, jd, smraw); break;
            case 4: if (CMAX >= 4) run_job_f32s<(CMAX >= 4 ? 4 : 1)>(fp, jd, smraw); break;
            default: if (CMAX >= 8) run_job_f32s<(CMAX >= 8 ? 8 : 1)>(fp, jd, smraw); break;
          }
        }
        // hand the chain's triangle to the FP64 tree storage
        const float *Vs = in.V + bj.piv_row;
        for (int e = threadIdx.x; e < in.n * in.n; e += blockDim.x) {
          const int i = e % in.n, j = e / in.n;
          if (i <= j) in.V64[bj.row64 + i + (int64_t)j * in.ldv64] = (double)__ldcg(Vs + i + (int64_t)j * in.ldv);
        }
        __syncthreads();
      } else {
        FactorParamsT<double> fp{};
        fp.A = in.A;
        fp.lda = in.lda;
        fp.V = in.V64;
        fp.ldv = in.ldv64;
        fp.B = in.B64;
        fp.ldb = in.ldv64;
        fp.Bin = in.B;
        fp.ldbin = in.ldb;
        fp.tiles = bp.tiles;
        fp.n = in.n;
        fp.nc = in.n + in.k;
        fp.ldt = in.ldt64;
        run_batch_job<CMAX, CHAINS, false>(fp, jd, smraw, !chain);
      }
      if (bj.parent < 0) {
        __threadfence();
        finish_instance(in, bj.row64, smraw);
        break;
      }
      // publish this job's triangle, then arrive at the parent; the last child combines
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) s_go = (atomicAdd(bp.counters + bj.parent, 1) == bp.jobs[bj.parent].nchild - 1);
      __syncthreads();
      const int go = s_go;
      __syncthreads();
      if (!go) break;
      __threadfence();
      jb = bj.parent;
    }
  }
}

template <typename K>
cudaError_t launch_batch_kernel(K kernel, const BatchParams &p, int grid, size_t smem_bytes, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
  if (e != cudaSuccess) return e;
  kernel<<<grid, kThreads, smem_bytes, s>>>(p);
  return cudaGetLastError();
}

}  // namespace
}  // namespace tsqr
