// The cluster-wide barrier of the factorization's cluster tier (sm_103a): what each CTA wrote
// before it is seen by the cluster's other CTAs after it.
#pragma once

namespace tsqr {

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace tsqr
