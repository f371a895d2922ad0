// Thread-block cluster helpers: rank, addresses in another CTA's shared memory,
// and the cluster barrier (a CTA barrier for a cluster of one).
#pragma once

#include <cuda_runtime.h>

namespace pf {

__device__ __forceinline__ int cluster_rank() {
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the address in CTA `rank` of the cluster of a shared-memory address of this CTA
template <typename T>
__device__ __forceinline__ T* cluster_map(T* p, int rank) {
    T* q;
    asm("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(rank));
    return q;
}
__device__ __forceinline__ void cluster_sync(int C) {
    if (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;\n"
                     "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

}  // namespace pf
