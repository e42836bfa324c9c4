// cluster.cuh -- the two halves of the barrier over a cluster's blocks.
//
// The aligned forms must be executed by all threads of a warp together, so the
// arrival brings the warp together first: what comes before it may have been done
// by some lanes alone, and after a branch nothing else says that the others wait.
#pragma once

namespace wx {

__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}

__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace wx
