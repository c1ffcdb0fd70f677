// rbe_cluster.cuh -- thread-block cluster primitives shared by the kernels that
// run as one cluster (rbe_small.cu, rbe_cells.cu).
#pragma once

#include <cstdint>

namespace rbe {

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t local_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// shared::cluster address in block `rank` of this block's shared address a
__device__ __forceinline__ uint32_t remote(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

}  // namespace rbe
