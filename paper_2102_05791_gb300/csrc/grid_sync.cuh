// Wait limit of grid-wide exchanges, and the cluster barrier and
// distributed-shared-memory accesses of one-cluster grids.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace softsim {

constexpr int kGridWaitPolls = 1 << 22;  // polls (L2 round trips) of one grid-barrier wait before it gives up

// Thread-block cluster primitives (the whole grid is one cluster of at most
// 16 CTAs): a hardware barrier over every thread of the cluster with
// release/acquire semantics at cluster scope, and loads from another CTA's
// shared memory (distributed shared memory).
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// This CTA's rank in its cluster.
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Address of the same shared-memory object in the CTA of the given cluster rank.
__device__ __forceinline__ uint32_t dsmem_addr(const void *local, uint32_t rank)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

__device__ __forceinline__ int ld_dsmem_s32(const void *local, uint32_t rank)
{
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(dsmem_addr(local, rank)) : "memory");
    return v;
}

}  // namespace softsim
