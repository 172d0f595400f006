// mg_cluster.cuh -- blocks of a thread-block cluster: ranks, the barrier and
// access to each other's shared memory.
//
// Another block's shared memory may be touched only between two cluster barriers:
// the first access (ld_cluster, st_cluster) comes after a barrier that every block
// has arrived at since it started, and a block leaves after a barrier that every
// block arrives at behind its last access.
#pragma once

#include "mg_bulk.cuh"  // smem_u32

namespace gbmg {

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The two halves of the cluster barrier: what a thread wrote before it arrives
// is seen by every thread that has waited.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}
// Address in block `rank` of the shared variable at `addr` in this one.
__device__ __forceinline__ unsigned map_rank(unsigned addr, unsigned rank)
{
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ double ld_cluster(unsigned addr)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(unsigned addr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

}  // namespace gbmg
