// cluster.cuh -- shared memory of a thread-block cluster: addresses in other
// blocks, loads, stores and atomics on them, and the cluster barrier.  SOLO:
// a "cluster" of one block, whose accesses are plain shared-memory ones.
#pragma once
#include <stdint.h>

namespace hp {

__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
template <bool SOLO>
__device__ __forceinline__ void cl_sync() {
    if (SOLO) {
        __syncthreads();
    } else {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n"
                     "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
// address of this block's shared address a in block `rank`
template <bool SOLO>
__device__ __forceinline__ uint32_t cl_map(uint32_t a, uint32_t rank) {
    if (SOLO) return a;
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
template <bool SOLO>
__device__ __forceinline__ uint32_t cl_load(uint32_t a) {
    uint32_t v;
    if (SOLO)
        asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    else
        asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
template <bool SOLO>
__device__ __forceinline__ void cl_store(uint32_t a, uint32_t v) {
    if (SOLO)
        asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
    else
        asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
template <bool SOLO>
__device__ __forceinline__ uint32_t cl_add(uint32_t a, uint32_t v) {
    uint32_t old;
    if (SOLO)
        asm volatile("atom.relaxed.cta.shared::cta.add.u32 %0, [%1], %2;"
                     : "=r"(old) : "r"(a), "r"(v) : "memory");
    else
        asm volatile("atom.relaxed.cluster.shared::cluster.add.u32 %0, [%1], %2;"
                     : "=r"(old) : "r"(a), "r"(v) : "memory");
    return old;
}
template <bool SOLO>
__device__ __forceinline__ void cl_red_add(uint32_t a, uint32_t v) {
    if (SOLO)
        asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
    else
        asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(v)
                     : "memory");
}
template <bool SOLO>
__device__ __forceinline__ void cl_red_or(uint32_t a, uint32_t v) {
    if (SOLO)
        asm volatile("red.relaxed.cta.shared::cta.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
    else
        asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(v)
                     : "memory");
}
template <bool SOLO>
__device__ __forceinline__ uint32_t cl_min(uint32_t a, uint32_t v) {
    uint32_t old;
    if (SOLO)
        asm volatile("atom.relaxed.cta.shared::cta.min.u32 %0, [%1], %2;"
                     : "=r"(old) : "r"(a), "r"(v) : "memory");
    else
        asm volatile("atom.relaxed.cluster.shared::cluster.min.u32 %0, [%1], %2;"
                     : "=r"(old) : "r"(a), "r"(v) : "memory");
    return old;
}

template <bool SOLO>
__device__ __forceinline__ void cl_red_min(uint32_t a, uint32_t v) {
    if (SOLO)
        asm volatile("red.relaxed.cta.shared::cta.min.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
    else
        asm volatile("red.relaxed.cluster.shared::cluster.min.u32 [%0], %1;" ::"r"(a), "r"(v)
                     : "memory");
}

}  // namespace hp
