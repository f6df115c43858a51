// Device helpers of the cluster-scope kernels: one thread-block cluster (8 to 16 CTAs) works
// on a system of its own, so a synchronisation is the hardware's cluster barrier and a sum over
// the system goes through distributed shared memory (a few hundred ns together), where a
// grid-wide step pays two to three microseconds for its counter and its partials in L2.
#pragma once

#include "common.cuh"

namespace asss {

constexpr int CL_MAX = 16;   // CTAs of a cluster (the non-portable maximum)

__device__ __forceinline__ unsigned cl_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cl_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cl_id() {
    unsigned r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cl_count() {
    unsigned r;
    asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
    return r;
}
// every thread of the cluster arrives and waits; what was written before (global or
// distributed shared memory) is visible to the whole cluster afterwards
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the two halves of cl_sync: work between them overlaps the barrier
__device__ __forceinline__ void cl_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// one value into the same shared variable of CTAs first, first + 4, ... (four lanes together
// reach them all)
__device__ __forceinline__ void cl_store_every4(float* var, unsigned first, unsigned n, float v) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(var);
#pragma unroll
    for (unsigned u = 0; u < CL_MAX / 4; ++u) {
        const unsigned q = first + 4 * u;
        if (q < n) {
            unsigned ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(q));
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(ra), "f"(v) : "memory");
        }
    }
}
__device__ __forceinline__ void cl_store_every4(double* var, unsigned first, unsigned n, double v) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(var);
#pragma unroll
    for (unsigned u = 0; u < CL_MAX / 4; ++u) {
        const unsigned q = first + 4 * u;
        if (q < n) {
            unsigned ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(q));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
        }
    }
}
// 8 bytes into the same shared variable of CTA `rank`
__device__ __forceinline__ void cl_store8(void* var, unsigned rank, unsigned long long bits) {
    unsigned a = (unsigned)__cvta_generic_to_shared(var), ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(ra), "l"(bits) : "memory");
}
__device__ __forceinline__ unsigned long long cl_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long cl_bits(float2 v) {
    return (unsigned long long)__float_as_uint(v.x) | ((unsigned long long)__float_as_uint(v.y) << 32);
}

}  // namespace asss
