// Device helpers shared by the solve-phase kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "amg.h"

namespace amg {

template <int W, typename T>
__device__ __forceinline__ T group_sum(T s) {
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off, W);
    return s;
}

__device__ __forceinline__ double fmad(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fmad(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// The checked build (compiled with AMG_DEVICE_CHECKS): every gathered index,
// restriction-list row and aggregate index is tested against its range
// before use; one outside it is recorded as AMG_ERANGE in the solve's status
// word and contributes zero instead of being read.  In the regular build the
// test is the constant true and costs nothing.
#ifdef AMG_DEVICE_CHECKS
constexpr bool kChecks = true;
#else
constexpr bool kChecks = false;
#endif
__device__ __forceinline__ bool index_ok(int j, int n, int32_t* err) {
    if (!kChecks) return true;
    if ((unsigned)j < (unsigned)n) return true;
    if (err) atomicCAS(err, 0, AMG_ERANGE);
    return false;
}

// programmatic dependent launch: let the next kernel of the stream start, and
// wait for every predecessor to finish (both are no-ops without the launch
// attribute)
__device__ __forceinline__ void pdl_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// thread-block clusters: the barrier in its two halves (release, acquire), the
// block's rank, and stores into another block's shared memory.  The barrier's
// aligned forms want the whole warp at the same instruction, which the compiler
// does not know: the warp meets here, whatever the caller's loops did.
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t o;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(addr), "r"(rank));
    return o;
}
__device__ __forceinline__ void st_cluster(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

}  // namespace amg
