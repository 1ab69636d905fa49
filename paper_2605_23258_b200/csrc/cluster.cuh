// Thread block clusters: rank and size, the cluster barrier, and loads from another block's shared memory.
#ifndef VECTOR_CLUSTER_CUH_
#define VECTOR_CLUSTER_CUH_

#include <stdint.h>

namespace vec {
namespace cl {

__device__ __forceinline__ uint32_t rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t nctas() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(r));
    return r;
}
// The barrier in two halves; every thread of every block of the cluster executes both, warps converged.
__device__ __forceinline__ void arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

// Address of the same shared-memory variable in block `r` of the cluster.
__device__ __forceinline__ uint32_t map_to(uint32_t smem_addr, uint32_t r) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_addr), "r"(r));
    return a;
}
__device__ __forceinline__ float ld_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];\n" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_f32x4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

}  // namespace cl
}  // namespace vec
#endif
