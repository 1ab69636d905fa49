// TMA (cp.async.bulk.tensor) and mbarrier helpers for sm_100a, plus the host-side tensor-map encoder.
//
// Every wait is bounded: after kSpinLimit failed polls a waiter records a code in
// g_kernel_fault and gives up, so a logic error ends as an error status instead of a hang.
// Loads use the plain single-CTA form only (one destination CTA).
#ifndef VECTOR_TMA_CUH_
#define VECTOR_TMA_CUH_

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace vec {
namespace tma {

constexpr uint32_t kSpinLimit = 1u << 22;      // polls (each may suspend briefly): on the order of a second, then give up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// CTAS = 2, here and below: the phase has arrivals of the other block of a pair (mbar_arrive_at); acquire_pair() behind the wait.
template <int CTAS = 1>
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (CTAS == 1)
        asm volatile(
            "{\n .reg .pred p;\n"
            " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    else
        asm volatile(
            "{\n .reg .pred p;\n"
            " mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait; returns false (after recording `code` in *fault) if the phase never completed.
template <int CTAS = 1>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* fault, int code) {
    for (uint32_t i = 0; i < kSpinLimit; ++i)
        if (mbar_try_wait<CTAS>(bar, parity)) return true;
    atomicCAS(fault, 0, code);
    return false;
}

// The same wait for a whole warp: every lane polls, and the warp leaves the wait converged (the
// warp-wide .aligned instructions that follow such a wait -- ldmatrix, mma, tcgen05.ld -- require
// it).  All lanes get the same answer.
template <int CTAS = 1>
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, int* fault, int code) {
    const bool ok = mbar_wait<CTAS>(bar, parity, fault, code);
    __syncwarp();
    return __all_sync(0xffffffffu, ok);
}

// Whether the phase has completed, without waiting.
template <int CTAS = 1>
__device__ __forceinline__ uint32_t mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (CTAS == 1)
        asm volatile(
            "{\n .reg .pred p;\n"
            " mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    else
        asm volatile(
            "{\n .reg .pred p;\n"
            " mbarrier.test_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok;
}

// One box of a rank-3 tensor into shared memory; completion is signalled on `bar` by byte count.
__device__ __forceinline__ void load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];\n"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z) : "memory");
}
// The same with an L2 eviction policy: streams that are read once should not push reusable lines
// (partial records, maps, queries) out of L2.
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
    return p;
}
__device__ __forceinline__ void load_3d_hint(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar,
                                             uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5}], [%2], %6;\n"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "l"(policy) : "memory");
}
__device__ __forceinline__ void load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y) : "memory");
}
// For kernels that run alone (CTAS = 1) or as the two blocks of a cluster (CTAS = 2): the address of a shared-memory variable of
// block `block`, and an arrival there.
template <int CTAS>
__device__ __forceinline__ uint32_t block_addr(const void* p, uint32_t block) {
    uint32_t a = smem_u32(p);
    if constexpr (CTAS == 2) asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_u32(p)), "r"(block));
    return a;
}
// From block to block: an arrival there (mbar_arrive_at) releases, and acquire_pair() behind the wait for it acquires, at the scope of
// the cluster, what lies in shared memory -- the keys that a block's loaders wrote and fenced for the tensor cores, which products
// issued by the other block read there.  The order is made by fences that are restricted to shared memory, with the arrival and the polls
// relaxed: an arrival that releases and polls that acquire at that scope order all memory, at the cost of all that the multiprocessor has in
// flight and of its L1 (a route of 16 layers, 8 heads: 341 us; so 196, as without any order).
template <int CTAS>
__device__ __forceinline__ void mbar_arrive_at(uint32_t bar) {
    if constexpr (CTAS == 1) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
    } else {
        asm volatile("fence.release.sync_restrict::shared::cta.cluster;\n" ::: "memory");
        asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(bar) : "memory");
    }
}
template <int CTAS>
__device__ __forceinline__ void acquire_pair() {
    if constexpr (CTAS == 2) asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(map) : "memory");
}

// ---- host side -------------------------------------------------------------
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's encoder, looked up once through the runtime (no link-time dependency on libcuda).
inline EncodeFn encoder() {
    static EncodeFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return (EncodeFn)p;
    }();
    return fn;
}

// bf16 tensor [dim2][dim1][dim0 = 128B-swizzled inner boxes]: rows of `inner` elements, `rows` rows per
// slab at `row_stride_bytes`, `slabs` slabs at `slab_stride_bytes`; box = box_inner x box_rows x 1.
// Rows at or beyond `rows` read as zero.  Returns false if the driver rejects the description.
inline bool encode_bf16_3d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t rows, uint64_t slabs,
                           uint64_t row_stride_bytes, uint64_t slab_stride_bytes, uint32_t box_inner,
                           uint32_t box_rows, uint32_t box_slabs = 1) {
    EncodeFn fn = encoder();
    if (!fn) return false;
    cuuint64_t dims[3] = {inner, rows, slabs};
    cuuint64_t strides[2] = {row_stride_bytes, slab_stride_bytes};
    cuuint32_t box[3] = {box_inner, box_rows, box_slabs};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tma
}  // namespace vec
#endif
