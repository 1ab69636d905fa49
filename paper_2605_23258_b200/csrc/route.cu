// Three-way routing (paper Section 3.2): Step 1 pool selection by base score,
// Step 2 reconstruction residual on the pool, Step 3 truncation by residual.
//
// Both selections are exact top-k with the lower index winning ties (select.cuh): a
// most-significant-digit radix select on an order-preserving 32-bit image of the fp32
// value, followed by one ordered walk whose block-wide prefix sums place the chosen
// indices in ascending order.  One thread block per unit.
#include "common.cuh"
#include "internal.h"
#include "residual_layer_tc.cuh"
#include "residual_tc.cuh"
#include "select.cuh"

namespace vec {

using sel::Layout;

// Forms of a selection: the input in registers (select_regs), or two passes over it in memory (select.cuh) by blocks of 8 warps (four
// resident per multiprocessor), of 16 (two) or of 32 (one, with masks and list in up to 200 KB) warps.
constexpr int SEL_REGS16 = 16384, SEL_REGS = 32768, SEL_LONG = 262144;
constexpr size_t SEL_SMEM_LONG = 200 * 1024, SEL_SMEM_MID = 92 * 1024, SEL_SMEM_SHORT = 36 * 1024;
#define VEC_SEL_BOUNDS(NW) __launch_bounds__(32 * NW, NW == 32 ? 1 : NW == 16 ? 2 : 4)

// The general selection (select_emit) as functions of their own: the kernels run the lean path inline and
// come here only when it gives up, so its registers are not theirs to carry.
template <int NW>
__device__ __noinline__ void pool_select_general(const float* s, int n, int n_pool, int32_t* __restrict__ out,
                                                 sel::Scratch& S, const Layout& L, uint32_t* dyn) {
    sel::select_emit<false, NW, true>(s, n, n_pool, true, S, L, dyn, [&](int i, bool chosen, int pos) { if (chosen) out[pos] = i; });
}

struct PoolOut {
    int32_t* out;
    __device__ __forceinline__ int32_t* list() const { return out; }
};

struct TruncateOut {
    const int32_t* pool;
    uint8_t* tr;
    int32_t* ro;
    int32_t* ao;
    int64_t N;
    __device__ __forceinline__ int fetch(int p) const { return pool[p]; }
    __device__ __forceinline__ void put(int, int token, bool is_apx, int pos) const {
        if ((uint64_t)(int64_t)token >= (uint64_t)N) return;          // a pool entry outside the unit is dropped
        if (is_apx) { ao[pos] = token; tr[token] = 1; }
        else        { ro[pos] = token; tr[token] = 2; }
    }
    __device__ __forceinline__ void operator()(int p, bool is_apx, int pos) const { put(p, pool[p], is_apx, pos); }
};

template <int NW>
__device__ __noinline__ void truncate_general(const float* e, int n_pool, int n_apx, const TruncateOut& emit,
                                              sel::Scratch& S, const Layout& L, uint32_t* dyn) {
    sel::select_emit<true, NW, false>(e, n_pool, n_apx, n_apx > 0, S, L, dyn, emit);
}

// Step 1.  grid (U), 32 NW threads, L.bytes() of dynamic shared memory.  zero (nullable): [U][n_pool] floats set to zero,
// for a residual kernel that adds its results up.
template <int NW>
__global__ void VEC_SEL_BOUNDS(NW)
pool_select_kernel(const float* scores, int64_t N, int n_pool, int32_t* __restrict__ pool_idx, float* __restrict__ zero,
                   const Layout L) {
    __shared__ sel::Scratch S;
    extern __shared__ __align__(16) uint32_t sel_dyn[];
    // A programmatic dependent of what precedes it: nothing is touched before the wait.  Inside vector_route the residual
    // kernel is one of this kernel: its blocks may take SMs as this grid's blocks leave them -- what was before this kernel
    // has finished then -- and it reads the index lists only after its own wait.
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int u = blockIdx.x, n = (int)N;
    const float* s = scores + (size_t)u * N;
    int32_t* out = pool_idx + (size_t)u * n_pool;
    if (n_pool <= 0) return;
    if (zero)
        for (int i = threadIdx.x; i < n_pool; i += 32 * NW) zero[(size_t)u * n_pool + i] = 0.f;
    if (L.keyed && sel::select_lean<false, NW, true>(s, n, n_pool, S, L, sel_dyn, PoolOut{out})) return;
    pool_select_general<NW>(s, n, n_pool, out, S, L, sel_dyn);
}

// n bytes set to zero by a block, 16 at a time where they lie so.
template <int NW>
__device__ __forceinline__ void clear_bytes(uint8_t* p, int64_t n) {
    if (((n | (int64_t)(uintptr_t)p) & 15) == 0) {
        for (int64_t i = threadIdx.x; i < n / 16; i += 32 * NW) reinterpret_cast<uint4*>(p)[i] = make_uint4(0, 0, 0, 0);
    } else {
        for (int64_t i = threadIdx.x; i < n; i += 32 * NW) p[i] = 0;
    }
}

// Step 3.  grid (U), 32 NW threads, L.bytes() of dynamic shared memory.
template <int NW>
__global__ void VEC_SEL_BOUNDS(NW)
truncate_kernel(const float* eps, const int32_t* pool_idx, int64_t N, int n_pool,
                int n_apx, uint8_t* __restrict__ tier, int32_t* __restrict__ ret_idx,
                int32_t* __restrict__ apx_idx, const Layout L) {
    __shared__ sel::Scratch S;
    extern __shared__ __align__(16) uint32_t sel_dyn[];
    const int u = blockIdx.x;
    uint8_t* tr = tier + (size_t)u * N;
    clear_bytes<NW>(tr, N);
    // Everything above touches only the tier map, which the residual kernel, this one's primary, neither reads nor writes, and
    // nothing before that kernel is still under way: it waits before it lets this one start.  (No wait unless a dependent.)
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    __syncthreads();
    const float* e = eps + (size_t)u * n_pool;
    const int n_ret = n_pool - n_apx;
    const TruncateOut emit = {pool_idx + (size_t)u * n_pool, tr, ret_idx + (size_t)u * n_ret, apx_idx + (size_t)u * n_apx, N};
    if (L.keyed && n_apx > 0 && sel::select_lean<true, NW, false>(e, n_pool, n_apx, S, L, sel_dyn, emit)) return;
    truncate_general<NW>(e, n_pool, n_apx, emit, S, L, sel_dyn);
}

// Steps 1 and 3 with the input in registers.  grid (U), 32 NW threads.
struct PoolRegsOut {
    int32_t* out;
    __device__ __forceinline__ void put(int i, int pos) const { out[pos] = i; }
};
template <int E> struct TruncateRegsOut {
    TruncateOut to;
    const int32_t (&token)[E];
    __device__ __forceinline__ void put(int j, int p, bool is_apx, int pos) const { to.put(p, token[j], is_apx, pos); }
};
template <int NW, int E>
__global__ void VEC_SEL_BOUNDS(NW)
pool_select_regs(const float* scores, int64_t N, int n_pool, int32_t* __restrict__ pool_idx, float* __restrict__ zero) {
    __shared__ __align__(16) sel::RegScratch<NW> S;
    sel::regs_clear(S);
    // as in pool_select_kernel
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int u = blockIdx.x;
    if (n_pool <= 0) return;
    if (zero)
        for (int i = threadIdx.x; i < n_pool; i += 32 * NW) zero[(size_t)u * n_pool + i] = 0.f;
    __syncthreads();
    sel::select_regs<false, NW, E, true>(scores + (size_t)u * N, (int)N, n_pool, S, PoolRegsOut{pool_idx + (size_t)u * n_pool});
}

template <int NW, int E>
__global__ void VEC_SEL_BOUNDS(NW)
truncate_regs(const float* eps, const int32_t* pool_idx, int64_t N, int n_pool, int n_apx,
              uint8_t* __restrict__ tier, int32_t* __restrict__ ret_idx, int32_t* __restrict__ apx_idx) {
    __shared__ __align__(16) sel::RegScratch<NW> S;
    const int u = blockIdx.x;
    uint8_t* tr = tier + (size_t)u * N;
    clear_bytes<NW>(tr, N);
    sel::regs_clear(S);
    // as in truncate_kernel; the list of the pool, which a kernel of the same chain wrote, is read behind the wait as the residuals are
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    __syncthreads();
    const int32_t* pool = pool_idx + (size_t)u * n_pool;
    int32_t token[E];
    const int groups = sel::regs_groups<NW>(n_pool), p0 = (threadIdx.x >> 5) * groups * 32 + (threadIdx.x & 31);
#pragma unroll
    for (int j = 0; j < E; ++j) token[j] = j < groups && p0 + 32 * j < n_pool ? pool[p0 + 32 * j] : 0;
    const TruncateOut to = {pool, tr, ret_idx + (size_t)u * (n_pool - n_apx), apx_idx + (size_t)u * n_apx, N};
    sel::select_regs<true, NW, E, false>(eps + (size_t)u * n_pool, n_pool, n_apx, S, TruncateRegsOut<E>{to, token});
}

// Step 2 on CUDA cores (fp32, and 64-channel bf16 rows off a 16-byte boundary).  A warp takes RW listed rows at once, a lane the output channels lane, lane + 32, ...: an
// element of W^T read from shared memory serves the RW rows, and their loads are under way while W is staged (one row after
// the other, each from its load to its sum: 30 us for 2 units of 384 rows).  RW = 4 where that leaves a block for
// every multiprocessor, else 2.  grid (ceil(n_idx / (8 RW)), U), 256 threads; dynamic shared memory: W^T as D * (D+1)
// floats plus RW key rows per warp.
// With ROPE the regressor sees the key turned back by its position (the token index): channel c
// pairs with c + D/2, angle -pos * theta^(-2c/D).
template <typename T, int D, bool ROPE, int RW>
__global__ void __launch_bounds__(256)
residual_generic(const T* K, const T* V, const T* W, int64_t N,
                 int LH, const int32_t* idx, int n_idx, float theta, float* __restrict__ eps) {
    constexpr int CPL = D / 32;             // channels per lane
    extern __shared__ __align__(16) float smem[];
    __shared__ double inv_freq[ROPE ? D / 2 : 1];
    float* ks = smem;                       // [8][RW][D]
    float* Wt = smem + 8 * RW * D;          // Wt[c_in * (D+1) + c_out]
    if (ROPE) rope_fill_inv_freq(inv_freq, D, theta);
    asm volatile("griddepcontrol.wait;\n" ::: "memory");              // idx is complete and visible from here on
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int u = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int p0 = (blockIdx.x * 8 + wid) * RW;
    int64_t tok[RW];
    float kr[RW][CPL], vr[RW][CPL];
#pragma unroll
    for (int r = 0; r < RW; ++r) tok[r] = p0 + r < n_idx ? idx[(size_t)u * n_idx + p0 + r] : -1;
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const bool in = (uint64_t)tok[r] < (uint64_t)N;          // an index outside the unit reads as a row of zeros
#pragma unroll
        for (int m = 0; m < CPL; ++m) {
            kr[r][m] = in ? to_f32(K[((size_t)u * N + tok[r]) * D + lane + 32 * m]) : 0.f;
            vr[r][m] = in ? to_f32(V[((size_t)u * N + tok[r]) * D + lane + 32 * m]) : 0.f;
        }
    }
    const T* Wu = W + (size_t)(u % LH) * D * D;
#pragma unroll 16
    for (int e = threadIdx.x; e < D * D; e += 256) {
        const int co = e / D, ci = e % D;
        Wt[ci * (D + 1) + co] = to_f32(Wu[e]);
    }
    float* kw = ks + wid * RW * D;
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int m = 0; m < CPL; ++m) kw[r * D + lane + 32 * m] = kr[r][m];
    __syncthreads();
    if (ROPE) {
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int c = lane; c < D / 2; c += 32) {
                float cs, sn;
                rope_cos_sin((double)tok[r], inv_freq[c], cs, sn);
                const float x = kw[r * D + c], y = kw[r * D + c + D / 2];
                kw[r * D + c] = fmaf(x, cs, y * sn);
                kw[r * D + c + D / 2] = fmaf(y, cs, -x * sn);
            }
        __syncwarp();
    }
    float pred[RW][CPL];
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int m = 0; m < CPL; ++m) pred[r][m] = 0.f;
#pragma unroll 4
    for (int ci = 0; ci < D; ci += 4) {
        float4 k[RW];
#pragma unroll
        for (int r = 0; r < RW; ++r) k[r] = *reinterpret_cast<const float4*>(kw + r * D + ci);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int m = 0; m < CPL; ++m) {
                const float w = Wt[(ci + q) * (D + 1) + lane + 32 * m];
#pragma unroll
                for (int r = 0; r < RW; ++r) pred[r][m] = fmaf(w, q == 0 ? k[r].x : q == 1 ? k[r].y : q == 2 ? k[r].z : k[r].w, pred[r][m]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        float e = 0.f;
#pragma unroll
        for (int m = 0; m < CPL; ++m) {
            const float x = vr[r][m] - pred[r][m];
            e = fmaf(x, x, e);
        }
        e = warp_sum(e);
        if (lane == 0 && p0 + r < n_idx) eps[(size_t)u * n_idx + p0 + r] = e;
    }
}

template <typename T, int D, bool ROPE, int RW>
static vector_status launch_residual_rows(const Dims& dm, const void* K, const void* V, const void* W, int64_t N, const int32_t* idx,
                                          int64_t n_idx, float* eps, cudaStream_t st) {
    constexpr int SMEM = (D * (D + 1) + 8 * RW * D) * (int)sizeof(float);
    auto kern = residual_generic<T, D, ROPE, RW>;
    static PerDeviceOnce once;
    if (once.first()) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
        if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
    }
    VEC_CUDA_CHECK(launch_maybe_dependent(true, kern, dim3((unsigned)((n_idx + 8 * RW - 1) / (8 * RW)), dm.U), dim3(256), SMEM, st,
                                          (const T*)K, (const T*)V, (const T*)W, N, dm.LH, idx, (int)n_idx, dm.theta, eps));
    return VECTOR_OK;
}

template <typename T, int D>
static vector_status launch_residual(const Dims& dm, const void* K, const void* V, const void* W, int64_t N,
                                     const int32_t* idx, int64_t n_idx, float* eps, cudaStream_t st) {
    if (n_idx == 0) return VECTOR_OK;
    const bool many = (n_idx + 31) / 32 * dm.U >= sm_count();
    if (dm.rope)
        return many ? launch_residual_rows<T, D, true, 4>(dm, K, V, W, N, idx, n_idx, eps, st)
                    : launch_residual_rows<T, D, true, 2>(dm, K, V, W, N, idx, n_idx, eps, st);
    return many ? launch_residual_rows<T, D, false, 4>(dm, K, V, W, N, idx, n_idx, eps, st)
                : launch_residual_rows<T, D, false, 2>(dm, K, V, W, N, idx, n_idx, eps, st);
}

// bf16: gather + tcgen05 residual kernel.
template <int D>
static vector_status launch_residual_tc(const Dims& dm, const void* K, const void* V, const void* W, int64_t N,
                                        const int32_t* idx, int64_t n_idx, float* eps, cudaStream_t st, bool dependent) {
    if (n_idx == 0) return VECTOR_OK;
    using Plain = rtc::RCfg<D, false>;
    using Rope = rtc::RCfg<D, true>;
    static PerDeviceOnce once;
    if (once.first()) {
        cudaError_t e = cudaFuncSetAttribute(rtc::residual_tc<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Plain::SMEM_BYTES);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(rtc::residual_tc<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Rope::SMEM_BYTES);
        if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
    }
    int* fault = kernel_fault_address();
    if (!fault) return VECTOR_ERR_CUDA;
    CUtensorMap mapW;
    if (!tma::encode_bf16_3d(&mapW, W, D, D, (uint64_t)dm.LH, 2 * D, D * 2 * D, 64, D)) return VECTOR_ERR_CUDA;
    rtc::Params P;
    P.U = dm.U; P.LH = dm.LH; P.n_idx = (int)n_idx; P.N = N;
    P.tpu = (int)((n_idx + rtc::TILE - 1) / rtc::TILE);
    P.n_tiles = (long long)dm.U * P.tpu;
    const int sms = sm_count();
    const int blocks = (int)(P.n_tiles < sms ? P.n_tiles : sms);
    RopePhases ph = {};
    if (dm.rope) rope_phases(dm.theta, D, &ph);
    // dependent: blocks may take SMs while the kernel that writes idx drains; the loaders wait for it
    const __nv_bfloat16* Kp = (const __nv_bfloat16*)K;
    const __nv_bfloat16* Vp = (const __nv_bfloat16*)V;
    if (dm.rope)
        VEC_CUDA_CHECK(launch_maybe_dependent(dependent, rtc::residual_tc<D, true>, dim3(blocks), dim3(Rope::THREADS),
                                              Rope::SMEM_BYTES, st, Kp, Vp, mapW, idx, P, ph, eps, fault));
    else
        VEC_CUDA_CHECK(launch_maybe_dependent(dependent, rtc::residual_tc<D, false>, dim3(blocks), dim3(Plain::THREADS),
                                              Plain::SMEM_BYTES, st, Kp, Vp, mapW, idx, P, ph, eps, fault));
    return VECTOR_OK;
}

static vector_status residual_dispatch(const Dims& dm, const void* K, const void* V, const void* W, int64_t N,
                                       const int32_t* idx, int64_t n_idx, float* eps, cudaStream_t st,
                                       bool dependent = false) {
    if (dm.dtype == VECTOR_BF16 && dm.d == 64 && (((uintptr_t)K | (uintptr_t)V | (uintptr_t)W) & 15))
        return launch_residual<__nv_bfloat16, 64>(dm, K, V, W, N, idx, n_idx, eps, st);
    if (dm.dtype == VECTOR_BF16)
        return dm.d == 64 ? launch_residual_tc<64>(dm, K, V, W, N, idx, n_idx, eps, st, dependent)
                          : launch_residual_tc<128>(dm, K, V, W, N, idx, n_idx, eps, st, dependent);
    return dm.d == 64 ? launch_residual<float, 64>(dm, K, V, W, N, idx, n_idx, eps, st)
                      : launch_residual<float, 128>(dm, K, V, W, N, idx, n_idx, eps, st);
}

// One-time opt-in to the dynamic shared memory of the selection kernels.
static vector_status select_kernels_setup() {
    static PerDeviceOnce once;
    if (!once.first()) return VECTOR_OK;
    cudaError_t e = cudaFuncSetAttribute(pool_select_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_SMEM_LONG);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(pool_select_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_SMEM_MID);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(pool_select_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_SMEM_SHORT);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(truncate_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_SMEM_LONG);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(truncate_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_SMEM_MID);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(truncate_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_SMEM_SHORT);
    if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
    return VECTOR_OK;
}

static Layout selection_layout(int64_t n, int nw) {
    const size_t budget = nw == 8 ? SEL_SMEM_SHORT : nw == 16 ? SEL_SMEM_MID : SEL_SMEM_LONG;
    return sel::plan_layout(n, budget, nw == 8 ? 1024 : 2048, nw);
}
// Warps of a block that passes over memory, 0: the input in registers.  Registers win for every count of short lists and, up to their
// length, where a list has a multiprocessor to itself.  Many longer lists are served best by the small blocks, whose phases of latency
// overlap; their second round (4 to 8 lists a multiprocessor) is nearly empty.
// Step 1 writes its list out in one sweep where it fits the candidates' place in shared memory, by scattered stores where it does
// not, which decides between the forms.  us, scores from HBM, registers / 8 / 16 warps, `*`: the list does not fit.  148 lists of 12000
// 10.6 / 13.6 / 10.9, of 20011 14.4 / 26.8 / 19.2; 256 of 14000 16.5 / 19.8 / 15.8, of 20011 27.8 / 29.8 / 23.3; 444 of 6500 14.4 / 14.5 / 18.8, 592 of
// 8192 19.5 / 17.1 / 23.7; 592 of 14000, 0.3 of them listed, 30.6 / 26.1 / 30.6, half of them 30.6 / 40.4* / 31.8; 592 of 26000, 0.15 listed, 62.9 /
// 43.5 / 48.2, 0.3 listed 62.2 / 54.3* / 48.9, 0.8 listed 63.1 / 97.3* / 94.3*; 640 of 32767, 0.15 listed, 86 / 85 / 79; 1184 of 16384, 0.3 listed,
// 63 / 56 / -, half of them 64 / 84* / -.
static int pool_select_warps(int64_t n, int U, int64_t n_pool) {
    const int sms = sm_count();
    auto list_fits = [&](int nw) { return n_pool <= selection_layout(n, nw).cand_cap; };
    if (n <= 4096 || (n <= SEL_REGS && U <= sms)) return 0;
    if (n <= 8192) return U <= 3 * sms || !list_fits(8) ? 0 : 8;
    if (n <= SEL_REGS) {
        if (U > 2 * sms && list_fits(8) && (n <= 20480 || U <= 4 * sms || U >= 8 * sms)) return 8;
        return (n <= SEL_REGS16 ? U <= 2 * sms : list_fits(16)) ? 16 : 0;
    }
    return n < SEL_LONG ? 16 : 32;
}
// Step 3, us as above: 148 lists of 12000 12.8 / 21.9 / 16.1, 296 of 12000 24.5 / 25.9 / 22.4, 592 of 12000 49 / 41 / 45, 640 of 16384 77 / 76 / 73, 1184
// of 16384 126 / 107 / 113; 2368 of 5000 84 / 82 / 111, of 8192 108 / 111 / 135; 148 of 20011 in 64 registers a thread, which do not hold image
// and token, 41.9 / 35.0 / 25.3; 888 of 20011 - / 125 / 118, 1184 of 20011 - / 149 / 155, of 26000 - / 179 / 177.
static int truncate_warps(int64_t n, int U) {
    const int sms = sm_count();
    if (n <= 8192 || (n <= SEL_REGS16 && U <= sms)) return 0;
    if (n <= SEL_REGS16 ? U > 2 * sms && (U <= 4 * sms || U >= 8 * sms) : n <= 24576 && U >= 8 * sms) return 8;
    return n < SEL_LONG ? 16 : 32;
}

// With the input in registers, 32 warps a block instead of 16: half the elements a thread, where a list has a multiprocessor to itself
// (two blocks of 16 warps share one, which 32 would take for themselves) and is long enough that counting and handing out outweigh the
// barriers.  us in a graph, 16 / 32 warps, Step 1 and Step 3: 8 lists of 2048 3.8 / 3.7 and 4.5 / 4.6, of 3000 4.5 / 4.2 and 6.0 / 5.6, of
// 8192 6.9 / 6.2 and 9.3 / 8.4, of 16384 11.2 / 9.3 (Step 3 had 32 there already); 148 of 8192 7.2 / 6.4 and 9.6 / 8.8; 200 of 3000
// 5.9 / 6.4 and 8.1 / 10.3, of 8192 9.5 / 11.8 and 14.3 / 15.9.
static bool regs_wide(int64_t n, int U) { return n > 2048 && U <= sm_count(); }

static vector_status launch_pool_select(const Dims& dm, const vector_budget* budget, const float* scores, int32_t* pool,
                                        cudaStream_t st, float* zero = nullptr) {
    vector_status rc = select_kernels_setup();
    if (rc != VECTOR_OK) return rc;
    const int64_t n = budget->n_tokens;
    const int nw = pool_select_warps(n, dm.U, budget->n_pool);
    if (nw == 0) {
        // Beyond 8192 elements lists that share multiprocessors come here, too, where they do not fit the blocks' shared memory.
        const bool wide = regs_wide(n, dm.U) || n > SEL_REGS16;
        auto kern = wide ? (n <= 4096 ? pool_select_regs<32, 4> : n <= 8192 ? pool_select_regs<32, 8> : n <= SEL_REGS16 ? pool_select_regs<32, 16>
                                                                                                                  : pool_select_regs<32, 32>)
                         : n <= 2048 ? pool_select_regs<16, 4> : n <= 4096 ? pool_select_regs<16, 8> : n <= 8192 ? pool_select_regs<16, 16>
                                                                                                                 : pool_select_regs<16, 32>;
        VEC_CUDA_CHECK(launch_maybe_dependent(true, kern, dim3(dm.U), dim3(wide ? 1024 : 512), 0, st, scores, n,
                                              (int)budget->n_pool, pool, zero));
        return VECTOR_OK;
    }
    const Layout L = selection_layout(n, nw);
    auto kern = nw == 8 ? pool_select_kernel<8> : nw == 16 ? pool_select_kernel<16> : pool_select_kernel<32>;
    VEC_CUDA_CHECK(launch_maybe_dependent(true, kern, dim3(dm.U), dim3(32 * nw), L.bytes(), st, scores, n, (int)budget->n_pool, pool, zero, L));
    return VECTOR_OK;
}

static vector_status launch_truncate(const Dims& dm, const vector_budget* budget, const float* eps, const int32_t* pool,
                                     uint8_t* tier, int32_t* ret_idx, int32_t* apx_idx, cudaStream_t st,
                                     bool dependent = false) {
    vector_status rc = select_kernels_setup();
    if (rc != VECTOR_OK) return rc;
    // dependent: may start (and clear the tier map) while the kernel before it in the stream drains
    const int64_t n = budget->n_pool;
    const int nw = truncate_warps(n, dm.U);
    if (nw == 0) {
        const bool wide = regs_wide(n, dm.U);           // beyond 8192 elements Step 3 takes registers for at most one list a multiprocessor only
        auto kern = wide ? (n <= 4096 ? truncate_regs<32, 4> : n <= 8192 ? truncate_regs<32, 8> : truncate_regs<32, 16>)
                         : n <= 2048 ? truncate_regs<16, 4> : n <= 4096 ? truncate_regs<16, 8> : truncate_regs<16, 16>;
        VEC_CUDA_CHECK(launch_maybe_dependent(dependent, kern, dim3(dm.U), dim3(wide ? 1024 : 512), 0, st, eps, pool,
                                              (int64_t)budget->n_tokens, (int)n, (int)budget->n_apx, tier, ret_idx, apx_idx));
        return VECTOR_OK;
    }
    const Layout L = selection_layout(n, nw);
    auto kern = nw == 8 ? truncate_kernel<8> : nw == 16 ? truncate_kernel<16> : truncate_kernel<32>;
    VEC_CUDA_CHECK(launch_maybe_dependent(dependent, kern, dim3(dm.U), dim3(32 * nw), L.bytes(), st, eps, pool, (int64_t)budget->n_tokens,
                                          (int)n, (int)budget->n_apx, tier, ret_idx, apx_idx, L));
    return VECTOR_OK;
}

// ---- one map per layer: a token's tier holds for all KV heads of its layer -----------------------
// Layer score of a token = the sum of its per-head base scores (window tokens stay +inf), summed in
// head order.  grid (ceil(N / 256), B L), 256 threads.
__global__ void __launch_bounds__(256)
layer_scores_kernel(const float* __restrict__ scores, int64_t N, int Hkv, float* __restrict__ layer_scores) {
    const int ul = blockIdx.y;
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= N) return;
    float s = 0.f;
    for (int h = 0; h < Hkv; ++h) s += scores[((size_t)ul * Hkv + h) * N + i];
    layer_scores[(size_t)ul * N + i] = s;
}

// Step 2 with one map per layer on CUDA cores (any dtype and head size): a warp per listed token,
// the token's keys of all heads in shared memory, lane = output channels lane, lane + 32, ...
// grid (ceil(n_idx / 8), B L), 256 threads, dynamic shared memory 8 * Hkv * D floats.
template <typename T, int D>
__global__ void __launch_bounds__(256)
residual_layer_generic(const T* __restrict__ K, const T* __restrict__ V, const T* __restrict__ W, int64_t N, int L,
                       int Hkv, const int32_t* __restrict__ idx, int n_idx, float* __restrict__ eps) {
    extern __shared__ float ksm[];
    const int ul = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int DL = Hkv * D;
    const int p = blockIdx.x * 8 + wid;
    if (p >= n_idx) return;
    const int64_t tok = idx[(size_t)ul * n_idx + p];
    if ((uint64_t)tok >= (uint64_t)N) {              // an index outside the unit reads as rows of zeros
        if (lane == 0) eps[(size_t)ul * n_idx + p] = 0.f;
        return;
    }
    float* kw = ksm + (size_t)wid * DL;
    for (int c = lane; c < DL; c += 32) kw[c] = to_f32(K[(((size_t)ul * Hkv + c / D) * N + tok) * D + c % D]);
    __syncwarp();
    const T* Wl = W + (size_t)(ul % L) * DL * DL;
    float e = 0.f;
    for (int co = lane; co < DL; co += 32) {
        const T* row = Wl + (size_t)co * DL;
        float pred = 0.f;
        for (int ci = 0; ci < DL; ++ci) pred = fmaf(to_f32(row[ci]), kw[ci], pred);
        const float r = to_f32(V[(((size_t)ul * Hkv + co / D) * N + tok) * D + co % D]) - pred;
        e = fmaf(r, r, e);
    }
    e = warp_sum(e);
    if (lane == 0) eps[(size_t)ul * n_idx + p] = e;
}

static vector_status residual_layer_dispatch(const Dims& dm, int Hkv, int L, const void* K, const void* V, const void* W,
                                             int64_t N, const int32_t* idx, int64_t n_idx, float* eps, cudaStream_t st,
                                             bool dependent, bool eps_zeroed) {
    if (n_idx == 0) return VECTOR_OK;
    const int UL = dm.U / Hkv;
    if (dm.dtype == VECTOR_BF16 && dm.d == 128) {
        static PerDeviceOnce once;
        if (once.first()) {
            auto opt_in = [](auto kern, int bytes) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
            cudaError_t e = opt_in(rlt::residual_layer_tc<true, 1>, rlt::LCfg<1>::SMEM_BYTES);
            if (e == cudaSuccess) e = opt_in(rlt::residual_layer_tc<false, 1>, rlt::LCfg<1>::SMEM_BYTES);
            if (e == cudaSuccess) e = opt_in(rlt::residual_layer_tc<true, 2>, rlt::LCfg<2>::SMEM_BYTES);
            if (e == cudaSuccess) e = opt_in(rlt::residual_layer_tc<false, 2>, rlt::LCfg<2>::SMEM_BYTES);
            if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
        }
        int* fault = kernel_fault_address();
        if (!fault) return VECTOR_ERR_CUDA;
        const uint64_t DL = (uint64_t)Hkv * 128;
        CUtensorMap mapW;
        if (!tma::encode_bf16_3d(&mapW, W, DL, DL, (uint64_t)L, DL * 2, DL * DL * 2, 64, 128)) return VECTOR_ERR_CUDA;
        rlt::Params P;
        P.UL = UL; P.L = L; P.Hkv = Hkv; P.n_idx = (int)n_idx; P.N = N;
        P.pairs = (Hkv + 1) / 2;
        const int sms = sm_count();
        // A tile of 128 tokens a block or of 256 a pair of blocks.  A group (block or pair) gets at least a tile, or exactly half of
        // one where that leaves no more groups than places.
        struct Split { int tpu; long long tiles; int groups; long long items; } split[2];
        for (int c = 0; c < 2; ++c) {
            Split& x = split[c];
            const long long places = sms / (c + 1), tokens = 128 * (c + 1);
            x.tpu = (int)((n_idx + tokens - 1) / tokens);
            x.tiles = (long long)UL * x.tpu;
            x.groups = (int)(x.tiles >= places ? places : 2 * x.tiles <= places && P.pairs > 1 ? 2 * x.tiles : x.tiles);
            x.items = (x.tiles * P.pairs + x.groups - 1) / x.groups;
        }
        // us: a pair of blocks takes Hkv items + 2, the 2 for a cluster's start and a stage's first fill by one warp, a block by itself 1.175
        // Hkv items; rounded to 256, a short list costs the pairs more items.  A call of pairs / blocks: 16 layers of 5000 tokens, 8 heads 150 /
        // 169, 4 heads 51 / 55, 3 heads 41 / 46; one layer of 300 tokens, 4 heads 14.0 / 12.6, 3 heads 13.1 / 11.9, one head 10.5 / 8.5; 37
        // layers of 700 tokens, 3 heads 18.0 / 17.8.  One and two heads leave the second block's half of the map short: 16 layers of 5000
        // tokens, one head 16.7 / 15.1, two heads 27.4 / 26.3.
        const bool pair = Hkv > 2 && 40 * Hkv * split[1].items + 80 <= 47 * Hkv * split[0].items;
        P.tpu = split[pair].tpu;
        P.n_items = split[pair].tiles * P.pairs;
        const int blocks = split[pair].groups * (pair ? 2 : 1);
        if (!eps_zeroed) VEC_CUDA_CHECK(cudaMemsetAsync(eps, 0, (size_t)UL * (size_t)n_idx * sizeof(float), st));
        const bool wide = ((uintptr_t)V & 31) == 0;
        auto kern = pair ? (wide ? rlt::residual_layer_tc<true, 2> : rlt::residual_layer_tc<false, 2>)
                         : (wide ? rlt::residual_layer_tc<true, 1> : rlt::residual_layer_tc<false, 1>);
        VEC_CUDA_CHECK(launch_maybe_dependent(dependent, pair ? 2 : 1, kern, dim3(blocks), dim3(pair ? rlt::LCfg<2>::THREADS : rlt::LCfg<1>::THREADS),
                                              pair ? rlt::LCfg<2>::SMEM_BYTES : rlt::LCfg<1>::SMEM_BYTES, st, (const __nv_bfloat16*)K,
                                              (const __nv_bfloat16*)V, mapW, idx, P, eps, fault));
        return VECTOR_OK;
    }
    const dim3 grid((unsigned)((n_idx + 7) / 8), UL);
    const size_t smem = (size_t)8 * Hkv * dm.d * sizeof(float);
#define VEC_RL(T, D)                                                                                                   \
    do {                                                                                                               \
        VEC_CUDA_CHECK(cudaFuncSetAttribute(residual_layer_generic<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                            (int)smem));                                                               \
        residual_layer_generic<T, D><<<grid, 256, smem, st>>>((const T*)K, (const T*)V, (const T*)W, N, L, Hkv, idx,   \
                                                              (int)n_idx, eps);                                        \
    } while (0)
    if (dm.dtype == VECTOR_F32) { if (dm.d == 64) VEC_RL(float, 64); else VEC_RL(float, 128); }
    else { if (dm.d == 64) VEC_RL(__nv_bfloat16, 64); else VEC_RL(__nv_bfloat16, 128); }
#undef VEC_RL
    VEC_LAUNCH_CHECK();
    return VECTOR_OK;
}

}  // namespace vec

using namespace vec;

extern "C" vector_status vector_pool_select(const vector_shape* shape, const vector_budget* budget,
                                            const float* scores, int32_t* pool_idx, void* ws, size_t ws_bytes,
                                            void* stream) {
    (void)ws; (void)ws_bytes;
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if ((rc = check_budget(budget, dm.w)) != VECTOR_OK) return rc;
    if (!scores || !pool_idx) return VECTOR_ERR_NULL;
    return launch_pool_select(dm, budget, scores, pool_idx, (cudaStream_t)stream);
}

extern "C" vector_status vector_residual(const vector_shape* shape, const void* K, const void* V, const void* W,
                                         int64_t N, const int32_t* idx, int64_t n_idx, float* eps, void* stream) {
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if (!K || !V || !W || !idx || !eps) return VECTOR_ERR_NULL;
    if (N <= 0 || N > (int64_t(1) << 30) || n_idx < 0 || n_idx > N) return VECTOR_ERR_SHAPE;
    return residual_dispatch(dm, K, V, W, N, idx, n_idx, eps, (cudaStream_t)stream);
}

extern "C" vector_status vector_truncate(const vector_shape* shape, const vector_budget* budget, const float* eps,
                                         const int32_t* pool_idx, uint8_t* tier, int32_t* ret_idx,
                                         int32_t* apx_idx, void* ws, size_t ws_bytes, void* stream) {
    (void)ws; (void)ws_bytes;
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if ((rc = check_budget(budget, dm.w)) != VECTOR_OK) return rc;
    if (!eps || !pool_idx || !tier) return VECTOR_ERR_NULL;
    if ((budget->n_ret > 0 && !ret_idx) || (budget->n_apx > 0 && !apx_idx)) return VECTOR_ERR_NULL;
    return launch_truncate(dm, budget, eps, pool_idx, tier, ret_idx, apx_idx, (cudaStream_t)stream);
}

extern "C" vector_status vector_route(const vector_shape* shape, const vector_budget* budget, const float* scores,
                                      const void* K, const void* V, const void* W, uint8_t* tier,
                                      int32_t* ret_idx, int32_t* apx_idx, float* eps_out, int32_t* pool_idx_out,
                                      void* ws, size_t ws_bytes, void* stream) {
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if ((rc = check_budget(budget, dm.w)) != VECTOR_OK) return rc;
    if (!scores || !K || !V || !W || !tier) return VECTOR_ERR_NULL;
    if ((budget->n_ret > 0 && !ret_idx) || (budget->n_apx > 0 && !apx_idx)) return VECTOR_ERR_NULL;
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < select_ws_bytes(dm, *budget)) return VECTOR_ERR_WORKSPACE;
    char* p = (char*)ws;
    int32_t* pool = pool_idx_out ? pool_idx_out : (int32_t*)p;
    p += align256((size_t)dm.U * (size_t)budget->n_pool * sizeof(int32_t));
    float* eps = eps_out ? eps_out : (float*)p;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = launch_pool_select(dm, budget, scores, pool, st)) != VECTOR_OK) return rc;
    rc = residual_dispatch(dm, K, V, W, budget->n_tokens, pool, budget->n_pool, eps, st, true);
    if (rc != VECTOR_OK) return rc;
    return launch_truncate(dm, budget, eps, pool, tier, ret_idx, apx_idx, st, true);
}

extern "C" vector_status vector_layer_scores(const vector_shape* shape, const float* scores, int64_t N,
                                             float* layer_scores, void* stream) {
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if (!scores || !layer_scores) return VECTOR_ERR_NULL;
    if (N <= 0 || N > (int64_t(1) << 30)) return VECTOR_ERR_SHAPE;
    const int Hkv = shape->n_kv_heads;
    const dim3 grid((unsigned)((N + 255) / 256), dm.U / Hkv);
    layer_scores_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(scores, N, Hkv, layer_scores);
    VEC_LAUNCH_CHECK();
    return VECTOR_OK;
}

extern "C" vector_status vector_residual_layer(const vector_shape* shape, const void* K, const void* V, const void* W_layer,
                                               int64_t N, const int32_t* idx, int64_t n_idx, float* eps, void* stream) {
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if (!K || !V || !W_layer || !idx || !eps) return VECTOR_ERR_NULL;
    if (N <= 0 || N > (int64_t(1) << 30) || n_idx < 0 || n_idx > N) return VECTOR_ERR_SHAPE;
    if (dm.rope) return VECTOR_ERR_UNSUPPORTED;
    return residual_layer_dispatch(dm, shape->n_kv_heads, shape->n_layers, K, V, W_layer, N, idx, n_idx, eps,
                                   (cudaStream_t)stream, false, false);
}

extern "C" vector_status vector_route_layer(const vector_shape* shape, const vector_budget* budget, const float* layer_scores,
                                            const void* K, const void* V, const void* W_layer, uint8_t* tier,
                                            int32_t* ret_idx, int32_t* apx_idx, float* eps_out, int32_t* pool_idx_out,
                                            void* ws, size_t ws_bytes, void* stream) {
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if ((rc = check_budget(budget, dm.w)) != VECTOR_OK) return rc;
    if (!layer_scores || !K || !V || !W_layer || !tier) return VECTOR_ERR_NULL;
    if ((budget->n_ret > 0 && !ret_idx) || (budget->n_apx > 0 && !apx_idx)) return VECTOR_ERR_NULL;
    if (dm.rope) return VECTOR_ERR_UNSUPPORTED;
    const int Hkv = shape->n_kv_heads;
    Dims dl = dm;                       // the selections run per (sequence, layer)
    dl.U = dm.U / Hkv;
    const size_t need = align256((size_t)dl.U * (size_t)budget->n_pool * sizeof(int32_t)) +
                        align256((size_t)dl.U * (size_t)budget->n_pool * sizeof(float));
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < need) return VECTOR_ERR_WORKSPACE;
    char* p = (char*)ws;
    int32_t* pool = pool_idx_out ? pool_idx_out : (int32_t*)p;
    p += align256((size_t)dl.U * (size_t)budget->n_pool * sizeof(int32_t));
    float* eps = eps_out ? eps_out : (float*)p;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = launch_pool_select(dl, budget, layer_scores, pool, st, eps)) != VECTOR_OK) return rc;      // zeroes eps as well
    rc = residual_layer_dispatch(dm, Hkv, shape->n_layers, K, V, W_layer, budget->n_tokens, pool, budget->n_pool, eps, st, true, true);
    if (rc != VECTOR_OK) return rc;
    return launch_truncate(dl, budget, eps, pool, tier, ret_idx, apx_idx, st, true);
}
