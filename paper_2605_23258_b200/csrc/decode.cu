// Generation-time attention over the mixed cache (paper Section 3.2, Step 3):
// one softmax over the exact keys of the retained and the key-only pool; a
// retained token contributes its stored value, an approximated token W k.
// Factored form: o = sum_R p_i v_i + W (sum_A p_i k_i), so the kernel streams
// both pools once, accumulating p-weighted values and p-weighted keys, and the
// d x d map is applied once per query head in the merge step.
//
// bf16 runs the kernels of decode_bf16.cuh and decode_pertile_tc.cuh; below, for fp32 (and 64-channel bf16 rows off a
// 16-byte boundary), one launch: a thread block cluster per unit, its blocks a slice each of the logical key range
// [0, n_ret + n_apx); the blocks' sums are merged over distributed shared memory.
#include <cmath>
#include <mutex>
#include <type_traits>

#include "cluster.cuh"
#include "common.cuh"
#include "decode_bf16.cuh"
#include "decode_pertile_tc.cuh"
#include "decode_rope.cuh"
#include "internal.h"

namespace vec {

// EPL consecutive elements of a row; WIDE: fp32 rows at multiples of 16 bytes, otherwise one by one.
template <bool WIDE, int EPL, typename T>
__device__ __forceinline__ void row_load(const T* p, int lane, float (&o)[EPL]) {
    if constexpr (WIDE) {
        if constexpr (EPL == 4) {
            const float4 v = reinterpret_cast<const float4*>(p)[lane];
            o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
        } else {
            const float2 v = reinterpret_cast<const float2*>(p)[lane];
            o[0] = v.x; o[1] = v.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < EPL; ++e) o[e] = to_f32(p[lane * EPL + e]);
    }
}

// Record of a warp or a block, per head: m, l, pad, acc_v[D], acc_k[D].
template <int D> struct Rec { static constexpr int floats = 4 + 2 * D; };
constexpr int F32_WARPS = 8, F32_ROWS = 4, F32_MAX_CLUSTER = 16;

// A warp takes four rows at a time, a row across its lanes: the loads and the dot products' reductions of the four are
// independent, where one row at a time left a chain of load, five shuffles and two exponentials per row and head (2 units of
// 2 heads and 384 rows: 43 us, and 12 us for a merge kernel of two blocks).
// With ROPE the approximated value is W applied to the key turned back by its original position
// (apx_pos): the logit still uses the stored key, only the p-weighted key sum takes the turned one.
// A lane holds EPL consecutive channels; the partner channel c +- D/2 sits in lane ^ 16.
// grid (U x cluster size), 256 threads, F32_WARPS * g records of dynamic shared memory.
template <typename T, int D, int G, bool ROPE, bool WIDE>
__global__ void __launch_bounds__(32 * F32_WARPS)
decode_rows(const T* q, const T* ret_k, const T* ret_v, const T* apx_k,
           const int32_t* apx_pos, int64_t cap_ret, int64_t cap_apx, int n_ret, int n_apx, int g, int LH, float scale,
           float theta, const T* W, void* __restrict__ out, int out_bf16) {
    constexpr int EPL = D / 32, REC = Rec<D>::floats, NT = 32 * F32_WARPS;
    extern __shared__ __align__(16) float recs[];               // [F32_WARPS][g][REC]
    __shared__ __align__(16) float comb[G][REC];                // this block's sums, read by the whole cluster
    __shared__ __align__(16) float aks[G][D];                   // merged key sums of this block's heads, and their value sums
    __shared__ float avs[G][D], fac[G][F32_MAX_CLUSTER], Ls[G];
    __shared__ double inv_freq[ROPE ? D / 2 : 1];
    if (ROPE) { rope_fill_inv_freq(inv_freq, D, theta); __syncthreads(); }
    // a programmatic dependent of what precedes it; nothing of its inputs is touched before this
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int C = (int)cl::nctas(), rank = (int)cl::rank(), u = blockIdx.x / C;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int total = n_ret + n_apx;
    const int lo = (int)((long long)rank * total / C), hi = (int)((long long)(rank + 1) * total / C);

    float qr[G][EPL], av[G][EPL], ak[G][EPL], m[G], l[G];
#pragma unroll
    for (int a = 0; a < G; ++a) {
        m[a] = -INFINITY;
        l[a] = 0.f;
#pragma unroll
        for (int e = 0; e < EPL; ++e) { av[a][e] = 0.f; ak[a][e] = 0.f; qr[a][e] = 0.f; }
        if (a < g) {
            row_load<WIDE>(q + ((size_t)u * g + a) * D, lane, qr[a]);
#pragma unroll
            for (int e = 0; e < EPL; ++e) qr[a][e] *= scale;
        }
    }
    for (int i0 = lo + wid; i0 < hi; i0 += F32_ROWS * F32_WARPS) {
        float kx[F32_ROWS][EPL], vx[F32_ROWS][EPL], kt[F32_ROWS][EPL];        // kt: what an approximated token contributes
#pragma unroll
        for (int r = 0; r < F32_ROWS; ++r) {
            const int i = i0 + r * F32_WARPS;
#pragma unroll
            for (int e = 0; e < EPL; ++e) { kx[r][e] = 0.f; vx[r][e] = 0.f; }
            if (i < hi) {
                row_load<WIDE>(i < n_ret ? ret_k + ((size_t)u * cap_ret + i) * D : apx_k + ((size_t)u * cap_apx + (i - n_ret)) * D, lane, kx[r]);
                if (i < n_ret) row_load<WIDE>(ret_v + ((size_t)u * cap_ret + i) * D, lane, vx[r]);
            }
        }
#pragma unroll
        for (int r = 0; r < F32_ROWS; ++r) {
            const int i = i0 + r * F32_WARPS;
            const bool apx = i < hi && i >= n_ret;
#pragma unroll
            for (int e = 0; e < EPL; ++e) kt[r][e] = apx ? kx[r][e] : 0.f;
            if (ROPE && apx) {
                const double pos = (double)apx_pos[(size_t)u * cap_apx + (i - n_ret)];
#pragma unroll
                for (int e = 0; e < EPL; ++e) {
                    float cs, sn;
                    rope_cos_sin(pos, inv_freq[(lane * EPL + e) % (D / 2)], cs, sn);
                    const float other = __shfl_xor_sync(0xffffffffu, kx[r][e], 16);
                    kt[r][e] = lane < 16 ? fmaf(kx[r][e], cs, other * sn) : fmaf(kx[r][e], cs, -other * sn);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < G; ++a) {
            if (a < g) {
                float s[F32_ROWS];
#pragma unroll
                for (int r = 0; r < F32_ROWS; ++r) {
                    s[r] = 0.f;
#pragma unroll
                    for (int e = 0; e < EPL; ++e) s[r] = fmaf(qr[a][e], kx[r][e], s[r]);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int r = 0; r < F32_ROWS; ++r) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
                float mn = m[a];
#pragma unroll
                for (int r = 0; r < F32_ROWS; ++r) {
                    if (i0 + r * F32_WARPS >= hi) s[r] = -INFINITY;
                    mn = fmaxf(mn, s[r]);                       // finite: row i0 is valid
                }
                const float corr = __expf(m[a] - mn);           // first rows: exp(-inf) = 0
                m[a] = mn;
                l[a] *= corr;
#pragma unroll
                for (int e = 0; e < EPL; ++e) { av[a][e] *= corr; ak[a][e] *= corr; }
#pragma unroll
                for (int r = 0; r < F32_ROWS; ++r) {
                    const float p = __expf(s[r] - mn);
                    l[a] += p;
#pragma unroll
                    for (int e = 0; e < EPL; ++e) { av[a][e] = fmaf(p, vx[r][e], av[a][e]); ak[a][e] = fmaf(p, kt[r][e], ak[a][e]); }
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < G; ++a) {
        if (a < g) {
            float* r = recs + (wid * g + a) * REC;
            if (lane == 0) { r[0] = m[a]; r[1] = l[a]; }
#pragma unroll
            for (int e = 0; e < EPL; ++e) { r[4 + lane * EPL + e] = av[a][e]; r[4 + D + lane * EPL + e] = ak[a][e]; }
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < g * 2 * D; e += NT) {         // the block's sums
        const int a = e / (2 * D), c = e % (2 * D);
        float M = -INFINITY, L = 0.f, v = 0.f;
#pragma unroll
        for (int w = 0; w < F32_WARPS; ++w) M = fmaxf(M, recs[(w * g + a) * REC]);
#pragma unroll
        for (int w = 0; w < F32_WARPS; ++w) {
            const float* r = recs + (w * g + a) * REC;
            const float f = r[0] > -INFINITY ? __expf(r[0] - M) : 0.f;
            L = fmaf(f, r[1], L);
            v = fmaf(f, r[4 + c], v);
        }
        if (c == 0) { comb[a][0] = M; comb[a][1] = L; }
        comb[a][4 + c] = v;
    }
    // the map, a row across a warp's lanes, requested before the cluster's barrier
    constexpr int ROWS = D / F32_WARPS;
    const T* Wu = W + (size_t)(u % LH) * D * D;
    float wr[ROWS][EPL];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) row_load<WIDE>(Wu + (size_t)(r * F32_WARPS + wid) * D, lane, wr[r]);
    cl::arrive_release();
    cl::wait_acquire();                                         // every block's sums are ready
    const int mine = rank < g ? (g - rank + C - 1) / C : 0;     // this block merges heads rank, rank + C, ...
    for (int k = wid; k < mine; k += F32_WARPS) {
        const int a = rank + k * C;
        float mj = -INFINITY, lj = 0.f;
        if (lane < C) {
            const uint32_t at = cl::map_to(tma::smem_u32(&comb[a][0]), (uint32_t)lane);
            mj = cl::ld_f32(at);
            lj = cl::ld_f32(at + 4);
        }
        const float M = warp_max(mj);
        const float f = mj > -INFINITY ? __expf(mj - M) : 0.f;
        const float L = warp_sum(f * lj);
        if (lane < C) fac[k][lane] = f;
        if (lane == 0) Ls[k] = L;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < mine * 2 * D; e += NT) {
        const int k = e / (2 * D), c = e % (2 * D);
        const uint32_t at = tma::smem_u32(&comb[rank + k * C][4 + c]);
        float v = 0.f;
        for (int j0 = 0; j0 < C; j0 += 8) {                     // eight remote loads in flight
            float x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = cl::ld_f32(cl::map_to(at, (uint32_t)min(j0 + j, C - 1)));
#pragma unroll
            for (int j = 0; j < 8; ++j) v = fmaf(j0 + j < C ? fac[k][j0 + j] : 0.f, x[j], v);
        }
        if (c < D) avs[k][c] = v;
        else aks[k][c - D] = v;
    }
    cl::arrive_release();                                       // this block reads no other block's memory from here on
    __syncthreads();
    for (int k = 0; k < mine; ++k) {
        float a[EPL];
        row_load<true>(aks[k], lane, a);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            float x = 0.f;
#pragma unroll
            for (int e = 0; e < EPL; ++e) x = fmaf(wr[r][e], a[e], x);
            x = warp_sum(x);
            const int c = r * F32_WARPS + wid;
            const size_t at = ((size_t)u * g + rank + k * C) * D + c;
            const float o = (avs[k][c] + x) / Ls[k];
            if (lane == 0) {
                if (out_bf16) reinterpret_cast<__nv_bfloat16*>(out)[at] = __float2bfloat16_rn(o);
                else reinterpret_cast<float*>(out)[at] = o;
            }
        }
    }
    __syncwarp();
    cl::wait_acquire();                                         // nobody reads this block's memory any more
}

static bool rows_at_16_bytes(const void* q, const vector_cache* ch, const void* W) {
    uintptr_t all = (uintptr_t)q | (uintptr_t)W;
    if (ch->n_ret > 0) all |= (uintptr_t)ch->ret_k | (uintptr_t)ch->ret_v;
    if (ch->n_apx > 0) all |= (uintptr_t)ch->apx_k;
    return (all & 15) == 0;
}

template <typename T, int D, int G, bool ROPE, bool WIDE>
static vector_status launch_decode_rows(const Dims& dm, const void* q, const vector_cache* ch, const void* W, void* out,
                                       int out_dtype, cudaStream_t st) {
    auto kern = decode_rows<T, D, G, ROPE, WIDE>;
    static PerDeviceOnce once;
    if (once.first()) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, F32_WARPS * G * Rec<D>::floats * 4);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
    }
    // blocks a unit: one pass over the rows of a block's warps at the least, four blocks a multiprocessor at the most
    const int64_t rows = ch->n_ret + ch->n_apx;
    int64_t c = (rows + F32_ROWS * F32_WARPS - 1) / (F32_ROWS * F32_WARPS);
    const int64_t fill = (4 * (int64_t)sm_count() + dm.U - 1) / dm.U;
    if (c > fill) c = fill;
    if (c > F32_MAX_CLUSTER) c = F32_MAX_CLUSTER;
    if (c > 8 && c < F32_MAX_CLUSTER) c = 8;                    // beyond the portable size only the largest
    VEC_CUDA_CHECK(launch_maybe_dependent(true, (int)c, kern, dim3((unsigned)(c * dm.U)), dim3(32 * F32_WARPS),
                                          (size_t)F32_WARPS * dm.g * Rec<D>::floats * 4, st, (const T*)q, (const T*)ch->ret_k,
                                          (const T*)ch->ret_v, (const T*)ch->apx_k, ch->apx_pos, ch->cap_ret, ch->cap_apx,
                                          (int)ch->n_ret, (int)ch->n_apx, dm.g, dm.LH, dm.scale, dm.theta, (const T*)W, out,
                                          out_dtype == VECTOR_BF16 ? 1 : 0));
    return VECTOR_OK;
}

// Fault word that bounded waits inside kernels write to (0 = none).
static __device__ int g_kernel_fault;
int* kernel_fault_address() {
    static int* addr[PerDeviceOnce::kMax] = {};      // per device, looked up with that device current
    static std::mutex mu;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= PerDeviceOnce::kMax) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_kernel_fault) == cudaSuccess) addr[dev] = (int*)p;
    }
    return addr[dev];
}

// Blocks per unit of the one-launch (cluster) form, 0 = stream and merge.  A cluster lies within one GPC and every
// block fills its multiprocessor, so the largest size is taken at which all U clusters are resident at once.  That may
// use fewer multiprocessors than the streaming form (48 units would need clusters of three that fit), whose second
// kernel and records in global memory cost as much as some tiles of a block: more of 64 channels, which are half
// the size, and fewer with RoPE, whose tiles take longer.  The form with the fewer tiles a block, that cost included, runs.
// Measured, four query heads, us per step in a graph, cluster against stream: 128 channels, 8 units of 2457 rows 9.4 / 12.5,
// of 19660 rows 22.5 / 25.4; 48 units of 1200 rows 13.5 / 16.1, 2457 rows 18.5 / 19.5, 4800 rows 26.6 / 24.8, with RoPE 15.6 /
// 19.1, 23.7 / 23.8, 37.7 / 32.8; 64 channels, 48 units of 4800 rows 18.1 / 20.1, 7200 rows 23.3 / 23.4, with RoPE 1200 rows 16.9 /
// 21.2, 2457 rows 27.7 / 27.1, 4800 rows 45.2 / 38.2.
template <int D, bool ROPE>
static int decode_cluster_size(const dbf::Plan& pl, int U) {
    using C = dbf::Cfg<D, ROPE>;
    constexpr int MAXC = dbf::MAX_CLUSTER, EXTRA_TILES = D == 128 ? (ROPE ? 6 : 9) : ROPE ? 2 : 13;
    static int resident[PerDeviceOnce::kMax][MAXC + 1] = {};      // clusters of each size the device holds at once
    static std::mutex mu;
    int dev = -1;
    if (2 * U > sm_count() || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= PerDeviceOnce::kMax) return 0;
    std::lock_guard<std::mutex> lock(mu);
    int* r = resident[dev];
    if (r[0] == 0) {
        auto kern = [] { if constexpr (ROPE) return dbf::decode_stream_rope<D, true>; else return dbf::decode_stream_bf16<D, true>; }();
        bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::CLUSTER_SMEM_BYTES) == cudaSuccess &&
                  cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        for (int c = 2; ok && c <= MAXC; ++c) {
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = c; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(c); cfg.blockDim = dim3(C::THREADS); cfg.dynamicSmemBytes = C::CLUSTER_SMEM_BYTES;
            cfg.attrs = &attr; cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess) r[c] = n;
        }
        (void)cudaGetLastError();                                  // a size the device refuses counts as none resident
        r[0] = 1;
    }
    for (int c = pl.n_tiles < MAXC ? pl.n_tiles : MAXC; c >= 2; --c)
        if (r[c] >= U) return (pl.n_tiles + c - 1) / c <= (int)((pl.T + pl.B - 1) / pl.B) + EXTRA_TILES ? c : 0;
    return 0;
}

// bf16: persistent TMA + tensor-core streaming kernel and the record merge.
template <int D>
static vector_status launch_decode_bf16(const Dims& dm, const void* q, const vector_cache* ch, const void* W,
                                        void* out, int out_dtype, int mode, float* partial, cudaStream_t st) {
    using T = __nv_bfloat16;
    using Plain = dbf::Cfg<D, false>;
    using Rope = dbf::Cfg<D, true>;
    static PerDeviceOnce once;
    if (once.first()) {
        cudaError_t e = cudaFuncSetAttribute(dbf::decode_stream_bf16<D, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, Plain::SMEM_BYTES);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(dbf::decode_stream_rope<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     Rope::SMEM_BYTES);
        if (D == 128 && e == cudaSuccess)
            e = cudaFuncSetAttribute(dpt::decode_stream_pertile_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, dpt::SMEM_BYTES);
        if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
    }
    int* fault = kernel_fault_address();
    if (!fault) return VECTOR_ERR_CUDA;
    const dbf::Plan pl = dbf::make_plan(dm.U, ch->n_ret, ch->n_apx, sm_count());
    if (pl.s_max > decode_stream_slots(dm.U)) return VECTOR_ERR_WORKSPACE;
    dbf::Maps maps;
    const uint64_t row_b = 2 * D;
    bool ok = true;
    if (ch->n_ret > 0) {
        ok = ok && tma::encode_bf16_3d(&maps.ret_k, ch->ret_k, D, (uint64_t)ch->n_ret, (uint64_t)dm.U, row_b,
                                       (uint64_t)ch->cap_ret * row_b, 64, 64);
        ok = ok && tma::encode_bf16_3d(&maps.ret_v, ch->ret_v, D, (uint64_t)ch->n_ret, (uint64_t)dm.U, row_b,
                                       (uint64_t)ch->cap_ret * row_b, 64, 64);
    }
    if (ch->n_apx > 0)
        ok = ok && tma::encode_bf16_3d(&maps.apx_k, ch->apx_k, D, (uint64_t)ch->n_apx, (uint64_t)dm.U, row_b,
                                       (uint64_t)ch->cap_apx * row_b, 64, 64);
    if (!ok) return VECTOR_ERR_CUDA;
    if (ch->n_ret == 0) { maps.ret_k = maps.apx_k; maps.ret_v = maps.apx_k; }   // never dereferenced: no such tiles
    if (ch->n_apx == 0) maps.apx_k = maps.ret_k;
    const float c2 = dm.scale * 1.4426950408889634f;
    RopePhases ph = {};
    if (dm.rope) rope_phases(dm.theta, D, &ph);
    if (D == 128 && mode == 1) {
        // reconstruction tile by tile on the tensor cores: its own streaming kernel, two consumer warps
        dpt::Maps pm;
        pm.ret_k = maps.ret_k; pm.ret_v = maps.ret_v; pm.apx_k = maps.apx_k;
        if (!tma::encode_bf16_3d(&pm.w, W, 128, 128, (uint64_t)dm.LH, row_b, 128 * row_b, 64, 128)) return VECTOR_ERR_CUDA;
        if (ch->n_apx > 0 && !tma::encode_bf16_3d(&pm.apx_k, ch->apx_k, 128, (uint64_t)ch->n_apx, (uint64_t)dm.U, row_b,
                                                  (uint64_t)ch->cap_apx * row_b, 64, 128))
            return VECTOR_ERR_CUDA;
        dpt::decode_stream_pertile_tc<<<pl.B, dpt::THREADS, dpt::SMEM_BYTES, st>>>(
            (const T*)q, pm, pl, (int)ch->n_ret, (int)ch->n_apx, dm.g, dm.LH, c2, partial, fault);
        VEC_LAUNCH_CHECK();
    } else {
        const T* qp = (const T*)q;
        const T* Wq = (const T*)W;
        const int n_ret = (int)ch->n_ret, n_apx = (int)ch->n_apx, out_f32 = out_dtype == VECTOR_F32;
        const int csize = dm.rope ? decode_cluster_size<D, true>(pl, dm.U) : decode_cluster_size<D, false>(pl, dm.U);
        const dim3 grid(csize ? csize * dm.U : pl.B);
        const int cl = csize ? csize : 1;
        if (dm.rope) {
            auto kern = csize ? dbf::decode_stream_rope<D, true> : dbf::decode_stream_rope<D, false>;
            VEC_CUDA_CHECK(launch_maybe_dependent(true, cl, kern, grid, dim3(Rope::THREADS), csize ? Rope::CLUSTER_SMEM_BYTES : Rope::SMEM_BYTES,
                                                  st, qp, maps, pl, n_ret, n_apx, dm.g, dm.LH, c2, partial, fault, ch->apx_pos,
                                                  (long long)ch->cap_apx, ph, Wq, out, out_f32));
        } else {
            auto kern = csize ? dbf::decode_stream_bf16<D, true> : dbf::decode_stream_bf16<D, false>;
            VEC_CUDA_CHECK(launch_maybe_dependent(true, cl, kern, grid, dim3(Plain::THREADS), csize ? Plain::CLUSTER_SMEM_BYTES : Plain::SMEM_BYTES,
                                                  st, qp, maps, pl, n_ret, n_apx, dm.g, dm.LH, c2, partial, fault, Wq, out, out_f32));
        }
        if (csize) return VECTOR_OK;
    }
    // programmatic dependent launch: the merge blocks start while the streaming kernel drains
    const float* rec = partial;
    const int apply_w = mode == 1 ? 0 : 1;
    const int cw = mode == 1 ? dpt::CONSUMERS : dm.rope ? Rope::CONSUMER_WARPS : Plain::CONSUMER_WARPS;   // records a block leaves per unit
    const T* Wp = (const T*)W;
    // The form by units a multiprocessor (`full`, rounded up).  A block a unit with everything requested ahead is the fastest while all units' blocks are
    // resident at once; registers decide how many are.  us of a whole step in a graph, one sequence, 96 / 600 / 1800 rows a unit:
    //   128 channels, two heads, 592 units: four blocks of 128 threads 17.2 / 31.5 / 65.4, ranges by three of 256 threads 21.3 / 35.5 / 69.2, a thread
    //   a channel 19.3 / 35.5 / 69.7; 740 units, five blocks: 20.3 / 39.5 / 81.1 (22.8 / 41.9 / 83.6, 20.9 / 41.5 / 83.9); 900 units, a thread a channel
    //   25.3 / 48.2 / 96.9, ranges 28.8 / 50.5 / 99.1; 4096 units of one head and 96 / 600 rows 84.6 / 183 and 100 / 197.
    //   Three heads: 440 units, three blocks 14.6 / 26.7 / 49.1 (ranges by two 16.7 / 28.7 / 51.0, a thread a channel 16.2 / 29.1 / 51.9); 900 units,
    //   a thread a channel 27.2 / 49.8 / 99.2, ranges 29.1 / 50.9 / 100.2.
    //   Four heads: 440 units, three blocks 14.9 / 27.0 / 49.9 (ranges by two 16.8 / 29.3 / 51.6); 900 units, ranges 29.0 / 52.0 / 101.6, a thread a channel
    //   30.3 / 53.4 / 103.3.  Ranges go on paying where sequences share maps: 2048 units of eight sequences 0.95 to 0.98 of a thread a channel.
    //   64 channels: 740 units of four heads, a block a unit with seven resident 14.9 / 26.8 / 49.3, ranges by four 17.0 / 29.1 / 50.5; 1280 units of
    //   two heads, a block a unit 20.5 / 41.7 / 80.1, ranges 23.4 / 44.5 / 83.1.
    // More than four heads take a block a unit at any number of units.
    const int full = (dm.U + sm_count() - 1) / sm_count();
    auto merge = [&](auto* o) -> vector_status {
        using TO = std::remove_pointer_t<decltype(o)>;
        auto launch = [&](auto kern, int blocks, int threads) -> vector_status {
            VEC_CUDA_CHECK(launch_maybe_dependent(true, kern, dim3(blocks), dim3(threads), 0, st, rec, Wp, dm.LH, dm.U, dm.g, pl, apply_w, cw, o));
            return VECTOR_OK;
        };
#define VEC_MERGE(HEADS, RES) \
    return launch(dbf::decode_merge_bf16<TO, D, HEADS, RES>, dbf::MergeCfg<D, HEADS, RES>::blocks(dm.U, sm_count()), dbf::MergeCfg<D, HEADS, RES>::THREADS)
        if constexpr (D == 128) {
            if (dm.g <= 2 && full <= 4) VEC_MERGE(2, 4);
            if (dm.g <= 2 && full <= 5) VEC_MERGE(2, 5);
            if (dm.g <= 3 && full > 3) return launch(dbf::decode_merge_channels<TO, D>, dm.U, D * dm.g);
            if (dm.g <= 4 && full == 3) VEC_MERGE(4, 3);
            if (dm.g <= 4) VEC_MERGE(4, 2);
            VEC_MERGE(8, 2);
        } else {
            if (dm.g <= 2) VEC_MERGE(2, 8);
            if (dm.g <= 4 && full > 4) VEC_MERGE(4, 7);
            if (dm.g <= 4) VEC_MERGE(4, 4);
            VEC_MERGE(8, 4);
        }
#undef VEC_MERGE
    };
    return out_dtype == VECTOR_F32 ? merge((float*)out) : merge((T*)out);
}

template <typename T, int D, bool ROPE, bool WIDE>
static vector_status launch_decode_g(const Dims& dm, const void* q, const vector_cache* ch, const void* W, void* out, int out_dtype,
                                     cudaStream_t st) {
    if (dm.g <= 2) return launch_decode_rows<T, D, 2, ROPE, WIDE>(dm, q, ch, W, out, out_dtype, st);
    if (dm.g <= 4) return launch_decode_rows<T, D, 4, ROPE, WIDE>(dm, q, ch, W, out, out_dtype, st);
    return launch_decode_rows<T, D, 8, ROPE, WIDE>(dm, q, ch, W, out, out_dtype, st);
}

}  // namespace vec

using namespace vec;

extern "C" vector_status vector_decode_attn(const vector_shape* shape, const void* q, const vector_cache* cache,
                                            const void* W, void* out, int32_t out_dtype, int32_t mode, void* ws,
                                            size_t ws_bytes, void* stream) {
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if (!q || !cache || !W || !out) return VECTOR_ERR_NULL;
    if (out_dtype != VECTOR_F32 && out_dtype != VECTOR_BF16) return VECTOR_ERR_DTYPE;
    if (mode != 0 && mode != 1) return VECTOR_ERR_SHAPE;
    if (cache->n_ret < 0 || cache->n_apx < 0 || cache->n_ret + cache->n_apx <= 0 ||
        cache->n_ret + cache->n_apx > (int64_t(1) << 30) || cache->cap_ret < cache->n_ret ||
        cache->cap_apx < cache->n_apx)
        return VECTOR_ERR_SHAPE;
    if (cache->n_ret > 0 && (!cache->ret_k || !cache->ret_v)) return VECTOR_ERR_NULL;
    if (cache->n_apx > 0 && !cache->apx_k) return VECTOR_ERR_NULL;
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < decode_ws_bytes(dm)) return VECTOR_ERR_WORKSPACE;
    // per-tile reconstruction exists for bf16 with head_dim 128 and stored (not rotated-back) keys
    if (mode == 1 && (dm.rope || dm.dtype != VECTOR_BF16 || dm.d != 128)) return VECTOR_ERR_UNSUPPORTED;
    if (dm.rope && cache->n_apx > 0 && !cache->apx_pos) return VECTOR_ERR_NULL;
    cudaStream_t st = (cudaStream_t)stream;
    float* partial = (float*)ws;
    // Rows off a 16-byte boundary: element by element, 64-channel bf16 ones, which TMA would refuse, on the CUDA-core kernel too
    const bool wide = rows_at_16_bytes(q, cache, W);
    if (dm.dtype == VECTOR_F32) {
        auto launch = dm.d == 64 ? (dm.rope ? (wide ? launch_decode_g<float, 64, true, true> : launch_decode_g<float, 64, true, false>)
                                            : (wide ? launch_decode_g<float, 64, false, true> : launch_decode_g<float, 64, false, false>))
                                 : (dm.rope ? (wide ? launch_decode_g<float, 128, true, true> : launch_decode_g<float, 128, true, false>)
                                            : (wide ? launch_decode_g<float, 128, false, true> : launch_decode_g<float, 128, false, false>));
        return launch(dm, q, cache, W, out, out_dtype, st);
    }
    if (dm.d == 64 && !wide)
        return dm.rope ? launch_decode_g<__nv_bfloat16, 64, true, false>(dm, q, cache, W, out, out_dtype, st)
                       : launch_decode_g<__nv_bfloat16, 64, false, false>(dm, q, cache, W, out, out_dtype, st);
    if (dm.d == 64) return launch_decode_bf16<64>(dm, q, cache, W, out, out_dtype, mode, partial, st);
    return launch_decode_bf16<128>(dm, q, cache, W, out, out_dtype, mode, partial, st);
}

// ---------------------------------------------------------------------------
// Allocation-free variant: the split-KV partial records live in a fixed array
// of the library's device image instead of a caller-provided workspace.
namespace vec {

static __device__ __align__(256) unsigned char g_decode_scratch[VECTOR_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
static std::mutex g_scratch_mu;
static void* g_scratch_addr[kMaxDevices] = {};

// In host code `g_decode_scratch` is only a handle; the address a kernel can use
// comes from cudaGetSymbolAddress, once per device, with that device current.
static vector_status static_scratch_address(void** out) {
    int dev = -1;
    VEC_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return VECTOR_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        VEC_CUDA_CHECK(cudaGetSymbolAddress(&p, g_decode_scratch));
        if (!p) return VECTOR_ERR_CUDA;
        g_scratch_addr[dev] = p;
    }
    *out = g_scratch_addr[dev];
    return VECTOR_OK;
}

}  // namespace vec

extern "C" size_t vector_decode_scratch_bytes(const vector_shape* shape) {
    Dims dm;
    if (check_shape(shape, &dm) != VECTOR_OK) return 0;
    return decode_ws_bytes(dm);
}

extern "C" vector_status vector_decode_attn_static(const vector_shape* shape, const void* q,
                                                   const vector_cache* cache, const void* W, void* out,
                                                   int32_t out_dtype, int32_t mode, void* stream) {
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if (decode_ws_bytes(dm) > (size_t)VECTOR_STATIC_SCRATCH_BYTES) return VECTOR_ERR_WORKSPACE;
    void* scratch = nullptr;
    if ((rc = static_scratch_address(&scratch)) != VECTOR_OK) return rc;
    return vector_decode_attn(shape, q, cache, W, out, out_dtype, mode, scratch,
                              (size_t)VECTOR_STATIC_SCRATCH_BYTES, stream);
}

extern "C" int vector_device_fault(void) {
    int* addr = vec::kernel_fault_address();
    if (!addr) return -1;
    int v = 0, zero = 0;
    if (cudaDeviceSynchronize() != cudaSuccess) return -1;
    if (cudaMemcpy(&v, addr, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    if (v != 0) cudaMemcpy(addr, &zero, sizeof(int), cudaMemcpyHostToDevice);
    return v;
}
