// Base importance score (the scorer that Step 1 of the pipeline calls): causal
// observation-window attention mass per key, summed over window rows and the
// query heads of a KV head, then max-pooled along the sequence.
//
// The softmax normaliser of every window row is needed before the per-key sum
// over rows can be formed, so the logits are computed twice:
//   pass 1  per (unit, row tile, key chunk): running (max, sum exp) per row
//   combine per unit: lse[row] from the chunk partials
//   pass 2  per (unit, key tile): raw[key] = sum_rows exp(logit - lse[row])
//   pool    score[i] = max raw over the centred window (prefix only); +inf in the window
#include "common.cuh"
#include "internal.h"
#include "score_tc.cuh"

namespace vec {

constexpr int ST = 64;    // tile edge (rows and keys) of the CUDA-core score kernels

// The CUDA-core passes hold a whole 64 x D tile of each operand in shared memory (rows PITCH<D> apart) and request the next
// tile of the one that changes before they work on this one: with 32-channel slices loaded between barriers a pass was a
// chain of load latencies (13 + 11 us for 2 units of 64 rows and 1024 keys).
template <int D> struct TileRegs { float4 v[ST * D / 1024]; };
// WIDE: fp32 rows at multiples of 16 bytes; otherwise element by element.
template <bool WIDE, typename T, int D>
__device__ __forceinline__ void tile_request(const T* src, int64_t row0, int64_t n_rows, TileRegs<D>& t) {
#pragma unroll
    for (int e = 0; e < ST * D / 1024; ++e) {
        const int idx = threadIdx.x + 256 * e, r = idx / (D / 4), c4 = idx % (D / 4);
        const T* p = src + (row0 + r) * D + 4 * c4;
        const bool in = (uint64_t)(row0 + r) < (uint64_t)n_rows;            // rows before the first and behind the last read as zeros
        if constexpr (WIDE) {
            t.v[e] = in ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            t.v[e] = in ? make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3])) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}
// Rows of the tiles in shared memory are PITCH<D> floats apart: 16-byte accesses, whose rows begin four banks apart.
template <int D> constexpr int PITCH = D + 4;
template <int D>
__device__ __forceinline__ void tile_store(const TileRegs<D>& t, float* dst) {
#pragma unroll
    for (int e = 0; e < ST * D / 1024; ++e) {
        const int idx = threadIdx.x + 256 * e, r = idx / (D / 4), c = idx % (D / 4) * 4;
        *reinterpret_cast<float4*>(dst + r * PITCH<D> + c) = t.v[e];
    }
}
// acc[i][j] = sum_c Qs[ty + 16 i][c] * Ks[tx + 16 j][c].  Reads of shared memory are what bounds it: four channels a load, UNROLL loads
// of each row under way.
template <int D, int UNROLL>
__device__ __forceinline__ void tile_qk(const float* Qs, const float* Ks, float acc[4][4]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll (UNROLL)
    for (int kk = 0; kk < D; kk += 4) {
        float4 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(Qs + (ty + 16 * i) * PITCH<D> + kk);
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(Ks + (tx + 16 * j) * PITCH<D> + kk);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
                acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
                acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
                acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
            }
    }
}
// Blocks that outnumber four a multiprocessor (MANY, 64 channels): three resident at 80 registers instead of two at 114 to 127, which
// unroll the channels.  us, MANY / not: 148 units of 32 rows and 300 keys 35 / 39, 32 of 2000 keys 48 / 52; few blocks, 8 units of 2000 keys
// 21 / 16, one unit of 256 rows and 32768 keys 111 / 91.  At 128 channels two blocks are resident either way.
template <bool MANY> constexpr int MIN_BLOCKS = MANY ? 3 : 2;
template <int D> static bool many_blocks(int64_t blocks) { return D == 64 && blocks > 4 * (int64_t)sm_count(); }
template <int D> constexpr int tile_smem() { return 2 * ST * PITCH<D> * (int)sizeof(float); }

// grid (n_chunks, row_tiles, U), 256 threads, tile_smem of dynamic shared memory
template <typename T, int D, bool WIDE, bool MANY>
__global__ void __launch_bounds__(256, MIN_BLOCKS<MANY>)
score_pass1_generic(const T* Q, const T* K, int64_t N, int R, int w,
                    float scale, int64_t chunk_len, float2* __restrict__ partial) {
    extern __shared__ __align__(16) float tiles[];
    float *Qs = tiles, *Ks = tiles + ST * PITCH<D>;
    asm volatile("griddepcontrol.wait;\n" ::: "memory");        // launched as a programmatic dependent: nothing is touched before
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int u = blockIdx.z, row0 = blockIdx.y * ST, chunk = blockIdx.x, n_chunks = gridDim.x;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const T* Qu = Q + (size_t)u * R * D;
    const T* Ku = K + (size_t)u * N * D;
    const int64_t k_begin = (int64_t)chunk * chunk_len;
    const int64_t k_end = min(N, k_begin + chunk_len);
    TileRegs<D> next;
    tile_request<WIDE>(Ku, k_begin, k_end, next);
    {
        TileRegs<D> q;
        tile_request<WIDE>(Qu, row0, R, q);
        tile_store<D>(q, Qs);
    }
    float m[4], l[4];
    int64_t last_visible[4];   // row j of the window sits at position N - w + j
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m[i] = -INFINITY;
        l[i] = 0.f;
        int row = row0 + ty + 16 * i;
        last_visible[i] = row < R ? N - w + (row % w) : -1;
    }
    for (int64_t key0 = k_begin; key0 < k_end; key0 += ST) {
        __syncthreads();                                  // the tile before this one has been read
        tile_store<D>(next, Ks);
        __syncthreads();
        if (key0 + ST < k_end) tile_request<WIDE>(Ku, key0 + ST, k_end, next);
        float acc[4][4];
        tile_qk<D, MANY ? 1 : 4>(Qs, Ks, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float s[4], mx = m[i];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                int64_t key = key0 + tx + 16 * j;
                s[j] = (key < k_end && key <= last_visible[i]) ? acc[i][j] * scale : -INFINITY;
                mx = fmaxf(mx, s[j]);
            }
            if (mx > -INFINITY) {
                float sum = l[i] * __expf(m[i] - mx);   // m = -inf -> factor 0
#pragma unroll
                for (int j = 0; j < 4; ++j) sum += expf(s[j] - mx);
                m[i] = mx;
                l[i] = sum;
            }
        }
    }
    // combine the 16 threads (one half-warp) that share a row
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float M = m[i];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        float v = (m[i] > -INFINITY) ? l[i] * expf(m[i] - M) : 0.f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        int row = row0 + ty + 16 * i;
        if (tx == 0 && row < R) partial[((size_t)u * n_chunks + chunk) * R + row] = make_float2(M, v);
    }
}

// lse of a row from its chunk partials, `stride` apart, four lanes (of one aligned group) together.
__device__ __forceinline__ float row_lse(const float2* p, int stride, int n_chunks) {
    const int part = threadIdx.x & 3;
    float M = -INFINITY, L = 0.f;
    for (int c0 = part; c0 < n_chunks; c0 += 16) {
        float2 v[4];
        float m = M;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = c0 + 4 * k < n_chunks ? p[(size_t)(c0 + 4 * k) * stride] : make_float2(-INFINITY, 0.f);
            m = fmaxf(m, v[k].x);
        }
        if (m == -INFINITY) continue;
        L *= expf(M - m);
#pragma unroll
        for (int k = 0; k < 4; ++k) L += v[k].y * expf(v[k].x - m);
        M = m;
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        const float M2 = __shfl_xor_sync(0xffffffffu, M, o), L2 = __shfl_xor_sync(0xffffffffu, L, o);
        const float m = fmaxf(M, M2);
        L = m > -INFINITY ? L * expf(M - m) + L2 * expf(M2 - m) : 0.f;
        M = m;
    }
    return M + logf(L);
}
// lse[u][row].  grid (ceil(R / 64), U), 256 threads
__global__ void __launch_bounds__(256)
score_lse_rows(const float2* partial, int R, int n_chunks, float* __restrict__ lse) {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int row = blockIdx.x * 64 + (threadIdx.x >> 2);
    const float v = row_lse(partial + (size_t)blockIdx.y * n_chunks * R + min(row, R - 1), R, n_chunks);
    if (row < R && (threadIdx.x & 3) == 0) lse[(size_t)blockIdx.y * R + row] = v;
}

// grid (key_tiles, U), 256 threads, tile_smem of dynamic shared memory.  INLINE_LSE: a block forms the normalisers of its
// rows itself from the chunk partials (a launch less; every key tile repeats it).  POOLED: the block pools its sums itself (another
// launch less); its tiles overlap by the pooling radius on both sides, raw may be null.
template <typename T, int D, bool INLINE_LSE, bool WIDE, bool POOLED, bool MANY>
__global__ void __launch_bounds__(256, MIN_BLOCKS<MANY>)
score_pass2_generic(const T* Q, const T* K, int64_t N, int R, int w,
                    float scale, const float2* partial, int n_chunks, const float* lse,
                    float* __restrict__ raw, int r, float* __restrict__ score) {
    extern __shared__ __align__(16) float tiles[];
    float *Qs = tiles, *Ks = tiles + ST * PITCH<D>;
    __shared__ float red[16][ST];
    __shared__ float lse_s[ST];
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int u = blockIdx.y;
    const int64_t key0 = POOLED ? (int64_t)blockIdx.x * (ST - 2 * r) - r : (int64_t)blockIdx.x * ST;       // POOLED: -r at first
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const T* Qu = Q + (size_t)u * R * D;
    TileRegs<D> next;
    {
        TileRegs<D> k;
        tile_request<WIDE>(K + (size_t)u * N * D, key0, N, k);
        tile_request<WIDE>(Qu, 0, R, next);
        tile_store<D>(k, Ks);
    }
    float col[4] = {0.f, 0.f, 0.f, 0.f};
    for (int row0 = 0; row0 < R; row0 += ST) {
        __syncthreads();                                  // the rows before these have been read
        tile_store<D>(next, Qs);
        if (INLINE_LSE) {
            const int row = row0 + (tid >> 2);
            const float v = row_lse(partial + (size_t)u * n_chunks * R + min(row, R - 1), R, n_chunks);
            if ((tid & 3) == 0) lse_s[tid >> 2] = v;
        } else if (tid < ST && row0 + tid < R) {
            lse_s[tid] = lse[(size_t)u * R + row0 + tid];
        }
        __syncthreads();
        if (row0 + ST < R) tile_request<WIDE>(Qu, row0 + ST, R, next);
        float acc[4][4];
        tile_qk<D, MANY ? 1 : 4>(Qs, Ks, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int row = row0 + ty + 16 * i;
            if (row < R) {
                float ls = lse_s[ty + 16 * i];
                int64_t last_visible = N - w + (row % w);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    int64_t key = key0 + tx + 16 * j;
                    if (key <= last_visible) col[j] += expf(acc[i][j] * scale - ls);
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) red[ty][tx + 16 * j] = col[j];
    __syncthreads();
    if (tid < ST) {
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < 16; ++t) s += red[t][tid];
        int64_t key = key0 + tid;
        if constexpr (!POOLED) {
            if (key < N) raw[(size_t)u * N + key] = s;
        } else {
            const bool own = tid >= r && tid < ST - r && key < N;
            if (raw && own) raw[(size_t)u * N + key] = s;
            lse_s[tid] = key >= 0 && key < N - w ? s : -INFINITY;            // pooling looks at the prefix only
        }
    }
    if constexpr (POOLED) {
        __syncthreads();
        const int64_t key = key0 + tid;
        if (tid >= r && tid < ST - r && key < N) {
            float best = -INFINITY;
            for (int k = tid - r; k <= tid + r; ++k) best = fmaxf(best, lse_s[k]);
            score[(size_t)u * N + key] = key < N - w ? best : INFINITY;
        }
    }
}

// score[i] = max_{|j-i| <= r, 0 <= j < N-w} raw[j] for i < N-w ; +inf for the window tokens
__global__ void score_pool_kernel(const float* raw, int64_t N, int w, int r, int64_t total,
                                  float* __restrict__ score) {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= total) return;
    int64_t u = gi / N, i = gi - u * N;
    int64_t P = N - w;
    float best = INFINITY;
    if (i < P) {
        best = -INFINITY;
        int64_t lo = max((int64_t)0, i - r), hi = min(P - 1, i + r);
        for (int64_t j = lo; j <= hi; ++j) best = fmaxf(best, raw[u * N + j]);
    }
    score[gi] = best;
}

// Workspace: chunk partials | lse | raw, where the caller does not take it; fewer chunks where it would not hold theirs.
template <typename T, int D, bool WIDE>
static vector_status launch_score(const Dims& dm, const void* Q_, const void* K_, int64_t N, float* scores, float* raw_out, char* ws,
                                  size_t ws_bytes, cudaStream_t st) {
    constexpr int SMEM = tile_smem<D>();
    const T *Q = (const T*)Q_, *K = (const T*)K_;
    constexpr bool M = D == 64;              // the kernels for many blocks, where there are such
    static PerDeviceOnce once;
    if (once.first()) {
        auto opt_in = [](auto kern) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM); };
        cudaError_t e = opt_in(score_pass1_generic<T, D, WIDE, false>);
        if (e == cudaSuccess) e = opt_in(score_pass1_generic<T, D, WIDE, M>);
        if (e == cudaSuccess) e = opt_in(score_pass2_generic<T, D, true, WIDE, true, false>);
        if (e == cudaSuccess) e = opt_in(score_pass2_generic<T, D, true, WIDE, false, false>);
        if (e == cudaSuccess) e = opt_in(score_pass2_generic<T, D, true, WIDE, false, M>);
        if (e == cudaSuccess) e = opt_in(score_pass2_generic<T, D, false, WIDE, false, false>);
        if (e == cudaSuccess) e = opt_in(score_pass2_generic<T, D, false, WIDE, false, M>);
        if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
    }
    const size_t lse_b = align256((size_t)dm.U * dm.R * sizeof(float)), raw_b = raw_out ? 0 : align256((size_t)dm.U * (size_t)N * sizeof(float));
    int n_chunks = score_num_chunks(dm.U, dm.R, N);
    auto partial_b = [&] { return align256((size_t)dm.U * n_chunks * dm.R * sizeof(float2)); };
    while (n_chunks > 1 && partial_b() + lse_b + raw_b > ws_bytes) --n_chunks;
    float2* partial = (float2*)ws;
    float* lse = (float*)(ws + partial_b());
    float* raw = raw_out ? raw_out : (float*)(ws + partial_b() + lse_b);
    int64_t chunk_len = (N + n_chunks - 1) / n_chunks;
    chunk_len = (chunk_len + ST - 1) / ST * ST;
    n_chunks = (int)((N + chunk_len - 1) / chunk_len);            // none empty
    const int row_tiles = (dm.R + ST - 1) / ST;
    auto pass1 = many_blocks<D>((int64_t)n_chunks * row_tiles * dm.U) ? score_pass1_generic<T, D, WIDE, M> : score_pass1_generic<T, D, WIDE, false>;
    VEC_CUDA_CHECK(launch_maybe_dependent(true, pass1, dim3(n_chunks, row_tiles, dm.U), dim3(256), SMEM, st, Q, K, N, dm.R, dm.w, dm.scale,
                                          chunk_len, partial));
    // the partials of a row tile: no more than the rows' own elements
    const bool inline_lse = n_chunks <= 32;
    if (!inline_lse)
        VEC_CUDA_CHECK(launch_maybe_dependent(true, score_lse_rows, dim3((dm.R + 63) / 64, dm.U), dim3(256), 0, st, partial, dm.R,
                                              n_chunks, lse));
    // The launch that pooling costs counts where the second pass is short: no more blocks than multiprocessors, overlaps included.
    const int r = dm.pool_kernel / 2;
    const int64_t tiles_pooled = (N + ST - 2 * r - 1) / (ST - 2 * r);
    if (inline_lse && tiles_pooled * dm.U <= sm_count()) {
        VEC_CUDA_CHECK(launch_maybe_dependent(true, score_pass2_generic<T, D, true, WIDE, true, false>, dim3((unsigned)tiles_pooled, dm.U), dim3(256), SMEM, st,
                                              Q, K, N, dm.R, dm.w, dm.scale, partial, n_chunks, lse, raw_out, r, scores));
        return VECTOR_OK;
    }
    const int64_t tiles = (N + ST - 1) / ST;
    auto pass2 = many_blocks<D>(tiles * dm.U)
                     ? (inline_lse ? score_pass2_generic<T, D, true, WIDE, false, M> : score_pass2_generic<T, D, false, WIDE, false, M>)
                     : (inline_lse ? score_pass2_generic<T, D, true, WIDE, false, false> : score_pass2_generic<T, D, false, WIDE, false, false>);
    VEC_CUDA_CHECK(launch_maybe_dependent(true, pass2, dim3((unsigned)tiles, dm.U), dim3(256), SMEM, st, Q, K, N, dm.R, dm.w, dm.scale,
                                          partial, n_chunks, lse, raw, r, scores));
    int64_t total = (int64_t)dm.U * N;
    VEC_CUDA_CHECK(launch_maybe_dependent(true, score_pool_kernel, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, st, raw, N, dm.w,
                                          dm.pool_kernel / 2, total, scores));
    return VECTOR_OK;
}

// bf16: tcgen05 passes.  Workspace: chunk partials | lse | per-row-block key sums.
template <int D>
static vector_status launch_score_tc(const Dims& dm, const void* Q, const void* K, int64_t N, float* scores,
                                     float* raw_out, char* ws, cudaStream_t st) {
    constexpr int SMEM = stc::Cfg<D>::SMEM_BYTES, SMEM_POOLED = SMEM + 2 * stc::POOLED_KEYS * 4;
    const ScoreTcPlan pl = score_tc_plan(dm.U, dm.R, N);
    float2* partial = (float2*)ws;
    ws += align256((size_t)dm.U * 2 * pl.n_chunks * dm.R * 2 * sizeof(float));
    float* lse2 = (float*)ws;
    ws += align256((size_t)dm.U * dm.R * sizeof(float));
    float* raw_part = (float*)ws;
    static PerDeviceOnce once;
    if (once.first()) {
        auto opt_in = [](auto kern, int bytes) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
        cudaError_t e = opt_in(stc::score_pass1_tc<D, 1>, SMEM);
        if (e == cudaSuccess) e = opt_in(stc::score_pass1_tc<D, 2>, SMEM);
        if (e == cudaSuccess) e = opt_in(stc::score_pass2_tc<D, true, 1, true>, SMEM_POOLED);
        if (e == cudaSuccess) e = opt_in(stc::score_pass2_tc<D, true, 2, true>, SMEM_POOLED);
        if (e == cudaSuccess) e = opt_in(stc::score_pass2_tc<D, true, 1, false>, SMEM);
        if (e == cudaSuccess) e = opt_in(stc::score_pass2_tc<D, true, 2, false>, SMEM);
        if (e == cudaSuccess) e = opt_in(stc::score_pass2_tc<D, false, 1, false>, SMEM);
        if (e == cudaSuccess) e = opt_in(stc::score_pass2_tc<D, false, 2, false>, SMEM);
        if (e != cudaSuccess) { once.undo(); VEC_CUDA_CHECK(e); }
    }
    int* fault = kernel_fault_address();
    if (!fault) return VECTOR_ERR_CUDA;
    CUtensorMap mapQ, mapK;
    if (!tma::encode_bf16_3d(&mapQ, Q, D, (uint64_t)dm.R, (uint64_t)dm.U, 2 * D, (uint64_t)dm.R * 2 * D, 64, 128) ||
        !tma::encode_bf16_3d(&mapK, K, D, (uint64_t)N, (uint64_t)dm.U, 2 * D, (uint64_t)N * 2 * D, 64, 128))
        return VECTOR_ERR_CUDA;
    stc::Params P;
    P.U = dm.U; P.R = dm.R; P.RG = pl.RG; P.w = dm.w; P.N = N;
    P.tpc = pl.tpc; P.step = pl.tpc * stc::KT; P.lead = 0; P.n_chunks = P.lse_chunks = pl.n_chunks; P.n_items = pl.n_items;
    P.c = dm.scale * 1.4426950408889634f;
    const int sms = sm_count();
    const int blocks = pl.n_items < sms ? pl.n_items : sms;
    const bool one = dm.R <= 128;
    auto pass1 = one ? stc::score_pass1_tc<D, 1> : stc::score_pass1_tc<D, 2>;
    pass1<<<blocks, stc::THREADS, SMEM, st>>>(mapQ, mapK, P, partial, fault);
    VEC_LAUNCH_CHECK();
    // A block has one or two items: the passes are short, so the second forms the normalisers itself and each kernel after
    // the first is a programmatic dependent of the one before it.  Long passes are launched the ordinary way: as a
    // dependent, pass 2 has its blocks placed as multiprocessors fall free and no longer side by side, where the row
    // groups of a key chunk share what they fetch (640 units of 1024 rows, 131072 keys: 53.7 ms against 52.9).
    const bool few = pl.n_items <= 2 * blocks;
    if (few && pl.RG == 1) {
        // Pooling in the second pass: its chunks overlap, so they have a tile more where their number would go up.
        const int r = dm.pool_kernel / 2;
        stc::Params P2 = P;
        P2.lead = r;
        for (P2.tpc = pl.tpc; P2.tpc <= pl.tpc + 1 && P2.tpc * stc::KT <= stc::POOLED_KEYS; ++P2.tpc) {
            P2.step = P2.tpc * stc::KT - 2 * r;
            P2.n_chunks = (int)((N + P2.step - 1) / P2.step);
            const long long items = (long long)dm.U * P2.n_chunks;
            if (items > (long long)sms * ((pl.n_items + blocks - 1) / blocks)) continue;       // no more rounds than without
            P2.n_items = (int)items;
            auto pass2 = one ? stc::score_pass2_tc<D, true, 1, true> : stc::score_pass2_tc<D, true, 2, true>;
            VEC_CUDA_CHECK(launch_maybe_dependent(true, pass2, dim3(items < sms ? (unsigned)items : sms), dim3(stc::THREADS), SMEM_POOLED, st, mapQ,
                                                  mapK, P2, partial, lse2, raw_part, raw_out, scores, fault));
            return VECTOR_OK;
        }
    }
    auto pass2 = one ? (few ? stc::score_pass2_tc<D, true, 1, false> : stc::score_pass2_tc<D, false, 1, false>)
                     : (few ? stc::score_pass2_tc<D, true, 2, false> : stc::score_pass2_tc<D, false, 2, false>);
    if (!few)
        VEC_CUDA_CHECK(launch_maybe_dependent(false, stc::score_lse2_rows, dim3((dm.R + 127) / 128, dm.U), dim3(256), 0, st, partial, dm.R,
                                              pl.n_chunks, lse2));
    VEC_CUDA_CHECK(launch_maybe_dependent(few, pass2, dim3(blocks), dim3(stc::THREADS), SMEM, st, mapQ, mapK, P, partial, lse2, raw_part,
                                          raw_out, scores, fault));
    const dim3 gp((unsigned)((N + stc::POOL_TILE - 1) / stc::POOL_TILE), dm.U);
    VEC_CUDA_CHECK(launch_maybe_dependent(few, (N & 3) == 0 ? stc::score_pool_parts_v4 : stc::score_pool_parts, gp, dim3(256), 0, st,
                                          raw_part, (dm.R + 127) / 128, N, dm.w, dm.pool_kernel / 2, raw_out, scores));
    return VECTOR_OK;
}

}  // namespace vec

extern "C" float vector_score_exp2_fma_share(void) { return (float)vec::stc::POLY16 / 16.0f; }

extern "C" vector_status vector_score(const vector_shape* shape, const void* Q_obs, const void* K, int64_t N,
                                      float* scores, float* raw_out, void* ws, size_t ws_bytes, void* stream) {
    using namespace vec;
    Dims dm;
    vector_status rc = check_shape(shape, &dm);
    if (rc != VECTOR_OK) return rc;
    if (!Q_obs || !K || !scores) return VECTOR_ERR_NULL;
    if (N < dm.w || N > (int64_t(1) << 30)) return VECTOR_ERR_SHAPE;
    if ((int64_t)((N + ST - 1) / ST) > 0x7fffffff) return VECTOR_ERR_SHAPE;
    const bool need_raw = raw_out == nullptr;
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < score_ws_bytes(dm, N, need_raw)) return VECTOR_ERR_WORKSPACE;
    char* p = (char*)ws;
    cudaStream_t st = (cudaStream_t)stream;
    // Rows off a 16-byte boundary: element by element, 64-channel bf16 ones, which TMA would refuse, on the CUDA-core kernels too
    const bool wide = (((uintptr_t)Q_obs | (uintptr_t)K) & 15) == 0;
    if (score_uses_tc(dm) && (dm.d == 128 || (wide && (((uintptr_t)scores | (uintptr_t)raw_out) & 15) == 0)))
        return dm.d == 64 ? launch_score_tc<64>(dm, Q_obs, K, N, scores, raw_out, p, st)
                          : launch_score_tc<128>(dm, Q_obs, K, N, scores, raw_out, p, st);
    auto launch = dm.dtype == VECTOR_BF16 ? launch_score<__nv_bfloat16, 64, false>
                : dm.d == 64 ? (wide ? launch_score<float, 64, true> : launch_score<float, 64, false>)
                             : (wide ? launch_score<float, 128, true> : launch_score<float, 128, false>);
    return launch(dm, Q_obs, K, N, scores, raw_out, p, ws_bytes, st);
}
