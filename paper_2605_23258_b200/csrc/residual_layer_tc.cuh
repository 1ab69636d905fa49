// Reconstruction residual of Step 2 for ONE map per layer (bf16, head_dim 128): the map is
// calibrated layer-wise (paper Section 5.1) on the keys and values concatenated over the layer's
// KV heads, so
//   eps[p] = sum_h || v_{i,h} - sum_h' W[h][h'] k_{i,h'} ||^2,   i = idx[p],
// with W[h][h'] the 128 x 128 block (output head h, input head h') of the [Hkv d][Hkv d] map.
// A dense contraction with K = Hkv d: for a tile of 128 listed tokens and a pair of output heads the
// accumulator in tensor memory (256 columns) collects D = sum_h' K_h' W[h, h + 1][h']^T, 8 tcgen05.mma
// with N = 256 per h'; the epilogue subtracts the value rows of the two heads, squares and adds along
// its TMEM lane.
//
// What bounds it is what a tile fetches: the keys once per pair of output heads and the whole map, 3.25 MB for
// 17.7 us of tensor work at Hkv = 8, mostly from L2.  So the loads are kept in flight across steps (half a head's
// channels, 48 KB, in one of four stages), the products take two output heads at a time (a third fewer bytes than
// head by head), and the value rows, 256 KB of the 3.25 MB, go straight to the epilogue's registers.
//
// Persistent blocks (one per multiprocessor) own equal contiguous ranges of the sequence of items (tile, pair of output
// heads), which balances better than whole tiles: 624 tiles are 4.2 a block.  A tile cut by the end of a range is finished
// by the next block: both add their share to eps, which starts at zero (two addends: the order does not matter).
//   warps 0-7   loaders: gathers of the K rows of a step (cp.async, written in the 128-byte-swizzled operand layout),
//               published three steps behind the one being issued; thread 0 also issues the W loads (TMA)
//   warp  8     MMA issuer, TMEM owner (two 256-column accumulators: the epilogue of a pair runs under the next one)
//   warps 9-12  epilogue: thread = row; its value row comes in 32-byte loads (16-byte ones where it has to), a head ahead
// Measured on 16 layers of 4914 listed tokens and 8 heads: 245 us (388 before: one output head at a time, loads waited for in
// every step, 64-bit divisions in every role), 53 KB a microsecond and multiprocessor: the rate at which L2 delivers.
#ifndef VECTOR_RESIDUAL_LAYER_TC_CUH_
#define VECTOR_RESIDUAL_LAYER_TC_CUH_

#include "common.cuh"
#include "internal.h"
#include "residual_tc.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace vec {
namespace rlt {

using rtc::BOX_BYTES;
using rtc::TILE;

constexpr int STAGES = 4;
constexpr int STAGE_BYTES = 3 * BOX_BYTES;                // 64 channels of: the tile's keys of one head | the map's rows of two heads
constexpr int LOADER_WARPS = 8;
constexpr int EPI_WARPS = 4;
constexpr int THREADS = 32 * (LOADER_WARPS + 1 + EPI_WARPS);
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
constexpr int TMEM_COLS = 512;

struct Params {
    int UL, L, Hkv, n_idx, tpu;      // (sequence, layer) units, layers, KV heads, rows per unit, tiles per unit
    int pairs;                       // ceil(Hkv / 2)
    long long N, n_items;            // keys per head, UL * tpu * pairs
};
struct Sync {
    uint64_t full[STAGES], w_full[STAGES], empty[STAGES];
    uint64_t acc_full[2], acc_empty[2];
    uint32_t tmem_base;
};
// Position in the sequence of items, stepped along.
struct Cursor {
    int ul, t, pair;
    __device__ __forceinline__ void next(const Params& P) {
        if (++pair == P.pairs) { pair = 0; if (++t == P.tpu) { t = 0; ++ul; } }
    }
};
__device__ __forceinline__ Cursor cursor_at(long long item, const Params& P) {
    Cursor c;
    const long long tile = item / P.pairs;
    c.pair = (int)(item - tile * P.pairs);
    c.ul = (int)(tile / P.tpu);
    c.t = (int)(tile - (long long)c.ul * P.tpu);
    return c;
}
// 32 bytes through the read-only path: in one load (WIDE, the address a multiple of 32) or in two.
template <bool WIDE>
__device__ __forceinline__ void ldg32(const void* p, uint32_t (&r)[64], int at) {
    if constexpr (WIDE) {
        asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                     : "=r"(r[at]), "=r"(r[at + 1]), "=r"(r[at + 2]), "=r"(r[at + 3]), "=r"(r[at + 4]), "=r"(r[at + 5]), "=r"(r[at + 6]), "=r"(r[at + 7])
                     : "l"(p));
    } else {
#pragma unroll
        for (int h = 0; h < 8; h += 4)
            asm volatile("ld.global.nc.v4.b32 {%0,%1,%2,%3}, [%4];\n"
                         : "=r"(r[at + h]), "=r"(r[at + h + 1]), "=r"(r[at + h + 2]), "=r"(r[at + h + 3])
                         : "l"((const unsigned char*)p + 4 * h));
    }
}

// grid: at most one block per multiprocessor and a range of at least `pairs` items each (so that a tile is cut once at
// most), THREADS threads, SMEM_BYTES dynamic shared memory.
// K, V: [UL][Hkv][N][128]; idx: [UL][n_idx]; eps: [UL][n_idx], zero; mapW: (Hkv*128 in, Hkv*128 out, L), box 64 x 128.
// WIDE: V is a multiple of 32 bytes.  The interface promises 16; rows are 256 bytes apart, so the base decides for all of them.
template <bool WIDE>
__global__ void __launch_bounds__(THREADS, 1)
residual_layer_tc(const __nv_bfloat16* __restrict__ K, const __nv_bfloat16* __restrict__ V,
                  const __grid_constant__ CUtensorMap mapW, const int32_t* __restrict__ idx, const Params P,
                  float* __restrict__ eps, int* __restrict__ fault) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ Sync sy;
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long it_lo = rtc::range_begin(blockIdx.x, P.n_items, gridDim.x);
    const int n_my = (int)(rtc::range_begin(blockIdx.x + 1, P.n_items, gridDim.x) - it_lo);
    const int H = P.Hkv;

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < STAGES; ++s) {
            tma::mbar_init(&sy.full[s], 32 * LOADER_WARPS);
            tma::mbar_init(&sy.w_full[s], 1);
            tma::mbar_init(&sy.empty[s], 1);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) { tma::mbar_init(&sy.acc_full[k], 1); tma::mbar_init(&sy.acc_empty[k], EPI_WARPS); }
        tma::mbar_fence_init();
    }
    if (warp == LOADER_WARPS) {
        tc::tmem_alloc(&sy.tmem_base, TMEM_COLS);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();

    if (warp < LOADER_WARPS) {
        // ------------------------------------------------------------------ loaders
        const int qc = tid & 7, rsub = tid >> 3;                    // 16-byte chunk of the 64 channels, row inside a pass of 32 rows
        const uint32_t dst_thread = (uint32_t)rsub * 128u + (uint32_t)((qc ^ (rsub & 7)) << 4);   // + pass * 4096
        int32_t rows[4];                                             // this thread's four rows of the tile at hand
        bool ok = true;
        if (tid == 0) tma::prefetch_map(&mapW);
        asm volatile("griddepcontrol.wait;\n" ::: "memory");      // idx is complete and visible from here on
        asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
        Cursor at = cursor_at(it_lo, P);
        uint32_t step = 0;
        for (int i = 0; i < n_my && ok; ++i, at.next(P)) {
            if (i == 0 || at.pair == 0) {
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const int row = at.t * TILE + p * 32 + rsub;
                    const int32_t v = row < P.n_idx ? idx[(size_t)at.ul * P.n_idx + row] : -1;
                    rows[p] = (unsigned long long)v < (unsigned long long)P.N ? v : -1;     // an index outside the unit reads as zeros
                }
            }
            const int heads = min(2, H - 2 * at.pair), layer = at.ul % P.L;
            for (int hk = 0; hk < 2 * H && ok; ++hk, ++step) {     // (input head, half of its channels)
                const uint32_t s = step % STAGES, round = step / STAGES;
                if (round > 0 && !tma::mbar_wait(&sy.empty[s], (round - 1) & 1, fault, 81)) { ok = false; break; }
                unsigned char* st = smem + s * STAGE_BYTES;
                if (tid == 0) {                                     // the blocks (h, h') of the pair's output heads
                    tma::mbar_expect_tx(&sy.w_full[s], heads * BOX_BYTES);
                    for (int e = 0; e < heads; ++e)
                        tma::load_3d(st + (1 + e) * BOX_BYTES, &mapW, hk * 64, (2 * at.pair + e) * 128, layer, &sy.w_full[s]);
                }
                const uint32_t kdst = tma::smem_u32(st) + dst_thread;
                const __nv_bfloat16* Ku = K + ((size_t)at.ul * H + (hk >> 1)) * P.N * 128 + (hk & 1) * 64 + qc * 8;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const bool valid = rows[p] >= 0;
                    rtc::cp_async16(kdst + p * 4096, Ku + (valid ? (size_t)rows[p] * 128 : 0), valid ? 16u : 0u);   // zero fill past the end
                }
                rtc::cp_async_commit();
                if (step >= STAGES - 1) {                           // this thread's copies of the step STAGES - 1 before this one have landed
                    rtc::cp_async_wait<STAGES - 1>();
                    rtc::fence_async_proxy();
                    tma::mbar_arrive(&sy.full[(step - (STAGES - 1)) % STAGES]);
                }
            }
        }
        if (ok) {
            auto publish = [&](uint32_t behind) {                   // step `behind` before the last, if there is one
                if (step > behind) { rtc::fence_async_proxy(); tma::mbar_arrive(&sy.full[(step - 1 - behind) % STAGES]); }
            };
            rtc::cp_async_wait<2>(); publish(2);
            rtc::cp_async_wait<1>(); publish(1);
            rtc::cp_async_wait<0>(); publish(0);
        } else {
            rtc::cp_async_wait<0>();
        }
    } else if (warp == LOADER_WARPS) {
        // ------------------------------------------------------------------ MMA issue
        if (lane == 0) {
            asm volatile("griddepcontrol.wait;\n" ::: "memory");    // the bounded waits below time this kernel only
            Cursor at = cursor_at(it_lo, P);
            uint32_t step = 0;
            bool ok = true;
            for (int i = 0; i < n_my && ok; ++i, at.next(P)) {
                const uint32_t buf = i & 1, use = i >> 1;
                const uint32_t idesc = H - 2 * at.pair > 1 ? tc::instr_desc(128, 256) : tc::instr_desc(128, 128);
                const uint32_t d = sy.tmem_base + buf * 256;
                if (use > 0 && !tma::mbar_wait(&sy.acc_empty[buf], (use - 1) & 1, fault, 83)) break;
                for (int hk = 0; hk < 2 * H; ++hk, ++step) {
                    const uint32_t s = step % STAGES, round = step / STAGES;
                    if (!tma::mbar_wait(&sy.w_full[s], round & 1, fault, 85) || !tma::mbar_wait(&sy.full[s], round & 1, fault, 84)) { ok = false; break; }
                    tc::fence_after_sync();
                    const uint32_t k_addr = tma::smem_u32(smem + s * STAGE_BYTES), w_addr = k_addr + BOX_BYTES;
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        tc::mma_bf16(d, tc::smem_desc(k_addr + ks * 32), tc::smem_desc(w_addr + ks * 32), idesc, (hk > 0 || ks > 0) ? 1u : 0u);
                    tc::mma_commit(&sy.empty[s]);                   // the stage is free once these products have read it
                }
                if (ok) tc::mma_commit(&sy.acc_full[buf]);
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3;                       // TMEM lanes this warp may read: 32 (warp % 4) ..
        const int r = quarter * 32 + lane;
        const uint32_t lane_addr = sy.tmem_base + ((uint32_t)(quarter * 32) << 16);
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
        Cursor at = cursor_at(it_lo, P);
        auto token_of = [&](const Cursor& c) -> int32_t {
            const int row = c.t * TILE + r;
            const int32_t v = c.ul < P.UL && row < P.n_idx ? idx[(size_t)c.ul * P.n_idx + row] : -1;
            return (unsigned long long)v < (unsigned long long)P.N ? v : -1;
        };
        auto value_row = [&](const Cursor& c, int32_t tok, int e) -> const unsigned char* {
            return tok < 0 ? nullptr : reinterpret_cast<const unsigned char*>(V + (((size_t)c.ul * H + 2 * c.pair + e) * P.N + tok) * 128);
        };
        uint32_t vv[64];                                    // the value row of the head at hand, replaced 64 bytes at a time by the next one's
        auto fetch = [&](const unsigned char* src, int ch) {
            if (src) { ldg32<WIDE>(src + ch * 64, vv, 16 * ch); ldg32<WIDE>(src + ch * 64 + 32, vv, 16 * ch + 8); }
            else {
#pragma unroll
                for (int k = 0; k < 16; ++k) vv[16 * ch + k] = 0u;
            }
        };
        int32_t tok = n_my > 0 ? token_of(at) : -1;
        if (n_my > 0) {
            const unsigned char* src = value_row(at, tok, 0);
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) fetch(src, ch);
        }
        float e_tok = 0.f;
        bool whole = true;                                  // this block has had all of the tile's items so far
        for (int i = 0; i < n_my; ++i) {
            const uint32_t buf = i & 1, use = i >> 1;
            Cursor nx = at;
            nx.next(P);
            const bool last = at.pair + 1 == P.pairs || i + 1 == n_my;      // of this tile, here
            const int32_t tok_next = at.pair + 1 == P.pairs && i + 1 < n_my ? token_of(nx) : tok;
            if (i == 0 && at.pair > 0) whole = false;
            if (!tma::mbar_wait_warp(&sy.acc_full[buf], use & 1, fault, 87)) break;
            tc::fence_after_sync();
            const int heads = min(2, H - 2 * at.pair);
            for (int e = 0; e < heads; ++e) {
                // the head after this one: of the same pair, or of the next item
                const unsigned char* src = e + 1 < heads ? value_row(at, tok, e + 1) : i + 1 < n_my ? value_row(nx, tok_next, 0) : nullptr;
                uint32_t ra[32], rb[32];
                const uint32_t taddr = lane_addr + buf * 256 + e * 128;
                tc::tmem_ld32(taddr, ra);
                float e0 = 0.f, e1 = 0.f, e2 = 0.f, e3 = 0.f;
#pragma unroll
                for (int ch = 0; ch < 4; ++ch) {
                    uint32_t (&cur)[32] = (ch & 1) ? rb : ra;
                    uint32_t (&nxt)[32] = (ch & 1) ? ra : rb;
                    tc::tmem_ld_wait(cur);
                    if (ch < 3) tc::tmem_ld32(taddr + (ch + 1) * 32, nxt);
#pragma unroll
                    for (int k = 0; k < 32; k += 4) {
                        const uint32_t v0 = vv[16 * ch + (k >> 1)], v1 = vv[16 * ch + (k >> 1) + 1];
                        const float a = __uint_as_float(cur[k]) - __uint_as_float(v0 << 16);
                        const float b = __uint_as_float(cur[k + 1]) - __uint_as_float(v0 & 0xffff0000u);
                        const float c2 = __uint_as_float(cur[k + 2]) - __uint_as_float(v1 << 16);
                        const float d2 = __uint_as_float(cur[k + 3]) - __uint_as_float(v1 & 0xffff0000u);
                        e0 = fmaf(a, a, e0); e1 = fmaf(b, b, e1); e2 = fmaf(c2, c2, e2); e3 = fmaf(d2, d2, e3);
                    }
                    fetch(src, ch);
                }
                e_tok += (e0 + e1) + (e2 + e3);
                __syncwarp();
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tma::mbar_arrive(&sy.acc_empty[buf]);
            if (last) {
                const int row = at.t * TILE + r;
                if (row < P.n_idx) {
                    float* dst = eps + (size_t)at.ul * P.n_idx + row;
                    if (whole && at.pair + 1 == P.pairs) *dst = e_tok;
                    else atomicAdd(dst, e_tok);             // the other share comes from a neighbouring block
                }
                e_tok = 0.f;
                whole = true;
            }
            at = nx;
            tok = tok_next;
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == LOADER_WARPS) {
        __syncwarp();
        tc::fence_after_sync();
        tc::tmem_dealloc(sy.tmem_base, TMEM_COLS);
    }
}

}  // namespace rlt
}  // namespace vec
#endif
