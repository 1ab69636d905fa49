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
// Two forms: a block by itself with tiles of 128 tokens, and a pair of blocks (cta_group::2) with tiles of 256, in which each
// block holds its 128 tokens' keys and half of the map's rows: 32 KB instead of 48 for 64 channels of a step, two thirds of the
// traffic into shared memory, which the products' own reads share.
//
// What bounds it is how soon a step's operands and products follow the last ones.  A thread that waits for its copies and fences
// them for the tensor cores waits for all that it has in flight, the next stages' copies among them: with eight warps filling
// every stage together, a step took the latency of memory (245 us for 16 layers of 4914 listed tokens and 8 heads).  So every
// stage has a loader warp of its own, which has nothing else in flight: 176 us, and 180 in pairs.  There the issue of the products
// was the longest chain of a step (see the MMA role): 154 us from start to end, 143 of them behind the selection that it waits for (by
// single blocks 161), of which the products need 75 at the tensor rate, 104 at the rate of a library product.  That is at 1965 MHz: a loop
// of these calls settles at 1340 MHz under the 1000 W cap, 173 us behind the selection.  The products take two output heads at a time (a
// third fewer bytes than head by head), and the value rows go straight to the epilogue's registers.
//
// Persistent groups (blocks or pairs, one block per multiprocessor) own equal contiguous ranges of the sequence of items (tile, pair
// of output heads), which balances better than whole tiles: 624 tiles are 4.2 a block.  A tile cut by the end of a range is finished
// by the next group: both add their share to eps, which starts at zero (two addends: the order does not matter).
//   a warp a stage   loaders: gathers of the K rows of a step (cp.async, written in the 128-byte-swizzled operand layout) and the W
//                    load (TMA)
//   one warp         MMA issuer, TMEM owner (two 256-column accumulators: the epilogue of a pair runs under the next one)
//   four warps       epilogue: thread = row; its value row comes in 32-byte loads (16-byte ones where it has to), a head ahead
#ifndef VECTOR_RESIDUAL_LAYER_TC_CUH_
#define VECTOR_RESIDUAL_LAYER_TC_CUH_

#include "cluster.cuh"
#include "common.cuh"
#include "internal.h"
#include "residual_tc.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace vec {
namespace rlt {

using rtc::BOX_BYTES;
using rtc::TILE;

constexpr int EPI_WARPS = 4;
constexpr int TMEM_COLS = 512;
// CTAS blocks share a tile of 128 CTAS tokens; a stage holds 64 channels of: this block's 128 keys of one head | its share of the
// map's rows of two output heads.
template <int CTAS> struct LCfg {
    static constexpr int STAGES = CTAS == 2 ? 6 : 4;
    static constexpr int STAGE_BYTES = (CTAS == 2 ? 2 : 3) * BOX_BYTES;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
    static constexpr int LOADER_WARPS = STAGES;                         // a warp for every stage
    static constexpr int THREADS = 32 * (LOADER_WARPS + 1 + EPI_WARPS);
    static constexpr int TOKENS = 128 * CTAS;
};

struct Params {
    int UL, L, Hkv, n_idx, tpu;      // (sequence, layer) units, layers, KV heads, rows per unit, tiles per unit
    int pairs;                       // ceil(Hkv / 2)
    long long N, n_items;            // keys per head, UL * tpu * pairs
};
struct Sync {
    uint64_t full[6], empty[6];
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
// 32 bytes: in one load (WIDE, the address a multiple of 32) or in two.
template <bool WIDE>
__device__ __forceinline__ void ldg32(const void* p, uint32_t (&r)[64], int at) {
    if constexpr (WIDE) {
        asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                     : "=r"(r[at]), "=r"(r[at + 1]), "=r"(r[at + 2]), "=r"(r[at + 3]), "=r"(r[at + 4]), "=r"(r[at + 5]), "=r"(r[at + 6]), "=r"(r[at + 7])
                     : "l"(p));
    } else {
#pragma unroll
        for (int h = 0; h < 8; h += 4)
            asm volatile("ld.global.v4.b32 {%0,%1,%2,%3}, [%4];\n"
                         : "=r"(r[at + h]), "=r"(r[at + h + 1]), "=r"(r[at + h + 2]), "=r"(r[at + h + 3])
                         : "l"((const unsigned char*)p + 4 * h));
    }
}

// grid: at most one block per multiprocessor and a range of at least `pairs` / 2 items for each group (so that a tile is cut once at
// most), clusters of CTAS blocks, LCfg::THREADS threads, LCfg::SMEM_BYTES dynamic shared memory.
// K, V: [UL][Hkv][N][128]; idx: [UL][n_idx]; eps: [UL][n_idx], zero; mapW: (Hkv*128 in, Hkv*128 out, L), box 64 x 128.
// WIDE: V is a multiple of 32 bytes.  The interface promises 16; rows are 256 bytes apart, so the base decides for all of them.
template <bool WIDE, int CTAS>
__global__ void __launch_bounds__(LCfg<CTAS>::THREADS, 1)
residual_layer_tc(const __nv_bfloat16* K, const __nv_bfloat16* V,
                  const __grid_constant__ CUtensorMap mapW, const int32_t* idx, const Params P,
                  float* __restrict__ eps, int* __restrict__ fault) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ Sync sy;
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;     // warp: known to be uniform
    using C = LCfg<CTAS>;
    constexpr int STAGES = C::STAGES, STAGE_BYTES = C::STAGE_BYTES, LOADER_WARPS = C::LOADER_WARPS;
    const int rank = CTAS == 2 ? (int)(blockIdx.x & 1) : 0, group = blockIdx.x / CTAS, groups = gridDim.x / CTAS;
    const long long it_lo = rtc::range_begin(group, P.n_items, groups);
    const int n_my = (int)(rtc::range_begin(group + 1, P.n_items, groups) - it_lo);
    const int H = P.Hkv;

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < STAGES; ++s) {
            tma::mbar_init(&sy.full[s], 32 + 1 + (CTAS == 2 && rank == 0 ? 1 : 0));    // a loader warp, the map's bytes, the other block's stage
            tma::mbar_init(&sy.empty[s], 1);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) { tma::mbar_init(&sy.acc_full[k], 1); tma::mbar_init(&sy.acc_empty[k], CTAS * EPI_WARPS); }
        tma::mbar_fence_init();
    }
    if (warp == LOADER_WARPS) {
        tc::tmem_alloc<CTAS>(&sy.tmem_base, TMEM_COLS);
        tc::tmem_relinquish<CTAS>();
    }
    tc::fence_before_sync();
    __syncthreads();
    if (CTAS == 2) { cl::arrive_release(); cl::wait_acquire(); }       // the peer's barriers are ready for arrivals
    tc::fence_after_sync();

    if (warp < LOADER_WARPS) {
        // ------------------------------------------------------------------ loaders
        constexpr int PASSES = 32;                                   // of four rows
        const int qc = lane & 7, rsub = lane >> 3;                  // 16-byte chunk of the 64 channels, row inside a pass
        // row 4 p + rsub of the swizzled tile: the chunk's place repeats every two passes
        const uint32_t dst0 = (uint32_t)rsub * 128u + (uint32_t)((qc ^ rsub) << 4), dst1 = (uint32_t)(rsub + 4) * 128u + (uint32_t)((qc ^ (rsub + 4)) << 4);
        int32_t rows[PASSES];                                        // this lane's rows of the tile at hand
        bool ok = true;
        if (tid == 0) tma::prefetch_map(&mapW);
        asm volatile("griddepcontrol.wait;\n" ::: "memory");      // idx is complete and visible from here on
        asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
        Cursor at = cursor_at(it_lo, P);
        uint32_t step = 0, round = 0;                                // step: of the item's first channels; round: of this warp's stage
        const uint32_t s = warp;
        unsigned char* st = smem + s * STAGE_BYTES;
        for (int i = 0; i < n_my && ok; ++i, at.next(P), step += 2 * H) {
            if (i == 0 || at.pair == 0) {
#pragma unroll
                for (int p = 0; p < PASSES; ++p) {
                    const int row = at.t * C::TOKENS + rank * TILE + p * 4 + rsub;
                    const int32_t v = row < P.n_idx ? idx[(size_t)at.ul * P.n_idx + row] : -1;
                    rows[p] = (unsigned long long)v < (unsigned long long)P.N ? v : -1;     // an index outside the unit reads as zeros
                }
            }
            const int heads = min(2, H - 2 * at.pair), layer = at.ul % P.L;
            // (input head, half of its channels) of this warp's steps in the item
            for (int hk = (int)((s + STAGES - step % STAGES) % STAGES); hk < 2 * H; hk += STAGES, ++round) {
                if (round > 0 && !tma::mbar_wait_warp(&sy.empty[s], (round - 1) & 1, fault, 81)) { ok = false; break; }
                if (lane == 0) {                                    // the blocks (h, h') of the pair's output heads
                    if constexpr (CTAS == 2) {                      // half of their rows (one head: 64, and 64 the product does not read)
                        tma::mbar_expect_tx(&sy.full[s], BOX_BYTES);
                        tma::load_3d(st + BOX_BYTES, &mapW, hk * 64, 2 * at.pair * 128 + rank * heads * 64, layer, &sy.full[s]);
                    } else {
                        tma::mbar_expect_tx(&sy.full[s], heads * BOX_BYTES);
                        for (int e = 0; e < heads; ++e)
                            tma::load_3d(st + (1 + e) * BOX_BYTES, &mapW, hk * 64, (2 * at.pair + e) * 128, layer, &sy.full[s]);
                    }
                }
                const uint32_t kdst = tma::smem_u32(st);
                const __nv_bfloat16* Ku = K + ((size_t)at.ul * H + (hk >> 1)) * P.N * 128 + (hk & 1) * 64 + qc * 8;
#pragma unroll
                for (int p = 0; p < PASSES; ++p) {
                    const bool valid = rows[p] >= 0;
                    rtc::cp_async16(kdst + (p >> 1) * 1024 + ((p & 1) ? dst1 : dst0), Ku + (valid ? (size_t)rows[p] * 128 : 0), valid ? 16u : 0u);   // zero fill past the end
                }
                rtc::cp_async_wait_all();
                rtc::fence_async_proxy();
                tma::mbar_arrive(&sy.full[s]);
            }
        }
    } else if (warp == LOADER_WARPS) {
        // ------------------------------------------------------------------ MMA issue
        // The warp walks the steps together and one lane issues: under a branch on the lane the operands' descriptors are not
        // known to be uniform, and the issue of a step's four products took 360 cycles.  Whether the next stage is full is asked
        // before this one's products go out: an answer takes 200 cycles while products read shared memory.
        asm volatile("griddepcontrol.wait;\n" ::: "memory");        // the bounded waits below time this kernel only
        const bool elected = tc::elect_one();
        const uint32_t n_steps = (uint32_t)n_my * 2 * H;
        Cursor at = cursor_at(it_lo, P);
        uint32_t step = 0, s = 0, round = 0;
        bool ok = true;
        uint32_t ready = 0;
        for (int i = 0; i < n_my && ok; ++i, at.next(P)) {
            const uint32_t buf = i & 1, use = i >> 1;
            const uint32_t idesc = H - 2 * at.pair > 1 ? tc::instr_desc(128 * CTAS, 256) : tc::instr_desc(128 * CTAS, 128);
            const uint32_t d = sy.tmem_base + buf * 256;
            if (rank == 0 && use > 0 && !tma::mbar_wait_warp<CTAS>(&sy.acc_empty[buf], (use - 1) & 1, fault, 83)) break;
            tma::acquire_pair<CTAS>();
            for (int hk = 0; hk < 2 * H; ++hk, ++step) {
                if (!__all_sync(0xffffffffu, ready) && !tma::mbar_wait_warp<CTAS>(&sy.full[s], round & 1, fault, 84)) { ok = false; break; }
                const uint32_t k_addr = tma::smem_u32(smem + s * STAGE_BYTES), w_addr = k_addr + BOX_BYTES;
                const uint32_t s_next = s + 1 == STAGES ? 0 : s + 1, round_next = round + (s + 1 == STAGES);
                ready = step + 1 < n_steps ? tma::mbar_test<CTAS>(&sy.full[s_next], round_next & 1) : 0u;
                tma::acquire_pair<CTAS>();                          // this block's loaders and, in the first block, the other's warp
                if (rank != 0) {                                    // the first block issues for both: tell it that this half is there
                    if (elected) tma::mbar_arrive_at<CTAS>(tma::block_addr<CTAS>(&sy.full[s], 0));
                } else {
                    tc::fence_after_sync();
                    if (elected) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            tc::mma_bf16<CTAS>(d, tc::smem_desc(k_addr + ks * 32), tc::smem_desc(w_addr + ks * 32), idesc, (hk > 0 || ks > 0) ? 1u : 0u);
                        tc::mma_commit<CTAS>(&sy.empty[s]);         // the stage is free once these products have read it
                        if (hk + 1 == 2 * H) tc::mma_commit<CTAS>(&sy.acc_full[buf]);
                    }
                }
                __syncwarp();
                s = s_next; round = round_next;
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
            const int row = c.t * C::TOKENS + rank * TILE + r;
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
            if (lane == 0) tma::mbar_arrive_at<CTAS>(tma::block_addr<CTAS>(&sy.acc_empty[buf], 0));
            if (last) {
                const int row = at.t * C::TOKENS + rank * TILE + r;
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
    if (CTAS == 2) { cl::arrive_release(); cl::wait_acquire(); }       // the products read the peer's stages, arrivals go to its barriers
    if (warp == LOADER_WARPS) {
        __syncwarp();
        tc::fence_after_sync();
        tc::tmem_dealloc<CTAS>(sy.tmem_base, TMEM_COLS);
    }
}

}  // namespace rlt
}  // namespace vec
#endif
