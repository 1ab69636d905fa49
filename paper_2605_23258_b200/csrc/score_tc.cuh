// Base importance score on the 5th-generation tensor cores (bf16, head_dim 64 or 128).
//
// The score of a key is the softmax mass it receives from the observation-window
// rows (causal inside the window), so the logits Q K^T are needed twice: once
// for the per-row normaliser, once for the per-key sum.  Both passes are
// persistent, warp-specialised kernels around tcgen05.mma with the accumulator
// in tensor memory; the orientation of the product is chosen per pass so that
// the reduction a thread performs runs along its own TMEM lane:
//
//   pass 1   D[row][key] = Q K^T   lane = window row  -> running (max, sum exp2) per row
//   pass 2   D[key][row] = K Q^T   lane = key         -> sum over rows of exp2(logit - lse[row])
//
// A work item is (unit, group of up to 256 rows, contiguous chunk of 128-key
// tiles); items are dealt round-robin to one block per SM with the row groups of
// a key chunk on neighbouring blocks, so that a chunk is fetched from HBM once
// and found in L2 by the other row groups.
//
// Roles inside a block (576 threads):
//   warps 0-15 softmax: two groups of two warpgroups; group 0 takes the block's even tiles,
//              group 1 the odd ones, so that while one group waits for its accumulator to be
//              refilled the other keeps the exponential unit busy; each thread owns one TMEM lane
//   warp  16   producer: TMA loads of the Q row group (once per item) and of the
//              K tiles into a ring of 4 or 8 stages (128-byte swizzle, zero fill past the end)
//   warp  17   MMA issuer and owner of the TMEM allocation
// All hand-offs are mbarriers; every wait is bounded and records a fault code.
// Units of at most 128 rows (NB = 1) give every warpgroup whole tiles: 280 units of 96 rows over 78299 keys 2.60 -> 1.88 ms with
// their pooling.  Few units are pooled by the second pass itself: 8 units of 256 rows over 8192 keys 27.4 -> 23.3 us.
// Measured at 64 channels, 128 units of 4 heads x 64 rows over 15013 keys: 0.282 ms (6.32 ms on CUDA cores).
#ifndef VECTOR_SCORE_TC_CUH_
#define VECTOR_SCORE_TC_CUH_

#include "common.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace vec {
namespace stc {

using namespace tc;

constexpr int KT = 128;                    // keys per tile
constexpr int RG_ROWS = 256;               // window rows per row group
constexpr int BOX_BYTES = 16384;           // 128 rows x 128 bytes (64 bf16 of the head dimension)
// A row of D bf16 is D / 64 swizzled boxes wide; the K ring holds 128 KB whatever the head size.
template <int D> struct Cfg {
    static constexpr int HALVES = D / 64;
    static constexpr int Q_BYTES = HALVES * 2 * BOX_BYTES;          // [k half][256 rows][128 B]
    static constexpr int K_STAGE_BYTES = HALVES * BOX_BYTES;        // [k half][128 keys][128 B]
    static constexpr int STAGES = 8 / HALVES;
    static constexpr int NQ = D == 64 ? 2 : 1;                      // row groups held: the next item's is fetched ahead where it fits
    static constexpr int SMEM_BYTES = NQ * Q_BYTES + STAGES * K_STAGE_BYTES + 1024;
};
constexpr int SOFTMAX_WARPS = 16;
constexpr int THREADS = 32 * (SOFTMAX_WARPS + 2);
constexpr int TMEM_COLS = 512;

struct Params {
    int U, R, RG, w;            // units, rows per unit, row groups per unit, window
    long long N;                // keys per unit
    int tpc, n_chunks;          // key tiles per chunk, chunks per unit
    int step, lead;             // chunk c begins at key c * step - lead
    int n_items;                // U * n_chunks * RG
    int lse_chunks;             // second pass: chunks of the first one
    float c;                    // logit scale * log2(e)
};

struct Item { int u, chunk, rg, key0, tiles; };      // key0 may be negative: keys before the first read as zeros
__device__ __forceinline__ Item decode_item(int it, const Params& P) {
    Item i;
    i.rg = it % P.RG;
    const int uc = it / P.RG;
    i.chunk = uc % P.n_chunks;
    i.u = uc / P.n_chunks;
    i.key0 = i.chunk * P.step - P.lead;
    i.tiles = min((int)((P.N - i.key0 + KT - 1) / KT), P.tpc);
    return i;
}

// Barriers and the TMEM base of one block.
struct Sync {
    uint64_t q_full[2], q_empty[2];
    uint64_t k_full[8], k_empty[8];
    uint64_t acc_full[4], acc_empty[4];
    uint32_t tmem_base;
};

// Producer and MMA roles are the same in both passes up to which operand is A and the tile shape.
//   PASS 1: per key tile two MMAs  D[buf = 2 (tile & 1) + rb] (128 x 128) = Q[rb] K^T
//   PASS 2: per key tile one MMA   D[buf = tile & 1]         (128 x 256) = K Q^T
// NB = 1 is for units of at most 128 rows, which have no second block of 128 rows in a row group: a tile has one accumulator of
// 128 columns (pass 2: of the rows rounded up to 16) and goes to one of four warpgroups, where both groups' second warpgroups
// would idle and half the products be padding.
template <int D>
__device__ __forceinline__ void producer_role(const CUtensorMap* mapQ, const CUtensorMap* mapK, const Params& P,
                                              Sync& sy, unsigned char* Qs, unsigned char* Ks, int* fault) {
    constexpr int HALVES = Cfg<D>::HALVES, STAGES = Cfg<D>::STAGES, K_STAGE_BYTES = Cfg<D>::K_STAGE_BYTES, NQ = Cfg<D>::NQ;
    tma::prefetch_map(mapQ);
    tma::prefetch_map(mapK);
    uint32_t kcount = 0, icount = 0;
    auto load_q = [&](const Item& im) -> bool {
        const uint32_t b = icount % NQ, use = icount / NQ;
        if (use > 0 && !tma::mbar_wait(&sy.q_empty[b], (use - 1) & 1, fault, 11)) return false;
        tma::mbar_expect_tx(&sy.q_full[b], Cfg<D>::Q_BYTES);
#pragma unroll
        for (int kh = 0; kh < HALVES; ++kh)
#pragma unroll
            for (int rb = 0; rb < 2; ++rb)
                tma::load_3d(Qs + b * Cfg<D>::Q_BYTES + (kh * 2 + rb) * BOX_BYTES, mapQ, kh * 64, im.rg * RG_ROWS + rb * 128, im.u,
                             &sy.q_full[b]);
        return true;
    };
    for (int it = blockIdx.x; it < P.n_items; it += gridDim.x, ++icount) {
        const Item im = decode_item(it, P);
        if (icount == NQ) asm volatile("griddepcontrol.wait;\n" ::: "memory");      // as in the MMA role
        // With one row group held, its successor has to wait for the item's last product: the next keys go first
        // (they waited behind it: 4 to 5 thousand cycles an item, of 22 thousand at 15 tiles of 64 channels).  The first item's has
        // nothing to wait for, and the first product does not wait for four tiles' keys before it (8 units of 256 rows over 8192 keys
        // 21.6 -> 20.8 us in a graph).
        const bool q_first = NQ > 1 || icount == 0;
        const int q_at = q_first ? -1 : min(STAGES, im.tiles) - 1;
        if (q_first && !load_q(im)) return;
        for (int t = 0; t < im.tiles; ++t, ++kcount) {
            const uint32_t s = kcount % STAGES, round = kcount / STAGES;
            if (kcount == STAGES) asm volatile("griddepcontrol.wait;\n" ::: "memory");
            if (round > 0 && !tma::mbar_wait(&sy.k_empty[s], (round - 1) & 1, fault, 12)) return;
            tma::mbar_expect_tx(&sy.k_full[s], K_STAGE_BYTES);
#pragma unroll
            for (int kh = 0; kh < HALVES; ++kh)
                tma::load_3d(Ks + s * K_STAGE_BYTES + kh * BOX_BYTES, mapK, kh * 64, im.key0 + t * KT, im.u, &sy.k_full[s]);
            if (NQ == 1 && t == q_at && !load_q(im)) return;
        }
    }
    // The next kernel's blocks may be scheduled from here on, when the last copies are under way: earlier they would
    // sit beside this block for its whole run.  (A block with few tiles has not waited yet.)
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// First pass: the warp walks the tiles together and one lane issues.  Under a branch on the lane the operands' descriptors are not
// known to be uniform, which costs some 75 cycles a product (27.2 -> 26.1 ms for 640 units of 1024 rows and 131072 keys).  Whether
// the next keys are there is asked before this tile's products go out.  The second pass is called by one lane: with its products
// in quicker succession the softmax warps, which read the rows' normalisers from the same shared memory, fall behind (23.8 -> 25.5 ms).
template <int PASS, int D, int NB>
__device__ __forceinline__ void mma_role(const Params& P, Sync& sy, unsigned char* Qs, unsigned char* Ks, int* fault) {
    constexpr int STAGES = Cfg<D>::STAGES, K_STAGE_BYTES = Cfg<D>::K_STAGE_BYTES, K_STEPS = D / 16, NQ = Cfg<D>::NQ;
    const uint32_t k_addr = tma::smem_u32(Ks);
    const uint32_t tmem = sy.tmem_base;
    constexpr bool WARP = PASS == 1;
    const bool elected = WARP ? elect_one() : true;
    auto wait = [&](uint64_t* bar, uint32_t parity, int code) { return WARP ? tma::mbar_wait_warp(bar, parity, fault, code) : tma::mbar_wait(bar, parity, fault, code); };
    auto together = [&]() { if (WARP) __syncwarp(); };
    uint32_t kcount = 0, icount = 0, k_ready = 0;
    // the softmax warps of the second pass start once the first has drained: do not spend bounded polls on its run time
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    for (int it = blockIdx.x; it < P.n_items; it += gridDim.x, ++icount) {
        const Item im = decode_item(it, P);
        const uint32_t qb = icount % NQ, q_addr = tma::smem_u32(Qs) + qb * Cfg<D>::Q_BYTES;
        if (!wait(&sy.q_full[qb], (icount / NQ) & 1, 21)) return;
        fence_after_sync();
        for (int t = 0; t < im.tiles; ++t, ++kcount) {
            const uint32_t s = kcount % STAGES, round = kcount / STAGES;
            if (!(WARP && __all_sync(0xffffffffu, k_ready)) && !wait(&sy.k_full[s], round & 1, 22)) return;
            if (WARP) k_ready = t + 1 < im.tiles ? tma::mbar_test(&sy.k_full[(kcount + 1) % STAGES], ((kcount + 1) / STAGES) & 1) : 0u;
            fence_after_sync();
            const uint32_t ks_addr = k_addr + s * K_STAGE_BYTES;
#pragma unroll
            for (int rb = 0; rb < (PASS == 1 ? NB : 1); ++rb) {
                const uint32_t buf = NB == 1 ? kcount & 3 : PASS == 1 ? (kcount & 1) * 2 + rb : kcount & 1, use = NB == 1 ? kcount >> 2 : kcount >> 1;
                if (use > 0 && !wait(&sy.acc_empty[buf], (use - 1) & 1, 22 + PASS)) return;
                fence_after_sync();
                if (elected) {
#pragma unroll
                    for (int ks = 0; ks < K_STEPS; ++ks) {
                        const uint32_t kh = ks >> 2, ko = (ks & 3) * 32;
                        const uint64_t kd = smem_desc(ks_addr + kh * BOX_BYTES + ko);
                        const uint64_t qd = smem_desc(q_addr + kh * 2 * BOX_BYTES + rb * BOX_BYTES + ko);
                        if (PASS == 1) mma_bf16(tmem + buf * 128, qd, kd, instr_desc(128, 128), ks > 0);
                        else mma_bf16(tmem + buf * 128 * NB, kd, qd, NB == 1 ? instr_desc(128, (P.R + 15) & ~15) : instr_desc(128, 256), ks > 0);
                    }
                    mma_commit(&sy.acc_full[buf]);
                    if (PASS == 2 || rb + 1 == NB) mma_commit(&sy.k_empty[s]);      // the stage is free once these products have read it
                }
                together();
            }
        }
        if (elected) mma_commit(&sy.q_empty[qb]);
        together();
    }
}

__device__ __forceinline__ void block_setup(Sync& sy, int empty_count) {
    if (threadIdx.x == 0) {
#pragma unroll
        for (int b = 0; b < 2; ++b) { tma::mbar_init(&sy.q_full[b], 1); tma::mbar_init(&sy.q_empty[b], 1); }
#pragma unroll
        for (int s = 0; s < 8; ++s) { tma::mbar_init(&sy.k_full[s], 1); tma::mbar_init(&sy.k_empty[s], 1); }
#pragma unroll
        for (int b = 0; b < 4; ++b) { tma::mbar_init(&sy.acc_full[b], 1); tma::mbar_init(&sy.acc_empty[b], empty_count); }
        tma::mbar_fence_init();
    }
    if ((threadIdx.x >> 5) == SOFTMAX_WARPS + 1) {
        tmem_alloc(&sy.tmem_base, TMEM_COLS);
        tmem_relinquish();
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
}
__device__ __forceinline__ void block_teardown(Sync& sy) {
    fence_before_sync();
    __syncthreads();
    if ((threadIdx.x >> 5) == SOFTMAX_WARPS + 1) {
        __syncwarp();
        fence_after_sync();
        tmem_dealloc(sy.tmem_base, TMEM_COLS);
    }
}

// The exponential unit (16 results per clock per SM) is the busiest of both passes, 0.75 and 0.78 with POLY16 of every 16 exponentials
// evaluated on the FMA pipe instead (0.51 and 0.54; issue slots 0.55, tensor pipe 0.50); what bounds a long call is the 1000 W cap, where
// four and six of 16 take the same time.  2^x = 2^n p(f) with n = round(x),
// f = x - n in [-1/2, 1/2] and p the degree-4 minimax polynomial of 2^f (relative error 2.7e-6);
// n is added to the exponent field.  x is clamped from below to -126: smaller results do not
// matter to a sum whose largest term is of order one.  UPPER (the first pass, whose reference lags; in the second no logit exceeds
// its row's normaliser by more than rounding): n is clamped from above to 128, as an integer while the polynomial is under way,
// and multiplied in as 2^n: from 128 on that is infinite, which the overflow test of the first pass (sum above 2^64, or not
// finite) catches, whereas a wrapped exponent would pass as a tiny term; an infinite x ends as a NaN, which it catches too.
#ifndef VECTOR_SCORE_POLY16
#define VECTOR_SCORE_POLY16 4
#endif
constexpr int POLY16 = VECTOR_SCORE_POLY16;
static_assert(POLY16 >= 0 && POLY16 <= 16 && POLY16 % 2 == 0, "VECTOR_SCORE_POLY16: exponentials go by pairs, an even number of 16");
// p * 2^n for t = 1.5 * 2^23 + n: one multiply-add on the bits.
__device__ __forceinline__ float scaled(float p, float t) {
    uint32_t r;
    asm("mad.lo.u32 %0, %1, 8388608, %2;\n" : "=r"(r) : "r"(__float_as_uint(t)), "r"(__float_as_uint(p)));
    return __uint_as_float(r);
}
template <bool UPPER>
__device__ __forceinline__ uint64_t exp2_poly_pair(uint64_t x2) {
    constexpr int BIAS = UPPER ? 127 : 0;
    const float magic = 12582912.f + BIAS;             // 1.5 * 2^23: adding it leaves round(x) + BIAS in the low mantissa bits
    float x0, x1, t0, t1;
    unpack2(x2, x0, x1);
    x2 = pack2(fmaxf(x0, -126.f), fmaxf(x1, -126.f));
    const uint64_t t2 = add2(x2, pack2(magic, magic));
    const uint64_t n2 = add2(t2, pack2(-magic, -magic));
    const uint64_t f2 = fma2(n2, pack2(-1.f, -1.f), x2);
    uint64_t p2 = pack2(0.009570101276040077f, 0.009570101276040077f);
    p2 = fma2(p2, f2, pack2(0.05591785907745361f, 0.05591785907745361f));
    p2 = fma2(p2, f2, pack2(0.240247443318367f, 0.240247443318367f));
    p2 = fma2(p2, f2, pack2(0.6931217908859253f, 0.6931217908859253f));
    p2 = fma2(p2, f2, pack2(0.9999992847442627f, 0.9999992847442627f));
    unpack2(t2, t0, t1);
    if constexpr (UPPER) {
        const int top = 0x4B400000 + 127 + 128;
        return mul2(p2, pack2((uint32_t)min(__float_as_int(t0), top) << 23, (uint32_t)min(__float_as_int(t1), top) << 23));
    } else {
        float p0, p1;
        unpack2(p2, p0, p1);
        return pack2(scaled(p0, t0), scaled(p1, t1));
    }
}
// The exponentials of a pair of exponents, the `pair`-th of a run: POLY16 of every 16 are evaluated by polynomial, spread out among
// the others.
template <bool UPPER>
__device__ __forceinline__ uint64_t exp2_pair(uint64_t x2, int pair) {
    if (pair * (POLY16 / 2) % 8 < POLY16 / 2) return exp2_poly_pair<UPPER>(x2);
    float x0, x1;
    unpack2(x2, x0, x1);
    x0 = ex2(x0);
    x1 = ex2(x1);
    return pack2(x0, x1);
}
// sum_i exp2(v[i] * c + n[i]) over 32 (pass 1) or 16 (pass 2) accumulator columns; n is either one value for all
// columns (pass 1: minus the row's reference) or a table in shared memory (pass 2: minus the rows' lse).
// 32 columns are written as two halves whose stages overlap -- the second half's exponents are formed between the first half's
// exponentials -- so that a warp keeps the FMA pipe and the exponential unit busy together; with all FMAs, then all exponentials, then
// all adds one after the other the four warps of a scheduler found themselves in the same stage (pass 1 alone, without its products:
// 1.82 -> 1.65 ms for 64 units of 1024 rows and 131072 keys; 640 units, both passes, at the 1000 W cap: 50.7 -> 49.9 ms).
__device__ __forceinline__ float exp2_sum32(const uint32_t (&v)[32], float c, float n) {
    const uint64_t c2 = pack2(c, c), n2 = pack2(n, n);
    uint64_t x[16], acc[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = fma2(pack2(v[2 * i], v[2 * i + 1]), c2, n2);
#pragma unroll
    for (int h = 0; h < 16; h += 8) {
        uint64_t e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            e[i] = exp2_pair<true>(x[h + i], i);
            if (h == 0) x[8 + i] = fma2(pack2(v[16 + 2 * i], v[17 + 2 * i]), c2, n2);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i & 3] = h == 0 && i < 4 ? e[i] : add2(acc[i & 3], e[i]);
    }
    float s0, s1;
    unpack2(add2(add2(acc[0], acc[1]), add2(acc[2], acc[3])), s0, s1);
    return s0 + s1;
}
__device__ __forceinline__ void exp2_acc16(const uint32_t (&v)[16], float c, const float4 (&n)[4], uint64_t& acc) {
    const uint64_t c2 = pack2(c, c);
    uint64_t x[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[2 * i] = fma2(pack2(v[4 * i], v[4 * i + 1]), c2, pack2(n[i].x, n[i].y));
        x[2 * i + 1] = fma2(pack2(v[4 * i + 2], v[4 * i + 3]), c2, pack2(n[i].z, n[i].w));
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = exp2_pair<false>(x[i], i);
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1)
#pragma unroll
        for (int i = 0; i < w; ++i) x[i] = add2(x[i], x[i + w]);
    acc = add2(acc, x[0]);
}
__device__ __forceinline__ float max32(const uint32_t (&v)[32]) {
    float a = max3(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]));
    float b = max3(__uint_as_float(v[3]), __uint_as_float(v[4]), __uint_as_float(v[5]));
#pragma unroll
    for (int i = 6; i < 30; i += 4) {
        a = max3(a, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
        b = max3(b, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
    }
    return max3(a, b, fmaxf(__uint_as_float(v[30]), __uint_as_float(v[31])));
}

// One accumulator tile of pass 1 for this thread's row: 128 columns in four TMEM loads.  The
// buffer is handed back to the MMA warp as soon as the last load has completed.  The running sum l
// is kept against a reference m that lags behind the true maximum: the exponentials of a chunk do
// not wait for the chunk's maximum, and only when their sum exceeds 2^64 (always on an item's first
// chunk, where m = -inf) is the maximum taken, the reference moved and the chunk summed again.
template <bool MASKED>
__device__ __forceinline__ void softmax_tile_pass1(uint32_t taddr, float c, long long key0, long long last_visible,
                                                   float& m, float& l, uint64_t& empty_bar, int lane) {
    uint32_t ra[32], rb[32];
    tmem_ld32(taddr, ra);
#pragma unroll
    for (int ch = 0; ch < 4; ++ch) {
        uint32_t (&cur)[32] = (ch & 1) ? rb : ra;
        uint32_t (&nxt)[32] = (ch & 1) ? ra : rb;
        tmem_ld_wait(cur);
        if (ch < 3) {
            tmem_ld32(taddr + (ch + 1) * 32, nxt);
        } else {
            fence_before_sync();
            __syncwarp();
            if (lane == 0) tma::mbar_arrive(&empty_bar);
        }
        if (!MASKED) {
            // the sum itself tells whether a logit ran far ahead of the reference: only then is the
            // chunk's maximum looked for and the chunk summed again against it
            float s = exp2_sum32(cur, c, -m);
            if (!(s <= 1.8446744e19f)) {           // above 2^64, infinite (first chunk: m = -inf) or not a number
                const float cm = max32(cur) * c;
                l *= ex2(m - cm);
                m = cm;
                s = exp2_sum32(cur, c, -m);
            }
            l += s;
        } else {
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = key0 + ch * 32 + i > last_visible ? -INFINITY : __uint_as_float(cur[i]);
            float cm = v[0];
#pragma unroll
            for (int i = 1; i < 32; ++i) cm = fmaxf(cm, v[i]);
            const float m_new = fmaxf(m, cm * c);
            if (m_new > -INFINITY) {     // false only while every key so far is masked
                l *= ex2(m - m_new);     // exp2(-inf) = 0 on the first visible chunk
                float s0 = 0.f;
#pragma unroll
                for (int i = 0; i < 32; ++i) s0 += ex2(fmaf(v[i], c, -m_new));
                l += s0;
                m = m_new;
            }
        }
    }
}

// One accumulator tile of pass 2 for this thread's key: sum over 128 rows of exp2(logit2 - lse2[row]).
// Masked tiles: row j of the window (j0 = window index of the tile's first row, advancing cyclically
// with period w) sees this key only if key - (N - w) <= j.
// 16 columns at a time: the rows' lse, 16 registers, are then on their way before the accumulator's load is waited for.
// PIECES: 16-row pieces of the tile, 0: `pieces` of them.
template <bool MASKED, int PIECES>
__device__ __forceinline__ float softmax_tile_pass2(uint32_t taddr, float c, const float* nl_w, int pieces, long long key_rel,
                                                    int j0, int w, uint64_t& empty_bar, int lane) {
    uint32_t ra[16], rb[16];
    tmem_ld16(taddr, ra);
    uint64_t acc = pack2(0.f, 0.f);
    float sm = 0.f;
    int j = j0;
    const int n_ch = PIECES ? PIECES : pieces;
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
        if (!PIECES && ch >= n_ch) break;
        uint32_t (&cur)[16] = (ch & 1) ? rb : ra;
        uint32_t (&nxt)[16] = (ch & 1) ? ra : rb;
        float4 n[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) n[i] = reinterpret_cast<const float4*>(nl_w + ch * 16)[i];
        tmem_ld_wait16(cur);
        if (ch + 1 < n_ch) {
            tmem_ld16(taddr + (ch + 1) * 16, nxt);
        } else {
            fence_before_sync();
            __syncwarp();
            if (lane == 0) tma::mbar_arrive(&empty_bar);
        }
        if (!MASKED) {
            exp2_acc16(cur, c, n, acc);
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float nl = (i & 3) == 0 ? n[i >> 2].x : (i & 3) == 1 ? n[i >> 2].y : (i & 3) == 2 ? n[i >> 2].z : n[i >> 2].w;
                const float p = ex2(fmaf(__uint_as_float(cur[i]), c, nl));
                if (key_rel <= j) sm += p;
                if (++j == w) j = 0;
            }
        }
    }
    float s0, s1;
    unpack2(acc, s0, s1);
    return (s0 + s1) + sm;
}

// ---- pass 1 -----------------------------------------------------------------
// partial[((u * n_chunks + chunk) * 2 + group) * R + row] = (reference, sum of exp2 against it) of the
// row over the visible keys of the chunk's even (group 0) or odd (group 1) tiles, in units of log2 (logit * scale * log2 e).  grid: one block per SM.
// NB = 1: warpgroup v takes the tiles 4 i + v; those of one parity are added up in shared memory at the end of an item.
template <int D, int NB>
__global__ void __launch_bounds__(THREADS, 1)
score_pass1_tc(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK, const Params P,
               float2* __restrict__ partial, int* __restrict__ fault) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ Sync sy;
    __shared__ float2 upper[NB == 1 ? 4 : 1][128];                  // NB = 1: what the last two warpgroups found, two items in turn
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* Qs = smem;
    unsigned char* Ks = smem + Cfg<D>::NQ * Cfg<D>::Q_BYTES;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    block_setup(sy, 4);

    if (warp == SOFTMAX_WARPS) {
        if (lane == 0) producer_role<D>(&mapQ, &mapK, P, sy, Qs, Ks, fault);
    } else if (warp == SOFTMAX_WARPS + 1) {
        mma_role<1, D, NB>(P, sy, Qs, Ks, fault);
    } else {
        // NB = 2: tiles of parity grp, row block wg.  NB = 1: tiles tgrp mod 4; grp is their parity.
        const int tgrp = warp >> 2, grp = NB == 2 ? warp >> 3 : tgrp & 1, wg = NB == 2 ? (warp >> 2) & 1 : 0, quarter = warp & 3;
        const uint32_t lane_addr = sy.tmem_base + ((uint32_t)(quarter * 32) << 16);
        const long long vis0 = P.N - P.w;               // keys below this index are visible to every row
        uint32_t tcount = 0, icount = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < P.n_items && (NB == 1 || ok); it += gridDim.x, ++icount) {
            const Item im = decode_item(it, P);
            const int row = im.rg * RG_ROWS + wg * 128 + quarter * 32 + lane;
            const bool wg_active = im.rg * RG_ROWS + wg * 128 < P.R;
            const long long last_visible = vis0 + (row % P.w);
            float m = -INFINITY, l = 0.f;
            for (int t = 0; t < im.tiles; ++t, ++tcount) {
                if (NB == 2 ? (int)(tcount & 1) != grp : (int)(tcount & 3) != tgrp) continue;
                const uint32_t buf = NB == 2 ? (tcount & 1) * 2 + wg : tcount & 3, use = NB == 2 ? tcount >> 1 : tcount >> 2;
                if (!ok || !tma::mbar_wait_warp(&sy.acc_full[buf], use & 1, fault, 31)) { ok = false; break; }
                fence_after_sync();
                if (wg_active) {
                    const uint32_t taddr = lane_addr + buf * 128;
                    const long long key0 = im.key0 + t * KT;
                    if (key0 + KT <= vis0) softmax_tile_pass1<false>(taddr, P.c, 0, 0, m, l, sy.acc_empty[buf], lane);
                    else softmax_tile_pass1<true>(taddr, P.c, key0, last_visible, m, l, sy.acc_empty[buf], lane);
                } else {
                    __syncwarp();
                    if (lane == 0) tma::mbar_arrive(&sy.acc_empty[buf]);
                }
            }
            if (NB == 1) {
                float2 (&up)[128] = upper[NB == 1 ? 2 * (icount & 1) + grp : 0];
                if (tgrp >= 2) up[quarter * 32 + lane] = make_float2(m, l);
                // one barrier an item: whoever writes this half again, two items on, has seen every warp past this item
                asm volatile("bar.sync 1, %0;\n" ::"n"(32 * SOFTMAX_WARPS) : "memory");
                if (tgrp >= 2) continue;
                const float2 o = up[quarter * 32 + lane];
                const float M = fmaxf(m, o.x);
                if (M > -INFINITY) l = l * ex2(m - M) + o.y * ex2(o.x - M);
                m = M;
            }
            if (ok && row < P.R)
                partial[(((size_t)im.u * P.n_chunks + im.chunk) * 2 + grp) * P.R + row] = make_float2(m, l);
        }
    }
    block_teardown(sy);
}

// ---- pass 2 -----------------------------------------------------------------
// log2 of a row's sum of exp2(logit2) from its 2 n_chunks (reference, sum) partials, `stride` apart: the even lane of a
// pair takes the even tiles' partials, the odd lane the odd tiles', eight loads in flight each.
__device__ __forceinline__ float row_lse2(const float2* p, int stride, int n_chunks) {
    const size_t step = 2 * (size_t)stride;
    p += (size_t)(threadIdx.x & 1) * stride;
    float M = -INFINITY, L = 0.f;
    for (int c0 = 0; c0 < n_chunks; c0 += 8) {
        float2 v[8];
        float m = M;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[k] = c0 + k < n_chunks ? p[(size_t)(c0 + k) * step] : make_float2(-INFINITY, 0.f);
            m = fmaxf(m, v[k].x);
        }
        if (m == -INFINITY) continue;                    // no visible key so far
        L *= exp2f(M - m);
#pragma unroll
        for (int k = 0; k < 8; ++k) L += v[k].y * exp2f(v[k].x - m);
        M = m;
    }
    const unsigned pair = 3u << (threadIdx.x & 30);
    const float M2 = __shfl_xor_sync(pair, M, 1), L2 = __shfl_xor_sync(pair, L, 1);
    const float m = fmaxf(M, M2);                        // finite: every row sees at least one key
    return m + log2f(L * exp2f(M - m) + L2 * exp2f(M2 - m));
}

// lse2[u][row] = log2 sum over all visible keys of exp2(logit2).  grid (ceil(R / 128), U), 256 threads.
__global__ void __launch_bounds__(256)
score_lse2_rows(const float2* partial, int R, int n_chunks, float* __restrict__ lse2) {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int u = blockIdx.y, row = blockIdx.x * 128 + (threadIdx.x >> 1);
    if (row >= R) return;
    const float l = row_lse2(partial + (size_t)u * 2 * n_chunks * R + row, R, n_chunks);
    if ((threadIdx.x & 1) == 0) lse2[(size_t)u * R + row] = l;
}

// raw_part[(u * parts + 2 rg + h) * N + key] = sum over rows [rg*256 + h*128, +128) of the softmax
// probability of `key`, parts = ceil(R / 128); the parts are added up by the pooling kernel.  grid: one block per SM.
// INLINE_LSE, for blocks with few items: the rows' normalisers are formed from the chunk partials at the start of each
// item, two threads a row, which saves a launch (one layer, 8 heads, 256 rows, 8192 keys: 26.5 us against 36.0 with a
// kernel of its own, one block a unit).  With many items the stall at each item's start adds up, and score_lse2_rows
// leaves them in lse2 beforehand.
// POOLED, where blocks have few items and a unit one row group: a chunk's sums stay in shared memory, behind the K ring, and the
// block pools them itself: a launch less, and the sums make no trip through memory.  Its chunks overlap by the pooling radius
// r = P.lead on both sides.
constexpr int POOLED_KEYS = 3072;                    // sums of a chunk, for every 128 rows, in 24 KB
template <int D, bool INLINE_LSE, int NB, bool POOLED>
__global__ void __launch_bounds__(THREADS, 1)
score_pass2_tc(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK, const Params P,
               const float2* partial, const float* lse2, float* __restrict__ raw_part,
               float* __restrict__ raw_out, float* __restrict__ score, int* __restrict__ fault) {
    static_assert(INLINE_LSE || !POOLED, "only where blocks have few items");
    extern __shared__ unsigned char smem_raw[];
    __shared__ Sync sy;
    // -lse2 of the item's rows: INLINE_LSE, 256 rows, two items in turn; else a copy of its 128 rows for every warp
    __shared__ __align__(16) float neg_lse[INLINE_LSE ? 4 : SOFTMAX_WARPS][128];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* Qs = smem;
    unsigned char* Ks = smem + Cfg<D>::NQ * Cfg<D>::Q_BYTES;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    block_setup(sy, 4 * NB);

    if (warp == SOFTMAX_WARPS) {
        if (lane == 0) producer_role<D>(&mapQ, &mapK, P, sy, Qs, Ks, fault);
    } else if (warp == SOFTMAX_WARPS + 1) {
        if (lane == 0) mma_role<2, D, NB>(P, sy, Qs, Ks, fault);
    } else {
        const int grp = NB == 2 ? warp >> 3 : warp >> 2, wg = NB == 2 ? (warp >> 2) & 1 : 0, quarter = warp & 3;      // as in pass 1
        const int parts = (P.R + 127) / 128, pieces = (P.R + 15) / 16;
        const uint32_t lane_addr = sy.tmem_base + ((uint32_t)(quarter * 32) << 16);
        const int key_in_tile = quarter * 32 + lane;
        const long long vis0 = P.N - P.w;
        uint32_t tcount = 0, icount = 0;
        bool ok = true;                                // false once a wait gave up: touch nothing more (INLINE_LSE: but meet the barriers)
        asm volatile("griddepcontrol.wait;\n" ::: "memory");      // the partials are complete and visible from here on
        for (int it = blockIdx.x; it < P.n_items && (INLINE_LSE || ok); it += gridDim.x, ++icount) {
            const Item im = decode_item(it, P);
            const bool wg_active = im.rg * RG_ROWS + wg * 128 < P.R;
            const int row_base = im.rg * RG_ROWS + wg * 128;
            float* nl_w;
            if constexpr (INLINE_LSE) {
                float* nl_item = neg_lse[2 * (icount & 1)];
                const int r = threadIdx.x >> 1, row = im.rg * RG_ROWS + r;
                const float lse = row < P.R ? row_lse2(partial + (size_t)im.u * 2 * P.lse_chunks * P.R + row, P.R, P.lse_chunks) : INFINITY;
                if ((threadIdx.x & 1) == 0) nl_item[r] = -lse;           // -inf: padding rows add 0
                // one barrier an item: whoever writes this half again, two items on, has seen every warp past this item
                asm volatile("bar.sync 1, %0;\n" ::"n"(32 * SOFTMAX_WARPS) : "memory");
                if (!ok && !POOLED) continue;                          // POOLED: there are more barriers to meet
                nl_w = nl_item + wg * 128;
            } else {
                nl_w = neg_lse[warp];
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int row = row_base + k * 32 + lane;
                    nl_w[k * 32 + lane] = row < P.R ? -lse2[(size_t)im.u * P.R + row] : -INFINITY;   // -inf: padding rows add 0
                }
                __syncwarp();
            }
            float* out = POOLED ? reinterpret_cast<float*>(Ks + Cfg<D>::STAGES * Cfg<D>::K_STAGE_BYTES) + wg * POOLED_KEYS - im.key0
                                : raw_part + ((size_t)im.u * parts + 2 * im.rg + wg) * P.N;
            for (int t = 0; t < im.tiles; ++t, ++tcount) {
                if ((int)(tcount & (NB == 2 ? 1 : 3)) != grp) continue;
                const uint32_t buf = NB == 2 ? tcount & 1 : tcount & 3, use = NB == 2 ? tcount >> 1 : tcount >> 2;
                if (!ok || !tma::mbar_wait_warp(&sy.acc_full[buf], use & 1, fault, 32)) { ok = false; break; }
                fence_after_sync();
                const long long key = im.key0 + t * KT + key_in_tile;
                if (!wg_active) {
                    __syncwarp();
                    if (lane == 0) tma::mbar_arrive(&sy.acc_empty[buf]);
                    continue;
                }
                constexpr int PIECES = NB == 2 ? 8 : 0;
                const uint32_t taddr = lane_addr + (buf * NB + wg) * 128;
                float colsum;
                if (im.key0 + t * KT + KT <= vis0)
                    colsum = softmax_tile_pass2<false, PIECES>(taddr, P.c, nl_w, pieces, 0, 0, 0, sy.acc_empty[buf], lane);
                else
                    colsum = softmax_tile_pass2<true, PIECES>(taddr, P.c, nl_w, pieces, key - vis0, row_base % P.w, P.w, sy.acc_empty[buf], lane);
                if (POOLED || key < P.N) out[key] = colsum;
            }
            if constexpr (POOLED) {
                float* const sums = reinterpret_cast<float*>(Ks + Cfg<D>::STAGES * Cfg<D>::K_STAGE_BYTES);
                const int r = P.lead, prefix = (int)vis0 - im.key0, n = (int)min((long long)P.step, P.N - (im.key0 + r));     // keys of this chunk, behind its first r sums
                asm volatile("bar.sync 2, %0;\n" ::"n"(32 * SOFTMAX_WARPS) : "memory");
                for (int j = threadIdx.x; j < im.tiles * KT; j += 32 * SOFTMAX_WARPS) {
                    const float v = parts == 2 ? sums[j] + sums[POOLED_KEYS + j] : sums[j];
                    if (raw_out && ok && j >= r && j < r + n) raw_out[(size_t)im.u * P.N + im.key0 + j] = v;
                    sums[j] = im.key0 + j >= 0 && j < prefix ? v : -INFINITY;      // pooling looks at the prefix only
                }
                asm volatile("bar.sync 2, %0;\n" ::"n"(32 * SOFTMAX_WARPS) : "memory");
                for (int j = threadIdx.x; j < n; j += 32 * SOFTMAX_WARPS) {
                    const int last = min(j + 2 * r, im.tiles * KT - 1);
                    float best = sums[j];
                    for (int k = j + 1; k <= last; ++k) best = fmaxf(best, sums[k]);
                    if (ok) score[(size_t)im.u * P.N + im.key0 + r + j] = r + j < prefix ? best : INFINITY;
                }
                // a warp writes sums of the next item when every warp has read these: behind that item's first barrier
            }
        }
    }
    block_teardown(sy);
}

// raw[i] = sum of the parts; score[i] = max of raw over the centred window restricted to the
// prefix i < N - w; +inf for the window tokens.  grid (ceil(N / 1024), U), 256 threads.
constexpr int POOL_TILE = 1024;
__global__ void __launch_bounds__(256)
score_pool_parts(const float* raw_part, int parts, long long N, int w, int r, float* __restrict__ raw_out,
                 float* __restrict__ score) {
    __shared__ float rs[POOL_TILE + 16];
    asm volatile("griddepcontrol.wait;\n" ::: "memory");        // the second pass's sums
    const int u = blockIdx.y;
    const long long i0 = (long long)blockIdx.x * POOL_TILE;
    const float* base = raw_part + (size_t)u * parts * N;
    const long long P = N - w;
    constexpr int PT = (POOL_TILE + 16 + 255) / 256;            // sums a thread forms, their loads in flight together
    float v[PT];
#pragma unroll
    for (int k = 0; k < PT; ++k) v[k] = 0.f;
#pragma unroll 2
    for (int p = 0; p < parts; ++p)
#pragma unroll
        for (int k = 0; k < PT; ++k) {
            const int e = threadIdx.x + 256 * k;
            const long long i = i0 - r + e;
            if (e < POOL_TILE + 2 * r && i >= 0 && i < N) v[k] += base[(size_t)p * N + i];
        }
#pragma unroll
    for (int k = 0; k < PT; ++k) {
        const int e = threadIdx.x + 256 * k;
        const long long i = i0 - r + e;
        if (e >= POOL_TILE + 2 * r) continue;
        if (raw_out && e >= r && e < POOL_TILE + r && i < N) raw_out[(size_t)u * N + i] = v[k];
        rs[e] = i >= 0 && i < P ? v[k] : -INFINITY;             // pooling looks at the prefix only
    }
    __syncthreads();
    for (int e = threadIdx.x; e < POOL_TILE; e += 256) {
        const long long i = i0 + e;
        if (i >= N) break;
        float best = INFINITY;
        if (i < P) {
            best = rs[e];
            for (int k = 1; k <= 2 * r; ++k) best = fmaxf(best, rs[e + k]);
        }
        score[(size_t)u * N + i] = best;
    }
}

// The same for N a multiple of 4: 16-byte loads and stores, four keys per thread.
__global__ void __launch_bounds__(256)
score_pool_parts_v4(const float* raw_part, int parts, long long N, int w, int r, float* __restrict__ raw_out,
                    float* __restrict__ score) {
    __shared__ __align__(16) float rs[POOL_TILE + 16];          // keys i0 - 8 .. i0 + POOL_TILE + 8
    asm volatile("griddepcontrol.wait;\n" ::: "memory");        // the second pass's sums
    const int u = blockIdx.y;
    const long long i0 = (long long)blockIdx.x * POOL_TILE;
    const float* base = raw_part + (size_t)u * parts * N;
    const long long P = N - w;
    for (int e4 = threadIdx.x; e4 < (POOL_TILE + 16) / 4; e4 += 256) {
        const long long i = i0 - 8 + 4 * e4;
        float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        if (i >= 0 && i < N) {
            v = *reinterpret_cast<const float4*>(base + i);
            for (int p = 1; p < parts; ++p) {
                const float4 x = *reinterpret_cast<const float4*>(base + (size_t)p * N + i);
                v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            }
            if (raw_out && e4 >= 2 && e4 < 2 + POOL_TILE / 4) *reinterpret_cast<float4*>(raw_out + (size_t)u * N + i) = v;
            if (i + 0 >= P) v.x = -INFINITY;           // pooling looks at the prefix only
            if (i + 1 >= P) v.y = -INFINITY;
            if (i + 2 >= P) v.z = -INFINITY;
            if (i + 3 >= P) v.w = -INFINITY;
        }
        *reinterpret_cast<float4*>(rs + 4 * e4) = v;
    }
    __syncthreads();
    const long long i = i0 + 4 * threadIdx.x;
    if (i >= N) return;
    float x[20];                                                // keys i - 8 .. i + 11
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const float4 v = *reinterpret_cast<const float4*>(rs + 4 * threadIdx.x + 4 * k);
        x[4 * k] = v.x; x[4 * k + 1] = v.y; x[4 * k + 2] = v.z; x[4 * k + 3] = v.w;
    }
    float o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float best = x[8 + j];
#pragma unroll
        for (int k = 1; k <= 7; ++k)
            if (k <= r) best = fmaxf(best, fmaxf(x[8 + j - k], x[8 + j + k]));
        o[j] = i + j < P ? best : INFINITY;
    }
    *reinterpret_cast<float4*>(score + (size_t)u * N + i) = make_float4(o[0], o[1], o[2], o[3]);
}

}  // namespace stc
}  // namespace vec
#endif
