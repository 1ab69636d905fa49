// Decode attention over the mixed cache for bf16, head_dim 64 or 128 (HBM-bound).
//
// Every K/V row is read once.  Each unit's rows are cut into tiles of 128 rows (32 KB
// at head_dim 128, 16 KB at 64) -- a retained tile = 64 keys + their 64 values, a
// key-only tile = 128 keys -- and the global tile sequence is dealt out in equal contiguous ranges to one
// persistent block per SM: the load is balanced by bytes and there is no wave tail.
//
// Inside a block one producer thread streams the tiles with TMA
// (cp.async.bulk.tensor, 128-byte swizzle, zero fill past the end of a pool)
// into slots that fill 192 KB, guarded by full/empty mbarriers.  Tiles go round-robin
// to the consumer warps, each with slots of its own (head_dim 128: three warps with two
// 32 KB slots each, tile i to warp i % 3 and slot i % 6), so a warp sees every phase of the barriers it waits on -- with a
// parity wait, a waiter that skipped a phase could take an old completion for
// the one it wants, since TMA copies land out of order.  A warp works through a
// whole tile on its own, 64 keys at a time, and never synchronises with the others:
//   S = Q K^T      head_dim / 2 m16n8k16 bf16 MMAs (eight independent accumulators), the g
//                  query heads padded to the MMA rows
//   online softmax in fp32 registers, one rescale per 64 keys (exp2, scale folded in)
//   O += P V  (retained tile)  or  A += P K  (key-only tile: the p-weighted key
//             sum that the merge step multiplies by W); P enters as bf16 hi in
//             MMA rows 0-7 and bf16 lo in rows 8-15, one MMA for both parts; at head_dim 64
//             a third part keeps all 24 bits of a weight (Cfg::PARTS)
// A warp keeps one running state (m, l, O or A) per unit and writes it as its
// partial record when it leaves the unit; a warp that met no tile of a unit the
// block touches writes an empty record.  The merge kernel combines a unit's
// records, applies W and normalises.
//
// Few units (CLUSTER): one launch does it all.  A thread block cluster owns a unit, each of its
// blocks an equal share of the unit's tiles; the warps' records stay in shared memory, a block
// combines its own, and after a cluster barrier block r merges the query heads r, r + C, ... out of
// the other blocks' shared memory and applies W.  No records in global memory, no second kernel.
// RoPE decoupling has a streaming kernel of its own (decode_rope.cuh) with the same tiles and records.
#ifndef VECTOR_DECODE_BF16_CUH_
#define VECTOR_DECODE_BF16_CUH_

#include "cluster.cuh"
#include "common.cuh"
#include "internal.h"
#include "rope.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace vec {
namespace dbf {

constexpr int KEYS = 64;                     // keys per softmax step (and per TMA box)
constexpr int BOX_BYTES = 8192;              // 64 rows x 128 bytes
// 64 channels: the softmax's reference follows the running maximum only when that has moved by more than SLACK (in powers of two):
// any reference serves weights that keep all 24 bits, and the sums are rescaled a few times instead of in every other step.
// Weights that keep sixteen bits want the running maximum itself: the largest of them is one then, and exact (with the slack, 131.4
// against 132.1 us for 512 units of 4915 rows, 128 channels, the outputs were off by up to a quarter more).
// tc::ex2 gives zero below 2^-126: next to a weight of at least 2^-SLACK that changes no fp32 sum.
constexpr float SLACK = 8.f;
template <int D, bool ROPE> struct Cfg {
    static constexpr int HALF_BYTES = 64 * 2 * D;                    // 64 rows as D / 64 swizzled boxes
    // 64 channels: everything to fp32's own precision, as CUDA cores give it.  A softmax weight and a key sum on its way through the
    // map enter as three bf16 parts, which keep their 24 bits (two keep sixteen); an MMA cuts its sums off instead of rounding them, so
    // that the sums of 32 rows and of 32 columns of the map start at zero and are added up in fp32.  With up to
    // four heads the third parts take MMA rows that nobody else uses.  Error of an fp32 output against
    // fp64, median over the heads of ten sizes of 1 to 64 layers, 8 to 512 units and up to 78642 rows: 1.1e-7 to 1.8e-7 (two parts, sums
    // in the MMAs: 1.0e-6 to 2.2e-6; CUDA cores: 1.2e-7 to 4.4e-7).  512 units, 431 MB: 82 -> 85.5 us a step with the appended row.
    static constexpr bool EXACT = D == 64;
    static constexpr int PARTS = EXACT ? 3 : 2;
    static constexpr int SLOT_BYTES = 2 * HALF_BYTES;                // retained: K | V; key-only: keys 0-63 | keys 64-127
    // With 64-channel heads a softmax step brings in half the bytes for the same softmax arithmetic: a fourth consumer
    // warp (one to a warp scheduler) makes up for it.
    // Measured: 512 units, 1639 retained + 3276 key-only rows, 431 MB: 85.5 us with the appended row = 5.0 TB/s (856 us on
    // CUDA cores).
    // With RoPE decoupling a consumer is a team (decode_rope.cuh): a score warp and some sum warps.
    // Four teams at 64 channels, of two sum warps with as many channel pairs each as the four have at 128.
    static constexpr int CONSUMER_WARPS = D == 128 ? 3 : 4, SUM_WARPS = ROPE ? D / 32 : 0;
    static constexpr int SLOTS = D == 128 ? 6 : ROPE ? 8 : 12;       // a multiple of CONSUMER_WARPS: a slot always serves the same warp
    static constexpr int THREADS = 32 * (CONSUMER_WARPS * (1 + SUM_WARPS) + 1);
    // RoPE: a step buffer: weights [16 keys][first | second parts of 8 keys][head][8 keys], EXACT: third parts alike; positions; factors
    static constexpr int STEP_THIRD = 2048, STEP_POS = STEP_THIRD + (EXACT ? 1024 : 0), STEP_ALPHA = STEP_POS + 4 * KEYS;
    static constexpr int STEP_BYTES = STEP_ALPHA + 32;
    static constexpr int P_BYTES = ROPE ? CONSUMER_WARPS * 2 * STEP_BYTES : 0;
    static constexpr int SMEM_BYTES = SLOTS * SLOT_BYTES + P_BYTES + 1024;     // + alignment slack; barriers live in static smem
    static constexpr int REC = 4 + 2 * D;                            // m, l, value-scale, pad, acc_v[D], acc_k[D]
    // CLUSTER: the warps' headers and value sums behind the slots, [CONSUMER_WARPS][g][4 + D]; a warp's key sums, [g][D], take
    // the last of its own slots once it has worked through its tiles
    static constexpr int CREC = 4 + D;
    static constexpr int CLUSTER_SMEM_BYTES = SMEM_BYTES + CONSUMER_WARPS * 8 * CREC * 4;
    static_assert(CLUSTER_SMEM_BYTES + 1024 <= 227 * 1024, "shared memory of a block, barriers included");
    static_assert(SLOTS % CONSUMER_WARPS == 0, "a slot must always be consumed by the same warp");
};
constexpr int REC = Cfg<128, false>::REC;

// How the tile sequence is dealt to blocks; the same arithmetic runs on host and device.
struct Plan {
    int n_rt, n_at, n_tiles;   // retained / key-only / all tiles per unit
    long long T;               // tiles of all units
    int B;                     // blocks
    int s_max;                 // record slots per unit
    bool narrow;               // products of T and B fit 32 bits
};
__host__ __device__ inline Plan make_plan(int U, long long n_ret, long long n_apx, int max_blocks) {
    Plan p;
    p.n_rt = (int)((n_ret + KEYS - 1) / KEYS);
    p.n_at = (int)((n_apx + 2 * KEYS - 1) / (2 * KEYS));
    p.n_tiles = p.n_rt + p.n_at;
    p.T = (long long)U * p.n_tiles;
    long long b = p.T / 2;                       // at least two tiles per block
    if (b > max_blocks) b = max_blocks;               // one persistent block per multiprocessor
    if (b > 11LL * U) b = 11LL * U;              // at most 12 record slots per unit (merge kernel limit)
    p.B = (int)(b < 1 ? 1 : b);
    p.s_max = (p.B + U - 1) / U + 1;
    p.narrow = p.T * p.B < (1LL << 32);
    return p;
}
// Block b owns the tiles [b T / B, (b+1) T / B).  A division of 64 bits takes some hundred instructions, which every thread of the
// merge went through twice a unit.
__host__ __device__ inline long long tile_begin(int b, const Plan& p) { return (long long)b * p.T / p.B; }
__host__ __device__ inline int block_of_tile(long long x, const Plan& p) {
    if (p.narrow) return (int)((((unsigned)x + 1) * (unsigned)p.B - 1) / (unsigned)p.T);
    return (int)(((x + 1) * p.B - 1) / p.T);
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
// D(16x8) += A(16x16) B(16x8) with A rows 8..15 zero: the upper accumulator half is fed zeros and
// its (zero) result parked in a scratch pair.
__device__ __forceinline__ void mma_lo8(float& c0, float& c1, float& z0, float& z1, uint32_t a0, uint32_t a2,
                                        uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%10,%10};\n"
        : "+f"(c0), "+f"(c1), "=f"(z0), "=f"(z1)
        : "r"(a0), "r"(0u), "r"(a2), "r"(0u), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                       uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The same product with fp16 operands (the keys turned back under RoPE decoupling are held in fp16).
__device__ __forceinline__ void mma_16_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                           uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Two floats to an fp16 pair, low half first; values beyond the fp16 range go to its largest finite number.
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;\n" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ float f16_lo(uint32_t v) { return __half2float(__ushort_as_half((unsigned short)(v & 0xffffu))); }
__device__ __forceinline__ float f16_hi(uint32_t v) { return __half2float(__ushort_as_half((unsigned short)(v >> 16))); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

struct Maps {
    CUtensorMap ret_k, ret_v, apx_k;     // rank 3: (D dims, pool rows, U units), box 64 x 64 x 1, 128B swizzle
};

// This block's share of the tile sequence: never empty, there are no more blocks than tiles in either form.
template <bool CLUSTER>
__device__ __forceinline__ void block_range(const Plan& pl, long long& lo, long long& hi) {
    const int b = blockIdx.x;
    if (CLUSTER) {
        const int C = (int)cl::nctas(), r = (int)cl::rank(), u = b / C;
        lo = (long long)u * pl.n_tiles + (long long)r * pl.n_tiles / C;
        hi = (long long)u * pl.n_tiles + (long long)(r + 1) * pl.n_tiles / C;
    } else {
        lo = tile_begin(b, pl);
        hi = tile_begin(b + 1, pl);
    }
}
// The producer thread: the block's tiles in order, each into the next slot.
template <int D, bool ROPE>
__device__ __forceinline__ void produce(const Maps& maps, const Plan& pl, long long gt_lo, int n_my, unsigned char* smem,
                                        uint64_t* full_bar, uint64_t* empty_bar, int* fault) {
    using C = Cfg<D, ROPE>;
    constexpr int BOXES = D / 64;
    tma::prefetch_map(&maps.ret_k); tma::prefetch_map(&maps.ret_v); tma::prefetch_map(&maps.apx_k);
    const uint64_t pol = tma::policy_evict_first();      // the cache is read once per step
    int u = (int)(gt_lo / pl.n_tiles), t = (int)(gt_lo - (long long)u * pl.n_tiles);
    for (int i = 0; i < n_my; ++i) {
        const int s = i % C::SLOTS, round = i / C::SLOTS;
        if (round > 0 && !tma::mbar_wait(&empty_bar[s], (round - 1) & 1, fault, 1)) break;
        unsigned char* st = smem + s * C::SLOT_BYTES;
        tma::mbar_expect_tx(&full_bar[s], C::SLOT_BYTES);
        if (t < pl.n_rt) {
            const int row0 = t * KEYS;
#pragma unroll
            for (int x = 0; x < BOXES; ++x) {
                tma::load_3d_hint(st + x * BOX_BYTES, &maps.ret_k, 64 * x, row0, u, &full_bar[s], pol);
                tma::load_3d_hint(st + C::HALF_BYTES + x * BOX_BYTES, &maps.ret_v, 64 * x, row0, u, &full_bar[s], pol);
            }
        } else {
            const int row0 = (t - pl.n_rt) * 2 * KEYS;
#pragma unroll
            for (int x = 0; x < BOXES; ++x) {
                tma::load_3d_hint(st + x * BOX_BYTES, &maps.apx_k, 64 * x, row0, u, &full_bar[s], pol);
                tma::load_3d_hint(st + C::HALF_BYTES + x * BOX_BYTES, &maps.apx_k, 64 * x, row0 + KEYS, u, &full_bar[s], pol);
            }
        }
        if (++t == pl.n_tiles) { t = 0; ++u; }
    }
}
// The g query heads of a unit as A fragments, rows g .. 7 zero; twice: rows 4 .. 7 the same heads as rows 0 .. 3 (g <= 4).
template <int D>
__device__ __forceinline__ void load_queries(const __nv_bfloat16* q, int unit, int g, int lane, uint32_t (&qa)[D / 16][2],
                                             bool twice) {
    const int head = twice ? (lane >> 2) & 3 : lane >> 2, tig = lane & 3;
    const uint32_t* qrow = reinterpret_cast<const uint32_t*>(q + ((size_t)unit * g + min(head, g - 1)) * D);
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        qa[ks][0] = head < g ? qrow[ks * 8 + tig] : 0u;
        qa[ks][1] = head < g ? qrow[ks * 8 + 4 + tig] : 0u;
    }
}
// The weights of a softmax step over the 64 keys at kbase (D / 64 swizzled boxes), of which nrows >= 1 are valid: sc (this
// thread: head gid, keys 8 n + 2 tig, + 1) against the new running maximum m; l follows.  Returns the factor that what
// was summed up before has to take.
template <int D>
__device__ __forceinline__ float score_step(uint32_t kbase, int nrows, float scale_log2e, const uint32_t (&qa)[D / 16][2], int lane,
                                            float& m, float& l, float (&sc)[8][2]) {
    // per-lane ldmatrix geometry (swizzle: 16-byte chunk index XOR (row & 7), rows are 128 bytes): matrices =
    // (keys 0-7|8-15) x (chunk lo|hi)
    const int tig = lane & 3, mat = lane >> 3, r8 = lane & 7;
    const uint32_t qk_row = (uint32_t)(r8 + (mat >> 1) * 8) * 128u, qk_x = (uint32_t)(((mat & 1) ^ r8) << 4);
    // ---- S = Q K^T: eight 8-key column tiles, each its own accumulator chain over the D / 16 k-steps
    float zz[2];
#pragma unroll
    for (int n = 0; n < 8; ++n) { sc[n][0] = 0.f; sc[n][1] = 0.f; }
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {          // 16 keys per ldmatrix
            uint32_t b0, b1, b2, b3;
            // k-step ks covers 16-byte chunks 2ks, 2ks+1 of the row: box ks/4, chunk (2ks)%8 (+1)
            ldsm_x4(kbase + (ks >> 2) * BOX_BYTES + j * 16 * 128 + qk_row + ((((2 * ks) & 7) << 4) ^ qk_x), b0, b1, b2, b3);
            mma_lo8(sc[2 * j][0], sc[2 * j][1], zz[0], zz[1], qa[ks][0], qa[ks][1], b0, b1);
            mma_lo8(sc[2 * j + 1][0], sc[2 * j + 1][1], zz[0], zz[1], qa[ks][0], qa[ks][1], b2, b3);
        }
    }
    // ---- online softmax over these 64 keys (row = head gid, shared by the 4 threads of a quad)
    float mx = -INFINITY;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        const int kc = n * 8 + 2 * tig;
        sc[n][0] = kc < nrows ? sc[n][0] * scale_log2e : -INFINITY;
        sc[n][1] = kc + 1 < nrows ? sc[n][1] * scale_log2e : -INFINITY;
        mx = fmaxf(mx, fmaxf(sc[n][0], sc[n][1]));
    }
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float m_new = fmaxf(m, mx);                 // finite: key 0 of the step is valid for every row
    const float alpha = tc::ex2(m - m_new);           // 0 on the first step
    float ls = 0.f;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        sc[n][0] = tc::ex2(sc[n][0] - m_new);
        sc[n][1] = tc::ex2(sc[n][1] - m_new);
        ls += sc[n][0] + sc[n][1];
    }
    l = l * alpha + ls;
    m = m_new;
    return alpha;
}
// The same for 64 channels, on packed pairs: all rows of an accumulator are kept, so that nothing is moved between the MMAs.
__device__ __forceinline__ float score_step64(uint32_t kbase, int nrows, float scale_log2e, const uint32_t (&qa)[4][2], int lane,
                                              float& m, float& l, float (&sc)[8][2]) {
    const int tig = lane & 3, mat = lane >> 3, r8 = lane & 7;
    const uint32_t row = (uint32_t)(r8 + (mat >> 1) * 8) * 128u, x = (uint32_t)(((mat & 1) ^ r8) << 4);
    float s[8][4];
#pragma unroll
    for (int n = 0; n < 8; ++n) s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t b0, b1, b2, b3;
            ldsm_x4(kbase + j * 16 * 128 + row + ((2 * ks << 4) ^ x), b0, b1, b2, b3);
            mma_16(s[2 * j], qa[ks][0], 0u, qa[ks][1], 0u, b0, b1);
            mma_16(s[2 * j + 1], qa[ks][0], 0u, qa[ks][1], 0u, b2, b3);
        }
    }
    const uint64_t c2 = tc::pack2(scale_log2e, scale_log2e);
    uint64_t v[8];
    float mx = -INFINITY;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        v[n] = tc::mul2(tc::pack2(s[n][0], s[n][1]), c2);
        tc::unpack2(v[n], sc[n][0], sc[n][1]);
    }
    if (nrows < KEYS) {
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const int kc = n * 8 + 2 * tig;
            if (kc >= nrows) sc[n][0] = -INFINITY;
            if (kc + 1 >= nrows) sc[n][1] = -INFINITY;
            v[n] = tc::pack2(sc[n][0], sc[n][1]);
        }
    }
#pragma unroll
    for (int n = 0; n < 8; ++n) mx = fmaxf(mx, fmaxf(sc[n][0], sc[n][1]));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float m_new = mx > m + SLACK ? mx : m;      // finite: key 0 of the step is valid for every row
    const float alpha = tc::ex2(m - m_new);           // 0 on the first step
    const uint64_t neg = tc::pack2(-m_new, -m_new);
    uint64_t ls[2] = {tc::pack2(0.f, 0.f), tc::pack2(0.f, 0.f)};
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        float a, b;
        tc::unpack2(tc::add2(v[n], neg), a, b);
        sc[n][0] = tc::ex2(a);
        sc[n][1] = tc::ex2(b);
        ls[n & 1] = tc::add2(ls[n & 1], tc::pack2(sc[n][0], sc[n][1]));
    }
    float l0, l1;
    tc::unpack2(tc::add2(ls[0], ls[1]), l0, l1);
    l = fmaf(l, alpha, l0 + l1);
    m = m_new;
    return alpha;
}
// The weights of keys 16 kk .. + 15 as an A fragment: first parts in MMA rows 0-7, second parts in rows 8-15.  Third parts:
// of up to four heads (twice: this thread's head is gid & 3) in rows 4-7, else in a fragment of their own (rows 8-15, third).
template <int PARTS>
__device__ __forceinline__ void weights_bf16(const float (&sc)[8][2], int kk, bool twice, int gid, uint32_t (&a)[4], uint32_t (&third)[2]) {
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        uint32_t part[PARTS];
        split_bf16(sc[2 * kk + x][0], sc[2 * kk + x][1], part);
        const bool upper = PARTS == 3 && twice && gid >= 4;
        a[2 * x] = upper ? part[PARTS - 1] : part[0];
        a[2 * x + 1] = upper ? 0u : part[1];
        third[x] = PARTS == 3 ? part[PARTS - 1] : 0u;
    }
}
// acc += P x over rows 16 kk .. + 15 of the 64 rows at vbase: D / 8 column tiles of 8 dims.  with_third: P has a third fragment.
template <int D>
__device__ __forceinline__ void accumulate_step(uint32_t vbase, int kk, const uint32_t (&a)[4], bool with_third, const uint32_t (&third)[2],
                                                float (&acc)[D / 8][4], int lane) {
    const int mat = lane >> 3, r8 = lane & 7;             // matrices = (chunk lo|hi) x (rows 0-7|8-15)
    const uint32_t pv_row = (uint32_t)(r8 + (mat & 1) * 8) * 128u, pv_x = (uint32_t)(((mat >> 1) ^ r8) << 4);
#pragma unroll
    for (int np = 0; np < D / 16; ++np) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4_t(vbase + (np >> 2) * BOX_BYTES + kk * 16 * 128 + pv_row + ((((2 * np) & 7) << 4) ^ pv_x), b0, b1, b2, b3);
        mma_16(acc[2 * np], a[0], a[1], a[2], a[3], b0, b1);
        mma_16(acc[2 * np + 1], a[0], a[1], a[2], a[3], b2, b3);
        if (with_third) {
            mma_16(acc[2 * np], 0u, third[0], 0u, third[1], b0, b1);
            mma_16(acc[2 * np + 1], 0u, third[0], 0u, third[1], b2, b3);
        }
    }
}

// The key sums of up to eight heads on their way through the map, in bf16 parts: two (sixteen mantissa bits), or three (all 24).
template <int D> struct KeySums { __align__(16) __nv_bfloat16 part[Cfg<D, false>::PARTS][8][D]; };
template <int D>
__device__ __forceinline__ void store_key_sum(KeySums<D>& ks, int head, int c, float v) {
#pragma unroll
    for (int i = 0; i < Cfg<D, false>::PARTS; ++i) {
        const __nv_bfloat16 x = __float2bfloat16_rn(v);
        ks.part[i][head][c] = x;
        v -= __bfloat162float(x);
    }
}

// Rows 16 mt .. + 15 of W times the key sums of the heads.  One warp, M = 16 output channels, N = the heads
// (padded to 8), K = D: the A fragments are read straight from the map in global memory, 16 bytes a load -- thread
// (row r, quarter t) of a warp holds columns 8 (t + 4 jj) .. + 7 of rows r and r + 8, and the k slots of MMA step
// 2 jj + h stand for columns 8 (t + 4 jj) + 4 h .. + 3, which the B fragments follow; the map's elements are bf16 as stored.
// Three parts: the MMAs of the first start at zero and are added up in fp32, as the sums before them are (Cfg::EXACT).
// d[0], d[1]: row lane / 4 of the 16, heads 2 (lane % 4) and + 1; d[2], d[3]: row lane / 4 + 8.
template <int D>
__device__ __forceinline__ void map_fragments(const __nv_bfloat16* W, int mt, uint4 (&A)[D / 16], int lane) {
    constexpr int PIECES = D / 8;                                    // 16-byte pieces of a row of W
    const int row = lane >> 2, quarter = lane & 3;
    const uint4* Wu = reinterpret_cast<const uint4*>(W);
#pragma unroll
    for (int jj = 0; jj < D / 32; ++jj) {
        A[2 * jj + 0] = Wu[(16 * mt + row) * PIECES + quarter + 4 * jj];
        A[2 * jj + 1] = Wu[(16 * mt + row + 8) * PIECES + quarter + 4 * jj];
    }
}
template <int D>
__device__ __forceinline__ void map_product(const uint4 (&A)[D / 16], const KeySums<D>& ks, float (&d)[4], int lane) {
    constexpr int PARTS = Cfg<D, false>::PARTS;
    const int row = lane >> 2, quarter = lane & 3;
    float small[4] = {0.f, 0.f, 0.f, 0.f};
    d[0] = d[1] = d[2] = d[3] = 0.f;
#pragma unroll
    for (int jj = 0; jj < D / 32; ++jj) {
        const uint4 r0 = A[2 * jj], r1 = A[2 * jj + 1];
        const int col = 8 * (quarter + 4 * jj);
        uint4 b[PARTS];
#pragma unroll
        for (int i = 0; i < PARTS; ++i) b[i] = *reinterpret_cast<const uint4*>(&ks.part[i][row][col]);      // B column = head `row`
        if constexpr (PARTS == 3) {
            float t[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
            mma_16(t[0], r0.x, r1.x, r0.y, r1.y, b[0].x, b[0].y);
            mma_16(t[1], r0.z, r1.z, r0.w, r1.w, b[0].z, b[0].w);
#pragma unroll
            for (int i = 2; i > 0; --i) {
                mma_16(small, r0.x, r1.x, r0.y, r1.y, b[i].x, b[i].y);
                mma_16(small, r0.z, r1.z, r0.w, r1.w, b[i].z, b[i].w);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) d[e] += t[0][e] + t[1][e];
        } else {
#pragma unroll
            for (int i = 0; i < PARTS; ++i) mma_16(d, r0.x, r1.x, r0.y, r1.y, b[i].x, b[i].y);
#pragma unroll
            for (int i = 0; i < PARTS; ++i) mma_16(d, r0.z, r1.z, r0.w, r1.w, b[i].z, b[i].w);
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) d[e] += small[e];
}
// The same, of n heads, into pw[head][row].
template <int D>
__device__ __forceinline__ void map_rows(const __nv_bfloat16* W, int mt, int n, const KeySums<D>& ks, float (&pw)[8][D], int lane) {
    const int row = lane >> 2, quarter = lane & 3;
    uint4 A[D / 16];
    float d[4];
    map_fragments<D>(W, mt, A, lane);
    map_product<D>(A, ks, d, lane);
    if (2 * quarter < n) { pw[2 * quarter][16 * mt + row] = d[0]; pw[2 * quarter][16 * mt + row + 8] = d[2]; }
    if (2 * quarter + 1 < n) { pw[2 * quarter + 1][16 * mt + row] = d[1]; pw[2 * quarter + 1][16 * mt + row + 8] = d[3]; }
}

// The last part of the CLUSTER form: combines the records of a unit, which its cluster's blocks hold in shared
// memory, applies W and writes out.  Every warp of every block of the cluster calls it, converged; the warps come from
// different roles, so the block-wide barrier is the numbered one below.  recs: this block's [CONSUMER_WARPS][g][CREC] (header:
// m, l, value-scale, whether there are key sums); room: the slots, which nobody reads any more -- a MergeShared at their
// start, the warps' key sums in their last CONSUMER_WARPS.
template <int NT> __device__ __forceinline__ void merge_sync() { asm volatile("bar.sync 1, %0;\n" ::"n"(NT) : "memory"); }

constexpr int MAX_CLUSTER = 16;
template <int D> struct MergeShared {
    __align__(16) float comb[8 * (4 + 2 * D)];                        // this block's sums per head, read by the whole cluster
    KeySums<D> ks;                                                    // key sums of the heads this block merges
    float avs[8][D], pw[8][D];                                        // their value sums; W times the key sums
    float fac[8][MAX_CLUSTER], Ls[8];                                 // factor of every block's sums; sum of the weights
};
template <int D, bool ROPE>
__device__ __forceinline__ void cluster_merge(const float* recs, unsigned char* room, const __nv_bfloat16* Wu, int g,
                                              void* __restrict__ out_u, bool out_f32) {
    using C = Cfg<D, ROPE>;
    constexpr int REC = C::REC, CREC = C::CREC, CW = C::CONSUMER_WARPS, NT = C::THREADS, V4 = 2 * D / 4;
    static_assert(sizeof(MergeShared<D>) <= (C::SLOTS - CW) * C::SLOT_BYTES, "the key sums lie behind it");
    MergeShared<D>& S = *reinterpret_cast<MergeShared<D>*>(room);
    auto& comb = S.comb; auto& fac = S.fac; auto& Ls = S.Ls; auto& ks = S.ks; auto& avs = S.avs; auto& pw = S.pw;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nblk = (int)cl::nctas(), rank = (int)cl::rank();
    merge_sync<NT>();                                                 // the warps' records are written
    for (int e = tid; e < g * V4; e += NT) {
        const int a = e / V4, c4 = e - a * V4;
        float m[CW], M = -INFINITY, L = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < CW; ++w) { m[w] = recs[(w * g + a) * CREC]; M = fmaxf(M, m[w]); }
#pragma unroll
        for (int w = 0; w < CW; ++w) {
            if (m[w] == -INFINITY) continue;                          // a warp without tiles: its sums are not written
            const float* r = recs + (w * g + a) * CREC;
            float f = __expf(m[w] - M);
            L = fmaf(f, r[1], L);
            const float* src = r + 4 + 4 * c4;
            if (c4 < D / 4) f *= r[2];                                // the values were parked at another reference
            else if (r[3] == 0.f) continue;                           // no key-only tile
            else src = reinterpret_cast<const float*>(room + (C::SLOTS - CW + w) * C::SLOT_BYTES) + a * D + 4 * (c4 - D / 4);
            const float4 x = *reinterpret_cast<const float4*>(src);
            acc.x = fmaf(f, x.x, acc.x); acc.y = fmaf(f, x.y, acc.y); acc.z = fmaf(f, x.z, acc.z); acc.w = fmaf(f, x.w, acc.w);
        }
        if (c4 == 0) { comb[a * REC] = M; comb[a * REC + 1] = L; }
        *reinterpret_cast<float4*>(comb + a * REC + 4 + 4 * c4) = acc;
    }
    for (int e = tid; e < 8 * D; e += NT) store_key_sum(ks, e / D, e % D, 0.f);
    __syncwarp();
    cl::arrive_release();
    cl::wait_acquire();                                               // every block's sums are ready
    const int mine = rank < g ? (g - rank + nblk - 1) / nblk : 0;     // heads rank, rank + nblk, ...
    const uint32_t comb_addr = tma::smem_u32(comb);
    for (int k = wid; k < mine; k += NT / 32) {                       // a warp a head: the blocks' headers
        const int a = rank + k * nblk;
        float m = -INFINITY, l = 0.f;
        if (lane < nblk) {
            const uint32_t at = cl::map_to(comb_addr + (uint32_t)(a * REC) * 4u, (uint32_t)lane);
            m = cl::ld_f32(at);
            l = cl::ld_f32(at + 4);
        }
        const float M = warp_max(m);
        const float f = m > -INFINITY ? __expf(m - M) : 0.f;
        const float L = warp_sum(f * l);
        if (lane < nblk) fac[k][lane] = f;
        if (lane == 0) Ls[k] = L;
    }
    merge_sync<NT>();
    for (int e = tid; e < mine * V4; e += NT) {
        const int k = e / V4, c4 = e - k * V4, a = rank + k * nblk;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int j0 = 0; j0 < nblk; j0 += 8) {                        // eight remote loads in flight
            float4 x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = cl::ld_f32x4(cl::map_to(comb_addr + (uint32_t)(a * REC + 4 + 4 * c4) * 4u, (uint32_t)min(j0 + j, nblk - 1)));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float f = j0 + j < nblk ? fac[k][j0 + j] : 0.f;
                acc.x = fmaf(f, x[j].x, acc.x); acc.y = fmaf(f, x[j].y, acc.y); acc.z = fmaf(f, x[j].z, acc.z); acc.w = fmaf(f, x[j].w, acc.w);
            }
        }
        const float v[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = 4 * c4 + i;
            if (c < D) avs[k][c] = v[i];
            else store_key_sum(ks, k, c - D, v[i]);
        }
    }
    __syncwarp();
    cl::arrive_release();                                             // this block reads no other block's memory from here on
    merge_sync<NT>();
    if (mine > 0) {
        for (int mt = wid; mt < D / 16; mt += NT / 32) map_rows(Wu, mt, mine, ks, pw, lane);
        merge_sync<NT>();
        for (int e = tid; e < mine * D; e += NT) {
            const int k = e / D, c = e - k * D;
            const float o = (avs[k][c] + pw[k][c]) / Ls[k];
            const size_t at = (size_t)(rank + k * nblk) * D + c;
            if (out_f32) reinterpret_cast<float*>(out_u)[at] = o;
            else reinterpret_cast<__nv_bfloat16*>(out_u)[at] = __float2bfloat16_rn(o);
        }
    }
    __syncwarp();
    cl::wait_acquire();                                               // nobody reads this block's memory any more
}

// grid (plan.B), or (U x cluster size) in clusters, Cfg::THREADS threads, Cfg::SMEM_BYTES (CLUSTER_SMEM_BYTES) of
// dynamic shared memory.
// partial: [U][s_max][CONSUMER_WARPS][g][REC]; slot of (unit u, block b) = b - block_of_tile(first tile of u).
// CLUSTER writes out itself and does not use partial.
template <int D, bool CLUSTER>
__global__ void __launch_bounds__(Cfg<D, false>::THREADS, 1)
decode_stream_bf16(const __nv_bfloat16* q, const __grid_constant__ Maps maps, Plan pl, int n_ret,
                        int n_apx, int g, int LH, float scale_log2e, float* __restrict__ partial,
                        int* __restrict__ fault, const __nv_bfloat16* W, void* __restrict__ out, int out_f32) {
    using C = Cfg<D, false>;
    constexpr int HALF_BYTES = C::HALF_BYTES, SLOT_BYTES = C::SLOT_BYTES, SLOTS = C::SLOTS;
    constexpr int CONSUMER_WARPS = C::CONSUMER_WARPS, REC = C::REC, CREC = C::CREC;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[SLOTS];
    __shared__ __align__(8) uint64_t empty_bar[SLOTS];
    // 128B-swizzled TMA boxes want 1024-byte aligned destinations
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int b = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wq = tid >> 5;
    long long gt_lo, gt_hi;
    block_range<CLUSTER>(pl, gt_lo, gt_hi);
    const int n_my = (int)(gt_hi - gt_lo);
    const int u0 = (int)(gt_lo / pl.n_tiles);
    const int u_last = (int)((gt_hi - 1) / pl.n_tiles);
    float* const recs = reinterpret_cast<float*>(smem + SLOTS * SLOT_BYTES);      // CLUSTER: the warps' records

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) { tma::mbar_init(&full_bar[s], 1); tma::mbar_init(&empty_bar[s], 1); }
        tma::mbar_fence_init();
    }
    // Launched as a programmatic dependent itself: everything above touches only this block's own state.  The merge
    // kernel is one of this kernel: its blocks may be scheduled as soon as SMs free up -- what was before this kernel
    // has finished then -- and read the records only after their own wait.
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    __syncthreads();
    const __nv_bfloat16* const Wu = W + (size_t)(u0 % LH) * D * D;
    if (CLUSTER) {                                                    // the map's way into L2, for the blocks that will apply it
        const char* Wb = reinterpret_cast<const char*>(Wu);
        for (int e = tid; e < 2 * D * D / 128; e += C::THREADS) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(Wb + 128 * e));
        __syncwarp();
    }
    auto merge_unit = [&]() {                                         // CLUSTER: each role's last act
        if (CLUSTER)
            cluster_merge<D, false>(recs, smem, Wu, g,
                                   reinterpret_cast<char*>(out) + (size_t)u0 * g * D * (out_f32 ? 4 : 2), out_f32 != 0);
    };

    if (wq == CONSUMER_WARPS) {
        // ------------------------------------------------------------------ producer
        if (lane == 0) produce<D, false>(maps, pl, gt_lo, n_my, smem, full_bar, empty_bar, fault);
        // the consumers wait on every tile's full barrier, so no copy outlives the block
        __syncwarp();
        merge_unit();
        return;
    }
    // ---------------------------------------------------------------------- consumers
    const int gid = lane >> 2, tig = lane & 3;
    const bool twice = C::PARTS == 3 && g <= 4;        // MMA rows 4-7 repeat the heads and take the third parts
    uint32_t qa[D / 16][2];
    float acc[D / 8][4];                  // [dim tile][c0,c1: rows of first (and third) parts | c2,c3: of second parts]
    float m = -INFINITY, l = 0.f, stash_scale = 1.f;
    bool stashed = false;

    auto record_of = [&](int unit) -> float* {
        if (CLUSTER) return recs + (wq * g + gid) * CREC;
        int slot = b - block_of_tile((long long)unit * pl.n_tiles, pl);
        if (slot < 0 || slot >= pl.s_max) { atomicCAS(fault, 0, 5); slot = 0; }     // cannot happen; never write out of bounds
        return partial + ((((size_t)unit * pl.s_max + slot) * CONSUMER_WARPS + wq) * g + gid) * REC;
    };
    auto add_third = [&]() {                 // the whole warp, before store_acc: the third parts' sums to their heads' rows
        if (twice) {
#pragma unroll
            for (int n = 0; n < D / 8; ++n) {
                acc[n][2] += __shfl_xor_sync(0xffffffffu, acc[n][0], 16);
                acc[n][3] += __shfl_xor_sync(0xffffffffu, acc[n][1], 16);
            }
        }
    };
    auto store_acc = [&](float* dst) {       // dims n*8 + 2 tig + {0,1} of head row gid
#pragma unroll
        for (int n = 0; n < D / 8; ++n)
            *reinterpret_cast<float2*>(dst + n * 8 + 2 * tig) = make_float2(acc[n][0] + acc[n][2], acc[n][1] + acc[n][3]);
    };
    auto zero_acc = [&]() {
#pragma unroll
        for (int n = 0; n < D / 8; ++n) { acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f; }
    };
    // Writes this warp's record of `unit` (an all-zero one with m = -inf if it met none of its tiles).
    auto flush = [&](int unit) {
        float lt = l;
        lt += __shfl_xor_sync(0xffffffffu, lt, 1);
        lt += __shfl_xor_sync(0xffffffffu, lt, 2);
        add_third();
        if (gid < g) {
            float* rec = record_of(unit);
            if (tig == 0) *reinterpret_cast<float4*>(rec) = make_float4(m * 0.69314718055994531f, lt, stashed ? stash_scale : 1.f, stashed ? 1.f : 0.f);
            if (stashed) {                            // value part was written at the pool switch
                store_acc(CLUSTER ? reinterpret_cast<float*>(smem + (SLOTS - CONSUMER_WARPS + wq) * SLOT_BYTES) + gid * D : rec + 4 + D);
            } else if (!CLUSTER) {
                store_acc(rec + 4);
#pragma unroll
                for (int n = 0; n < D / 8; ++n) *reinterpret_cast<float2*>(rec + 4 + D + n * 8 + 2 * tig) = make_float2(0.f, 0.f);
            } else if (m > -INFINITY) {               // (the cluster's merge looks no further than the header says)
                store_acc(rec + 4);
            }
        }
        zero_acc();
        m = -INFINITY; l = 0.f; stash_scale = 1.f; stashed = false;
    };
    // One softmax step over the 64 keys at kbase, in two parts.  The first leaves the step's weights p in sc (this thread:
    // head gid, keys 8 n + 2 tig, + 1) and brings m, l and (unless EXACT) the accumulators to the new running maximum.
    auto scores64 = [&](uint32_t kbase, int nrows, bool retained, int unit, float (&sc)[8][2]) -> float {
        float alpha;
        if constexpr (C::EXACT) alpha = score_step64(kbase, nrows, scale_log2e, qa, lane, m, l, sc);
        else alpha = score_step<D>(kbase, nrows, scale_log2e, qa, lane, m, l, sc);
        if (!retained && !stashed) {           // first key-only keys of this unit for this warp: park sum p v
            add_third();
            if (gid < g) store_acc(record_of(unit) + 4);
            zero_acc();
            stashed = true;
            stash_scale = 1.f;
        }
        stash_scale *= alpha;
        if (!C::EXACT && __any_sync(0xffffffffu, alpha != 1.f)) {
#pragma unroll
            for (int n = 0; n < D / 8; ++n) { acc[n][0] *= alpha; acc[n][1] *= alpha; acc[n][2] *= alpha; acc[n][3] *= alpha; }
        }
        return alpha;
    };
    // The second part adds p x (the 64 rows at vbase: values, or the keys themselves for a key-only tile).
    auto accumulate64 = [&](uint32_t vbase, float (&sc)[8][2], float alpha) {
        if constexpr (!C::EXACT) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                uint32_t a[4], third[2];
                weights_bf16<C::PARTS>(sc, kk, twice, gid, a, third);
                accumulate_step<D>(vbase, kk, a, false, third, acc, lane);
            }
        } else {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float sum[D / 8][4];                   // of 32 rows, which the accumulators take together
#pragma unroll
                for (int n = 0; n < D / 8; ++n) sum[n][0] = sum[n][1] = sum[n][2] = sum[n][3] = 0.f;
#pragma unroll
                for (int kk = 2 * half; kk < 2 * half + 2; ++kk) {
                    uint32_t a[4], third[2];
                    weights_bf16<C::PARTS>(sc, kk, twice, gid, a, third);
                    accumulate_step<D>(vbase, kk, a, !twice, third, sum, lane);
                }
                const uint64_t f = tc::pack2(alpha, alpha);
#pragma unroll
                for (int n = 0; n < D / 8; ++n)
#pragma unroll
                    for (int e = 0; e < 4; e += 2) {
                        const uint64_t o = tc::pack2(acc[n][e], acc[n][e + 1]), x = tc::pack2(sum[n][e], sum[n][e + 1]);
                        tc::unpack2(half == 0 ? tc::fma2(o, f, x) : tc::add2(o, x), acc[n][e], acc[n][e + 1]);
                    }
            }
        }
    };

    auto step64 = [&](uint32_t kbase, uint32_t vbase, int nrows, bool retained, int unit) {
        float sc[8][2];
        const float alpha = scores64(kbase, nrows, retained, unit, sc);
        accumulate64(vbase, sc, alpha);
    };

    zero_acc();
    // Walk the units the block touches; this warp owns the block's tiles i with i % CONSUMER_WARPS == wq.
    int i = wq;                                        // index into the block's tile sequence
    bool ok = true;                                    // false once a wait gave up: keep walking, touch nothing
    for (int u = u0; u <= u_last; ++u) {
        const long long unit_end = (long long)(u + 1) * pl.n_tiles - gt_lo;     // first sequence index past the unit
        bool loaded = false;
        for (; i < n_my && i < unit_end; i += CONSUMER_WARPS) {
            const int s = i % SLOTS, round = i / SLOTS;
            const int t = (int)(gt_lo + i - (long long)u * pl.n_tiles);
            if (ok) {
                if (!loaded) { load_queries<D>(q, u, g, lane, qa, twice); loaded = true; }
                ok = tma::mbar_wait_warp(&full_bar[s], round & 1, fault, 2);
            }
            if (!ok) continue;
            const uint32_t base = tma::smem_u32(smem + s * SLOT_BYTES);
            if (t < pl.n_rt) {
                step64(base, base + HALF_BYTES, min(KEYS, n_ret - t * KEYS), true, u);
            } else {
                const int r0 = (t - pl.n_rt) * 2 * KEYS;
                step64(base, base, min(KEYS, n_apx - r0), false, u);
                if (n_apx - r0 > KEYS)
                    step64(base + HALF_BYTES, base + HALF_BYTES, min(KEYS, n_apx - r0 - KEYS), false, u);
            }
            __syncwarp();
            if (lane == 0) tma::mbar_arrive(&empty_bar[s]);
        }
        flush(u);
    }
    __syncwarp();
    merge_unit();
}

// Merge: combines the records of a unit, applies the unit's map to the p-weighted key sum and normalises:
//   o = (sum_j f_j s_j acc_v_j + W sum_j f_j acc_k_j) / sum_j f_j l_j,   f_j = exp(m_j - max m).
// A thread owns four channels of a head's value or key sum; its warp reads that head's headers, a record a lane, and hands the factors
// round by shuffles, so that sums and headers share one memory latency and no barrier lies between them.  The map's fragments (MMAs,
// map_fragments) are requested ahead of the wait for the streaming kernel, which does not touch the map: they come in while that
// kernel drains.  What bounds it is that chain, one trip to L2 and a product a unit, as long as every unit has its block on the chip at
// once (RESIDENT a multiprocessor); beyond, the units in flight.  Which form takes how many units: launch_decode_bf16.
// RANGE: as many blocks as are resident at once, each with an equal range of the units, ordered by map, so that the
// sequences that share one find it in their block's registers; the next unit's records are requested before this one's product.
// Otherwise a block a unit.  Spilled, bytes a thread: 52 with five resident blocks of two heads, 12 with three of four, 48 with two of eight
// (12 at 64 channels).
template <int D, int HEADS, int RES> struct MergeCfg {
    static constexpr int THREADS = HEADS * D / 2, RESIDENT = RES;      // a head's sums take D / 2
    static constexpr bool RANGE = HEADS == 4 && RES == (D == 128 ? 2 : 4);
    static constexpr int AHEAD = RANGE ? 6 : D == 128 && HEADS <= 4 ? 3 : 4;      // records whose sums are requested together
    static constexpr int MAP_WARPS = THREADS / 32 < D / 16 ? THREADS / 32 : D / 16, ROWS = D / 16 / MAP_WARPS;      // warps with rows of the map, blocks of 16 rows each
    static constexpr int blocks(int U, int sms) { return RANGE && U > RESIDENT * sms ? RESIDENT * sms : U; }
};
template <typename TO, int D, int HEADS, int RES>
__global__ void __launch_bounds__(MergeCfg<D, HEADS, RES>::THREADS, RES)
decode_merge_bf16(const float* partial, const __nv_bfloat16* W, int LH, int U, int g,
                       Plan pl, int apply_w, int cw, TO* __restrict__ out) {
    using C = MergeCfg<D, HEADS, RES>;
    constexpr int REC = 4 + 2 * D, NT = C::THREADS;
    constexpr int MAX_REC = 12 * Cfg<D, false>::CONSUMER_WARPS, REC_PER_LANE = (MAX_REC + 31) / 32;      // of a unit: twelve blocks' at the most
    constexpr int BUFS = C::RANGE ? 2 : 1;                  // of two units in turn
    __shared__ KeySums<D> ks[BUFS];
    __shared__ __align__(16) float sums[BUFS][HEADS][2 * D];      // value sums; without the map the key sums too
    __shared__ float Ls[BUFS][HEADS];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int a = tid / (D / 2), c4 = tid % (D / 2);        // a head's value sums, then its key sums, four channels a thread
    const bool mine = a < g, value = c4 < D / 4, mapping = apply_w && wid < C::MAP_WARPS;      // mine, mapping: whole warps
    const int batch = U / LH;
    const int i_lo = C::RANGE ? (int)((long long)blockIdx.x * U / gridDim.x) : (int)blockIdx.x;
    const int i_hi = C::RANGE ? (int)((long long)(blockIdx.x + 1) * U / gridDim.x) : i_lo + 1;
    uint4 A[C::ROWS][D / 16];
    auto map_of = [&](int i) {
#pragma unroll
        for (int r = 0; r < C::ROWS; ++r) map_fragments<D>(W + (size_t)(i / batch) * D * D, wid + r * C::MAP_WARPS, A[r], lane);
    };
    if (mapping) map_of(i_lo);
    for (int i = tid; i < BUFS * (8 - g) * D; i += NT) store_key_sum(ks[i % BUFS], g + i / BUFS / D, i / BUFS % D, 0.f);      // columns of B beyond the unit's heads
    // the streaming kernel's records from here on
    asm volatile("griddepcontrol.wait;\n" ::: "memory");

    constexpr int NPRE = C::AHEAD;                          // a unit lies in one or two blocks of the streaming kernel, three or four records each, unless it is very long
    const size_t step = (size_t)g * REC;                    // from record to record
    int n_rec;
    const float* base;
    float4 v[NPRE], hd[REC_PER_LANE];                       // sums; headers of records lane, lane + 32
    auto sums_from = [&](int j0) {
#pragma unroll
        for (int k = 0; k < NPRE; ++k) v[k] = *reinterpret_cast<const float4*>(base + min(j0 + k, n_rec - 1) * step + 4 + 4 * c4);
    };
    auto request = [&](int i) {
        const int u = i % batch * LH + i / batch;
        const int first = block_of_tile((long long)u * pl.n_tiles, pl);
        n_rec = (block_of_tile((long long)(u + 1) * pl.n_tiles - 1, pl) - first + 1) * cw;       // <= MAX_REC; cw records per block
        base = partial + ((size_t)u * pl.s_max * cw * g + a) * REC;
        sums_from(0);
#pragma unroll
        for (int k = 0; k < REC_PER_LANE; ++k)
            hd[k] = lane + 32 * k < n_rec ? *reinterpret_cast<const float4*>(base + (lane + 32 * k) * step) : make_float4(-INFINITY, 0.f, 0.f, 0.f);
    };
    if (mine) request(i_lo);
    for (int i = i_lo; i < i_hi; ++i) {
        const int buf = C::RANGE ? i & 1 : 0, u = i % batch * LH + i / batch;
        if (mine) {
            float M = hd[0].x;
#pragma unroll
            for (int k = 1; k < REC_PER_LANE; ++k) M = fmaxf(M, hd[k].x);
            M = warp_max(M);
            float Lsum = 0.f, fk[REC_PER_LANE], fv[REC_PER_LANE];                                // factors of the key and of the value sums
#pragma unroll
            for (int k = 0; k < REC_PER_LANE; ++k) {
                fk[k] = hd[k].x > -INFINITY ? __expf(hd[k].x - M) : 0.f;
                fv[k] = fk[k] * hd[k].z;
                Lsum += fk[k] * hd[k].y;
            }
            Lsum = warp_sum(Lsum);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int j0 = 0; j0 < n_rec; j0 += NPRE) {
                if (j0 > 0) sums_from(j0);
#pragma unroll
                for (int k = 0; k < NPRE; ++k) {
                    const int j = j0 + k;
                    if (j >= n_rec) break;
                    float f0 = fk[0], f1 = fv[0];
                    if (REC_PER_LANE > 1 && j >= 32) { f0 = fk[REC_PER_LANE - 1]; f1 = fv[REC_PER_LANE - 1]; }
                    f0 = __shfl_sync(0xffffffffu, f0, j & 31);
                    f1 = __shfl_sync(0xffffffffu, f1, j & 31);
                    const float f = value ? f1 : f0;
                    acc.x = fmaf(f, v[k].x, acc.x); acc.y = fmaf(f, v[k].y, acc.y); acc.z = fmaf(f, v[k].z, acc.z); acc.w = fmaf(f, v[k].w, acc.w);
                }
            }
            if (C::RANGE && i + 1 < i_hi) request(i + 1);
            if (c4 == 0) Ls[buf][a] = Lsum;
            if (value || !apply_w) {                        // per-tile form: the second part of a record is already sum p (W k)
                *reinterpret_cast<float4*>(&sums[buf][a][4 * c4]) = acc;
            } else {
                const int c = 4 * c4 - D;
                store_key_sum(ks[buf], a, c, acc.x); store_key_sum(ks[buf], a, c + 1, acc.y);
                store_key_sum(ks[buf], a, c + 2, acc.z); store_key_sum(ks[buf], a, c + 3, acc.w);
            }
        }
        // one barrier a unit: whoever writes this half again, two units on, has seen every warp past this unit
        __syncthreads();
        TO* const o = out + (size_t)u * g * D;
        if (mapping) {
            const int head = 2 * (lane & 3);
            float d[C::ROWS][4];
#pragma unroll
            for (int r = 0; r < C::ROWS; ++r) map_product<D>(A[r], ks[buf], d[r], lane);
            if (C::RANGE && i + 1 < i_hi && (i + 1) % batch == 0) map_of(i + 1);
#pragma unroll
            for (int r = 0; r < C::ROWS; ++r)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int h = head + (e & 1), c = 16 * (wid + r * C::MAP_WARPS) + (lane >> 2) + 8 * (e >> 1);
                    if (h < g) store_out(o + h * D + c, (sums[buf][h][c] + d[r][e]) / Ls[buf][h]);
                }
        } else if (!apply_w) {
            for (int e = tid; e < g * D; e += NT) store_out(o + e, (sums[buf][e / D][e % D] + sums[buf][e / D][D + e % D]) / Ls[buf][e / D]);
        }
    }
}

// The same for up to three heads in many units of 128 channels, where units in flight are what counts: a thread a channel, D g of them
// and 40 registers each (8 to 12 bytes spilled), the factors through shared memory and the map read behind them.
template <typename TO, int D>
__global__ void __launch_bounds__(3 * D, 4)
decode_merge_channels(const float* partial, const __nv_bfloat16* W, int LH, int U, int g,
                      Plan pl, int apply_w, int cw, TO* __restrict__ out) {
    constexpr int REC = 4 + 2 * D;
    constexpr int MAX_REC = 12 * Cfg<D, false>::CONSUMER_WARPS, REC_PER_LANE = (MAX_REC + 31) / 32;
    __shared__ KeySums<D> ks;
    __shared__ float pw[8][D];                 // W times the key sum
    __shared__ float fv[3][MAX_REC], fk[3][MAX_REC];     // per head, per record: factor for the value part / the key part
    __shared__ float Ls[3];
    const int u = blockIdx.x, tid = threadIdx.x, a = tid / D, c = tid % D, lane = tid & 31;
    const int wid = tid >> 5, nwarps = blockDim.x >> 5;
    const __nv_bfloat16* Wu = W + (size_t)(u % LH) * D * D;
    for (int i = tid; i < (8 - g) * D; i += blockDim.x) store_key_sum(ks, g + i / D, i % D, 0.f);      // columns of B beyond the unit's heads
    // the streaming kernel's records from here on
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    const int first = block_of_tile((long long)u * pl.n_tiles, pl);
    const int n_rec = (block_of_tile((long long)(u + 1) * pl.n_tiles - 1, pl) - first + 1) * cw;
    const float* base = partial + (size_t)u * pl.s_max * cw * g * REC;
    constexpr int NPRE = 6;                              // records whose sums are requested together, the first ones before the headers
    float rv[NPRE], rk[NPRE];
    auto sums_from = [&](int j0) {
#pragma unroll
        for (int k = 0; k < NPRE; ++k) {
            const int j = min(j0 + k, n_rec - 1);
            const float* r = base + ((size_t)j * g + a) * REC + 4;
            rv[k] = r[c];
            rk[k] = r[D + c];
        }
    };
    sums_from(0);
    if (c < 32) {
        // first warp of head a: headers of records lane, lane + 32, ...
        float mj[REC_PER_LANE], lj[REC_PER_LANE], sj[REC_PER_LANE], M = -INFINITY;
#pragma unroll
        for (int k = 0; k < REC_PER_LANE; ++k) {
            const int j = lane + 32 * k;
            mj[k] = -INFINITY; lj[k] = 0.f; sj[k] = 0.f;
            if (j < n_rec) {
                const float4 h = *reinterpret_cast<const float4*>(base + ((size_t)j * g + a) * REC);
                mj[k] = h.x; lj[k] = h.y; sj[k] = h.z;
            }
            M = fmaxf(M, mj[k]);
        }
        M = warp_max(M);
        float Lsum = 0.f;
#pragma unroll
        for (int k = 0; k < REC_PER_LANE; ++k) {
            const int j = lane + 32 * k;
            const float f = mj[k] > -INFINITY ? __expf(mj[k] - M) : 0.f;
            if (j < MAX_REC) { fk[a][j] = f; fv[a][j] = f * sj[k]; }
            Lsum += f * lj[k];
        }
        Lsum = warp_sum(Lsum);
        if (lane == 0) Ls[a] = Lsum;
    }
    __syncthreads();
    float av = 0.f, ak = 0.f;
    for (int j0 = 0; j0 < n_rec; j0 += NPRE) {
        if (j0 > 0) sums_from(j0);
#pragma unroll
        for (int k = 0; k < NPRE; ++k) {
            if (j0 + k < n_rec) {
                av = fmaf(fv[a][j0 + k], rv[k], av);
                ak = fmaf(fk[a][j0 + k], rk[k], ak);
            }
        }
    }
    if (!apply_w) {           // per-tile form: the second part of a record is already sum p (W k)
        store_out(out + ((size_t)u * g + a) * D + c, (av + ak) / Ls[a]);
        return;
    }
    store_key_sum(ks, a, c, ak);
    __syncthreads();
    for (int mt = wid; mt < D / 16; mt += nwarps) map_rows(Wu, mt, g, ks, pw, lane);
    __syncthreads();
    store_out(out + ((size_t)u * g + a) * D + c, (av + pw[a][c]) / Ls[a]);
}

}  // namespace dbf
}  // namespace vec
#endif
