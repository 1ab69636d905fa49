// Decode attention with one map per layer on warp-level MMAs (bf16, head_dim 128, 8 KV heads, at most
// 32 query heads per layer): the split and merge kernels of the factored form
//   o_a = sum_R p_i v_{i,h} + sum_h' W[h][h'] (sum_A p_i k_{i,h'})          (paper Sections 3.2 and 5.1)
// in which a block owns a slice of the tokens of one (sequence, layer) and ALL its heads, so that every
// approximated key is read once for the key sums of all query heads of the layer.
//
// Split kernel: 8 warps, warp w = KV head w.  The slice is walked in tiles that fill one 64 KB stage (three
// stages, TMA): 16 retained tokens (keys and values of the 8 heads) or 32 approximated tokens (keys of the 8
// heads).  Per tile
//   phase 1  warp h: logits of its g query heads against head h's keys (the keys fill the 16 rows of the MMAs, the heads
//            their eight columns), online softmax; for an approximated tile the probabilities go to shared memory as
//            bf16 hi + lo, P[32 query heads][32 tokens], with the rescaling factor of each query head;
//   phase 2  warp h': its accumulator acc_k[32 query heads][128] (key sums over head h') is rescaled and
//            takes P K_h' (both halves of P); for a retained tile warp h adds V_h^T P for its own heads.
// Phase 1 is a chain of dependent MMAs, shuffles and exponentials, phase 2 a run of independent MMAs: with two warps to a
// scheduler neither hides the other's latency unless they are the same warp's instructions.  So phase 1 of tile t + 1 is
// laid between the MMAs of phase 2 of tile t, one barrier a tile; the third stage is the tile in flight meanwhile.
// The tiles of all (sequence, layer) pairs form one row, dealt in equal contiguous pieces to persistent blocks (Plan).
// What bounds it: the warps' own instructions -- tensor pipe 41 % busy, HBM 0.74 of a copy's rate in the streaming
// kernel -- with eight warps, whose accumulators leave no room for more.  Measured, 32 pairs of 7200 rows, 630 MB, in a
// graph: 130 us; 143 with whole splits of a pair in two rounds of blocks, 173 with tiles copied in 16-byte pieces by all
// threads, 210 with the two phases one after the other.
// Records have the layout of the CUDA-core split kernel: per (unit, split, head) m, l, acc_v[128],
// acc_k[8][128].
#ifndef VECTOR_DECODE_LAYER_MMA_CUH_
#define VECTOR_DECODE_LAYER_MMA_CUH_

#include <type_traits>

#include "common.cuh"
#include "decode_bf16.cuh"

namespace vec {
namespace dlm {

constexpr int HKV = 8, THREADS = 32 * HKV, MQ = 32;        // query heads per layer the accumulators hold
constexpr int RT = 16, AT = 32;                            // tokens per retained / approximated tile
// A stage: boxes of 64 channels x the tile's tokens x the 8 heads (128-byte rows, 128-byte swizzle); retained: keys, channels
// 0-63 and 64-127, then values; approximated: keys.
constexpr int STAGE_BYTES = 65536, HEAD_RET = RT * 128, HEAD_APX = AT * 128, BOX_RET = HKV * HEAD_RET, BOX_APX = HKV * HEAD_APX;
constexpr int PS_ROW = 80;                                 // bytes per row of P: 32 tokens + padding (conflict-free ldmatrix)
constexpr int STAGES = 3;
constexpr int RET_COST = 1, APX_COST = 2;                  // relative time of a tile (measured in a graph: 1:1 176, 2:3 154, 1:2 144, 4:9 150,
                                                           // 2:5 157 us a step of 32 layers and 7200 rows; 48, 44, 43, 43, 43 for one layer)
constexpr int P_BYTES = 2 * MQ * PS_ROW + MQ * 4;          // P hi, P lo, factors: one set for each of two tiles
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 2 * P_BYTES + 128 + 1024;       // + alignment slack
constexpr int REC = 2 + 128 + HKV * 128;

// The weights' reference is the running maximum itself, so that the largest weight, which keeps sixteen bits like the others, is one
// and exact.  Letting it lag by up to eight powers of two spares most rescalings of the 160 accumulators (150 against 153 us for 32
// pairs of 7200 rows), at outputs that are off by a twentieth more.
// (tc::ex2 gives zero for results below 2^-126: next to a weight of one they do not change an fp32 sum.)

// How the work is dealt: the (sequence, layer) pairs' tiles in one row, weighted by their cost, cut into B equal pieces, one
// persistent block each.  A pair's records: one of every block that reaches into it.  The same arithmetic runs on host and device.
struct Plan {
    int n_rt, n_at, UL;        // retained / key-only tiles of a pair, pairs
    int weight, B, s_max;      // cost of a pair, blocks, record slots of a pair
};
constexpr int MAX_RECORDS = 32;
__host__ __device__ inline Plan make_plan(int UL, long long n_ret, long long n_apx, int max_blocks) {
    Plan p;
    p.UL = UL;
    p.n_rt = (int)((n_ret + RT - 1) / RT);
    p.n_at = (int)((n_apx + AT - 1) / AT);
    p.weight = RET_COST * p.n_rt + APX_COST * p.n_at;
    const long long total = (long long)UL * p.weight;
    const auto limit = [](long long x, long long most) { return x < most ? x : most; };
    long long b = limit(max_blocks, total / 4);                // two key-only tiles a block at the least
    b = b < 1 ? 1 : b;
    // The same number of blocks for every pair leaves some multiprocessors idle, but no block with the ends of two pairs; a
    // record costs a block about eight retained tiles (its first loads, 147 KB written, and read again by the merge).  Measured in
    // a graph, all multiprocessors against whole blocks a pair, us: 32 pairs of 600 rows 48 / 43, of 7200 rows 140 / 146; 16
    // pairs of 4900 rows 80 / 76 (the merge three blocks to a multiprocessor in all of them).
    if (b >= UL) {
        const long long whole = b / UL * UL;
        const long long reach = b == whole ? 1 : 2;            // pairs a block reaches into
        if (total / whole + 8 <= total / b + 8 * reach) b = whole;
    }
    if (b > (long long)UL * (MAX_RECORDS - 2)) b = (long long)UL * limit(b / UL, MAX_RECORDS);
    p.B = (int)b;
    p.s_max = b % UL == 0 ? (int)(b / UL) : (int)(b / UL) + 2;      // a pair's share of the blocks begins and ends inside one
    return p;
}
__host__ __device__ inline long long cost_begin(int b, const Plan& p) { return (long long)b * p.weight * p.UL / p.B; }
__host__ __device__ inline int block_of_cost(long long x, const Plan& p) { return (int)(((x + 1) * p.B - 1) / ((long long)p.weight * p.UL)); }

// grid (plan.B), THREADS threads, SMEM_BYTES dynamic shared memory.  partial: [U][s_max][g][REC]; slot of (pair, block b) =
// b - block_of_cost(first cost of the pair).
__global__ void __launch_bounds__(THREADS, 1)
decode_layer_mma(const __nv_bfloat16* q, const __grid_constant__ dbf::Maps maps, Plan pl, int n_ret, int n_apx, int g,
                 float scale_log2e, float* __restrict__ partial, int* __restrict__ fault) {
    __shared__ __align__(8) uint64_t full_bar[STAGES];
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) tma::mbar_init(&full_bar[s], 1);
        tma::mbar_fence_init();
    }
    asm volatile("griddepcontrol.wait;\n" ::: "memory");        // launched as a programmatic dependent: nothing of its inputs is touched before
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    extern __shared__ unsigned char lsm[];
    unsigned char* const stage0 = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(lsm) + 1023) & ~uintptr_t(1023));
    unsigned char* const ps = stage0 + STAGES * STAGE_BYTES;
    const uint32_t dump = tma::smem_u32(ps + 2 * P_BYTES);      // where the rows of absent heads go
    const int tid = threadIdx.x, lane = tid & 31, h = tid >> 5;
    const int gid = lane >> 2, tig = lane & 3, mat = lane >> 3, r8 = lane & 7;
    const int b = blockIdx.x, n_rt = pl.n_rt, n_tiles = pl.n_rt + pl.n_at;
    // A key-only tile takes 144 MMAs a warp, a retained one 24 (both bring in 64 KB): the pieces are equal in time, not in tiles.
    auto tile_at = [&](int x) -> int {                // first tile of a pair that begins at or after x
        return x <= RET_COST * n_rt ? (x + RET_COST - 1) / RET_COST : n_rt + (x - RET_COST * n_rt + APX_COST - 1) / APX_COST;
    };
    const long long c_lo = cost_begin(b, pl), c_hi = cost_begin(b + 1, pl);           // never empty
    const int u_first = (int)(c_lo / pl.weight), u_last = (int)((c_hi - 1) / pl.weight);
    const int first_lo = tile_at((int)(c_lo - (long long)u_first * pl.weight)), last_hi = tile_at((int)(c_hi - (long long)u_last * pl.weight));

    for (int i = tid; i < 2 * P_BYTES / 4; i += THREADS) reinterpret_cast<uint32_t*>(ps)[i] = 0u;
    uint32_t qa[8][2];                             // the g query rows of this head as B fragments (columns g .. 7 zero)
    float acc_k[2][16][4], acc_v[8][4];            // acc_v[n]: dims 16 n + gid (, + 8) of heads 2 tig, + 1
    auto zero_acc = [&]() {
#pragma unroll
        for (int n = 0; n < 16; ++n) {
            if (n < 8) acc_v[n][0] = acc_v[n][1] = acc_v[n][2] = acc_v[n][3] = 0.f;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) acc_k[mt][n][0] = acc_k[mt][n][1] = acc_k[mt][n][2] = acc_k[mt][n][3] = 0.f;
        }
    };
    zero_acc();
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};       // of heads 2 tig, + 1; l: this lane's tokens only

    bool ok = true;                            // false once a wait gave up: walk on and touch nothing
    // One thread requests tile t of pair u, or as many tiles into the following pairs as t lies past its end, into stage sg;
    // rows past the pool's end are filled with zeros.
    const uint64_t pol = tma::policy_evict_first();                 // the cache is read once per step
    auto request = [&](int u, int t, int sg) {
        if (tid == 0 && ok) {
            while (u <= u_last && t >= (u == u_last ? last_hi : n_tiles)) {
                t -= u == u_last ? last_hi : n_tiles;
                ++u;
            }
            if (u <= u_last) {
                unsigned char* st = stage0 + sg * STAGE_BYTES;
                tma::mbar_expect_tx(&full_bar[sg], STAGE_BYTES);
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    if (t < n_rt) {
                        tma::load_3d_hint(st + x * BOX_RET, &maps.ret_k, 64 * x, t * RT, u * HKV, &full_bar[sg], pol);
                        tma::load_3d_hint(st + 32768 + x * BOX_RET, &maps.ret_v, 64 * x, t * RT, u * HKV, &full_bar[sg], pol);
                    } else {
                        tma::load_3d_hint(st + x * BOX_APX, &maps.apx_k, 64 * x, (t - n_rt) * AT, u * HKV, &full_bar[sg], pol);
                    }
                }
            }
        }
        __syncwarp();
    };
    // Tile t of the pair at hand is tile t + off of the block's piece.
    int off = 0;
    auto landed = [&](int t) {
        if (ok) ok = tma::mbar_wait_warp(&full_bar[(t + off) % STAGES], ((t + off) / STAGES) & 1, fault, 2);
    };

    // State of a tile between its two phases: the factors of heads 2 tig, + 1 and, retained, P as B fragments.
    float alpha[2] = {1.f, 1.f}, sc[2][4];
    uint32_t bp[2][2];
    // ldmatrix of 16 rows, (rows 0-7 | 8-15) x (16-byte chunk 2 c | 2 c + 1): a lane's address for c is this one with bits 5 and 6
    // XORed by c % 4 (the swizzle), in box c / 4
    const uint32_t frag = (uint32_t)((r8 + (mat & 1) * 8) * 128 + (((mat >> 1) ^ r8) << 4));
    auto chunk = [](uint32_t base, int c, uint32_t box) { return (base ^ (uint32_t)((c & 3) << 5)) + (c >> 2) * box; };
    auto stage_of = [&](int t) { return tma::smem_u32(stage0 + ((t + off) % STAGES) * STAGE_BYTES); };
    // logits, k step `item / J` of the 16 tokens `item % J`, J = 1 (retained) or 2
    auto logit_item = [&](uint32_t kbase, int item, int J) {
        const int ks = item / J, j = item % J;
        uint32_t a0, a1, a2, a3;
        dbf::ldsm_x4(chunk(kbase, ks, J == 1 ? BOX_RET : BOX_APX) + j * 16 * 128, a0, a1, a2, a3);
        dbf::mma_16(sc[j], a0, a1, a2, a3, qa[ks][0], qa[ks][1]);
    };
    // softmax of a tile's logits; leaves P and the factors where phase 2 takes them
    auto softmax = [&](auto ret, int t, float (&al)[2], uint32_t (&b)[2][2]) {
        constexpr bool RET = decltype(ret)::value;
        constexpr int J = RET ? 1 : 2;
        const int ntok = RET ? min(RT, n_ret - t * RT) : min(AT, n_apx - (t - n_rt) * AT);
        float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                sc[j][e] *= scale_log2e;
                if (ntok < 16 * J && 16 * j + 8 * (e >> 1) + gid >= ntok) sc[j][e] = -INFINITY;
                mx[e & 1] = fmaxf(mx[e & 1], sc[j][e]);
            }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1)
#pragma unroll
            for (int e = 0; e < 2; ++e) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], o));
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float m_new = fmaxf(m[e], mx[e]);                            // finite: a tile holds at least one token
            al[e] = tc::ex2(m[e] - m_new);
            m[e] = m_new;
            l[e] *= al[e];
        }
        unsigned char* const pb = ps + ((t + off) & 1) * P_BYTES;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            uint32_t hi[2], lo[2];                         // tokens gid and gid + 8 of the 16
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float p0 = tc::ex2(sc[j][2 * e] - m[0]), p1 = tc::ex2(sc[j][2 * e + 1] - m[1]);
                l[0] += p0;
                l[1] += p1;
                hi[e] = dbf::pack_bf16(p0, p1);
                lo[e] = dbf::pack_bf16(p0 - __uint_as_float(hi[e] << 16), p1 - __uint_as_float(hi[e] & 0xffff0000u));
            }
            if (RET) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(b[0][e]) : "r"(hi[e]));
                    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(b[1][e]) : "r"(lo[e]));
                }
            } else {
                // matrices (hi | lo) x (tokens 0-7 | 8-15), transposed on the way: a row a head
                const uint32_t at = r8 < g ? tma::smem_u32(pb) + (mat >> 1) * MQ * PS_ROW + (h * g + r8) * PS_ROW + j * 32 + (mat & 1) * 16 : dump + r8 * 16;
                asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};\n" ::"r"(at), "r"(hi[0]), "r"(hi[1]), "r"(lo[0]), "r"(lo[1]) : "memory");
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (lane < 4 && 2 * lane + e < g) reinterpret_cast<float*>(pb + 2 * MQ * PS_ROW)[h * g + 2 * lane + e] = al[e];
    };
    // Phase 2 of tile t with phase 1 of tile t + 1 between its MMAs.  next: 0 none, 1 retained, 2 approximated.
    auto interval = [&](auto ret, auto next, int t, int changed) {
        constexpr bool RET = decltype(ret)::value;
        constexpr int NEXT = decltype(next)::value, J = NEXT == 1 ? 1 : 2, ITEMS = NEXT == 0 ? 0 : 8 * J;
        const uint32_t st = stage_of(t) + frag, kn = stage_of(t + 1) + frag + h * (NEXT == 1 ? HEAD_RET : HEAD_APX);
        if (changed) {
            const float* f = reinterpret_cast<const float*>(ps + ((t + off) & 1) * P_BYTES + 2 * MQ * PS_ROW);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const float f0 = f[16 * mt + gid], f1 = f[16 * mt + 8 + gid];
#pragma unroll
                for (int n = 0; n < 16; ++n) { acc_k[mt][n][0] *= f0; acc_k[mt][n][1] *= f0; acc_k[mt][n][2] *= f1; acc_k[mt][n][3] *= f1; }
            }
#pragma unroll
            for (int n = 0; n < 8; ++n) { acc_v[n][0] *= alpha[0]; acc_v[n][1] *= alpha[1]; acc_v[n][2] *= alpha[0]; acc_v[n][3] *= alpha[1]; }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.f;
        float al[2] = {1.f, 1.f};
        uint32_t b[2][2] = {};
        if (RET) {
            // sum p v for this head's own query rows; the hi and the lo product of an accumulator are kept apart: back to
            // back the second would wait for the first
            const uint32_t vbase = st + 32768 + h * HEAD_RET;
#pragma unroll
            for (int q4 = 0; q4 < 2; ++q4) {
                uint32_t a[4][4];
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    dbf::ldsm_x4_t(chunk(vbase, 4 * q4 + n, BOX_RET), a[n][0], a[n][2], a[n][1], a[n][3]);
#pragma unroll
                for (int part = 0; part < 2; ++part)
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        dbf::mma_16(acc_v[4 * q4 + n], a[n][0], a[n][1], a[n][2], a[n][3], bp[part][0], bp[part][1]);
                        const int it = 8 * q4 + 4 * part + n;                  // of 16
                        if (it < ITEMS) logit_item(kn, it, J);
                    }
            }
            if constexpr (NEXT != 0) softmax(std::bool_constant<NEXT == 1>{}, t + 1, al, b);
        } else {
            // key sums over head h (= this warp) for all query heads of the layer: P[32 x 32] K_h[32 x 128]
            const uint32_t kbase = st + h * HEAD_APX;
            const uint32_t ph = tma::smem_u32(ps + ((t + off) & 1) * P_BYTES) + (uint32_t)((r8 + (mat & 1) * 8) * PS_ROW + (mat >> 1) * 16);
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
                for (int part = 0; part < 2; ++part) {             // hi sweep, then lo sweep (see above)
                    uint32_t a[2][4];
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt)
                        dbf::ldsm_x4(ph + part * MQ * PS_ROW + mt * 16 * PS_ROW + kk * 32, a[mt][0], a[mt][1], a[mt][2], a[mt][3]);
#pragma unroll
                    for (int np = 0; np < 8; ++np) {
                        uint32_t b0, b1, b2, b3;
                        dbf::ldsm_x4_t(chunk(kbase, np, BOX_APX) + kk * 16 * 128, b0, b1, b2, b3);
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt) {
                            dbf::mma_16(acc_k[mt][2 * np], a[mt][0], a[mt][1], a[mt][2], a[mt][3], b0, b1);
                            dbf::mma_16(acc_k[mt][2 * np + 1], a[mt][0], a[mt][1], a[mt][2], a[mt][3], b2, b3);
                        }
                        const int it = 16 * kk + 8 * part + np;                // of 32
                        if (it < ITEMS) logit_item(kn, it, J);
                    }
                }
                if constexpr (NEXT != 0) if (kk == 0) softmax(std::bool_constant<NEXT == 1>{}, t + 1, al, b);
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) { alpha[e] = al[e]; bp[0][e] = b[0][e]; bp[1][e] = b[1][e]; }
    };
    using Ret = std::true_type;
    using Apx = std::false_type;
    using None = std::integral_constant<int, 0>;
    using NextRet = std::integral_constant<int, 1>;
    using NextApx = std::integral_constant<int, 2>;

    __syncthreads();                           // the barriers, P and the factors are initialised
    request(u_first, first_lo, 0);
    request(u_first, first_lo + 1, 1);
    for (int ul = u_first; ul <= u_last; ++ul) {
        const int t_lo = ul == u_first ? first_lo : 0, t_hi = ul == u_last ? last_hi : n_tiles;
        const size_t u = (size_t)ul * HKV + h;
        off -= t_lo;
        if (t_lo < t_hi) {
            const uint32_t* qrow = reinterpret_cast<const uint32_t*>(q + (u * g + min(gid, g - 1)) * 128);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                qa[ks][0] = gid < g ? qrow[ks * 8 + tig] : 0u;
                qa[ks][1] = gid < g ? qrow[ks * 8 + 4 + tig] : 0u;
            }
            landed(t_lo);
            if (ok) {
#pragma unroll
                for (int j = 0; j < 2; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.f;
                if (t_lo < n_rt) {
#pragma unroll
                    for (int it = 0; it < 8; ++it) logit_item(stage_of(t_lo) + frag + h * HEAD_RET, it, 1);
                    softmax(Ret{}, t_lo, alpha, bp);
                } else {
#pragma unroll
                    for (int it = 0; it < 16; ++it) logit_item(stage_of(t_lo) + frag + h * HEAD_APX, it, 2);
                    softmax(Apx{}, t_lo, alpha, bp);
                }
            }
        }
        for (int t = t_lo; t < t_hi; ++t) {
            // P and the factors of tile t are written; everyone is done with the tile before it, whose stage is the next to fill
            const int changed = __syncthreads_or((2 * tig < g && alpha[0] != 1.f) || (2 * tig + 1 < g && alpha[1] != 1.f));
            request(ul, t + 2, (t + 2 + off) % STAGES);
            if (t + 1 < t_hi) landed(t + 1);
            if (!ok) continue;
            if (t + 1 == t_hi) { if (t < n_rt) interval(Ret{}, None{}, t, changed); else interval(Apx{}, None{}, t, changed); }
            else if (t + 1 < n_rt) interval(Ret{}, NextRet{}, t, changed);
            else if (t < n_rt) interval(Ret{}, NextApx{}, t, changed);
            else interval(Apx{}, NextApx{}, t, changed);
        }
        off += t_hi;
        int slot = b - block_of_cost((long long)ul * pl.weight, pl);
        if (slot < 0 || slot >= pl.s_max) { atomicCAS(fault, 0, 5); slot = 0; }     // cannot happen; never write out of bounds
        // ---- records.  Warp h: m, l and sum p v of its own query rows; every warp: its head's key sums for all rows
#pragma unroll
        for (int e = 0; e < 2; ++e) {
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) l[e] += __shfl_xor_sync(0xffffffffu, l[e], o);
            if (2 * tig + e < g) {
                float* rec = partial + ((u * pl.s_max + slot) * g + 2 * tig + e) * REC;
                if (gid == 0) { rec[0] = m[e] * 0.69314718055994531f; rec[1] = l[e]; }
#pragma unroll
                for (int n = 0; n < 8; ++n) { rec[2 + 16 * n + gid] = acc_v[n][e]; rec[2 + 16 * n + 8 + gid] = acc_v[n][2 + e]; }
            }
        }
        const int n_q = HKV * g;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int a = 16 * mt + 8 * half + gid;                 // query head of the layer
                if (a < n_q) {
                    float* rec = partial + ((((size_t)ul * HKV + a / g) * pl.s_max + slot) * g + a % g) * REC + 2 + 128 + h * 128;
#pragma unroll
                    for (int n = 0; n < 16; ++n)
                        *reinterpret_cast<float2*>(rec + n * 8 + 2 * tig) = make_float2(acc_k[mt][n][2 * half], acc_k[mt][n][2 * half + 1]);
                }
            }
        }
        zero_acc();
        m[0] = m[1] = -INFINITY;
        l[0] = l[1] = 0.f;
    }
}

// Two neighbouring elements of a column's records, which begin at src and lie g * REC apart, under the factors f of its splits.
__device__ __forceinline__ void merge_two(const float* src, int n_splits, int g, const float (&fs)[32], float& v0, float& v1) {
    v0 = v1 = 0.f;
    for (int s0 = 0; s0 < n_splits; s0 += 8) {
        float2 x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = *reinterpret_cast<const float2*>(src + (size_t)min(s0 + k, n_splits - 1) * g * REC);   // always a valid record
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float f = s0 + k < n_splits ? fs[s0 + k] : 0.f;
            v0 = fmaf(f, x[k].x, v0);
            v1 = fmaf(f, x[k].y, v1);
        }
    }
}
// d += rows Wr and Wr + 8 of the map (this thread's columns of them) times the key sums of four input heads, the first or the last four.
__device__ __forceinline__ void map_rows_times_keys(const __nv_bfloat16* Wr, const __nv_bfloat16 (&akh)[8][HKV * 128],
                                                    const __nv_bfloat16 (&akl)[8][HKV * 128], int half, int row, int quarter, float (&d)[4]) {
    constexpr int KD = HKV * 128;
    const uint4* Wr0 = reinterpret_cast<const uint4*>(Wr);
    const uint4* Wr1 = Wr0 + 8 * (KD / 8);                 // row + 8
#pragma unroll 2
    for (int kc = half * (HKV / 2); kc < (half + 1) * (HKV / 2); ++kc) {                     // 128 columns a time: 16 pieces of 16 bytes per row
        uint4 A[8];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            A[2 * jj + 0] = Wr0[kc * 16 + quarter + 4 * jj];
            A[2 * jj + 1] = Wr1[kc * 16 + quarter + 4 * jj];
        }
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const uint4 a0 = A[2 * jj], a1 = A[2 * jj + 1];
            const int col = kc * 128 + 8 * (quarter + 4 * jj);
            const uint4 bh = *reinterpret_cast<const uint4*>(&akh[row][col]);      // B column = head `row`
            const uint4 bl = *reinterpret_cast<const uint4*>(&akl[row][col]);
            dbf::mma_16(d, a0.x, a1.x, a0.y, a1.y, bh.x, bh.y);
            dbf::mma_16(d, a0.x, a1.x, a0.y, a1.y, bl.x, bl.y);
            dbf::mma_16(d, a0.z, a1.z, a0.w, a1.w, bh.z, bh.w);
            dbf::mma_16(d, a0.z, a1.z, a0.w, a1.w, bl.z, bl.w);
        }
    }
}

// Merge for the same shapes: combines the splits' records of a unit, applies row block h of the layer's map
// to the merged key sums of all heads and normalises,
//   o_a = (sum_s f_s acc_v_s + W[h rows] sum_s f_s acc_k_s) / sum_s f_s l_s,   f_s = exp(m_s - max m).
// grid (U), 512 threads.  The product runs on warp-level MMAs: M = the head's 128 output channels (warps w and w + 8:
// rows 16 w .., each half of the input heads), N = the unit's g query heads (padded to 8), K = 8 x 128; A fragments straight
// from the map (16-byte loads: thread (row r, quarter t) holds columns 8 (t + 4 jj) .. + 7 of rows r and r + 8 of a
// 128-column block, the k slots of an MMA step follow that order in both operands), the key sums as bf16
// hi + lo in shared memory.  What it costs is memory latency (42 MB of records and 64 MB of map from L2 over 256 blocks):
// hence eight-byte loads with eight splits of two elements in flight, and 16 warps on the map's rows.
constexpr int MERGE_THREADS = 512, MERGE_PAD = 72 * 1024;     // + 46 KB of its own: one block to a multiprocessor, with half of it two
template <typename TO>
__global__ void __launch_bounds__(MERGE_THREADS)
decode_layer_merge_mma(const float* partial, const __nv_bfloat16* W, int L, int g, Plan pl,
                       TO* __restrict__ out) {
    constexpr int KD = HKV * 128;
    __shared__ __align__(16) __nv_bfloat16 akh[8][KD], akl[8][KD];          // 32 KB
    __shared__ float accv[8][128], pw[2][8][128], fs[8][32], Ls[8];
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int h = u % HKV, layer = (u / HKV) % L;
    const int row = lane >> 2, quarter = lane & 3;
    const float* rec0 = partial + (size_t)u * pl.s_max * g * REC;
    const long long c0 = (long long)(u / HKV) * pl.weight;
    const int n_splits = block_of_cost(c0 + pl.weight - 1, pl) - block_of_cost(c0, pl) + 1;
    for (int i = tid; i < (8 - g) * KD; i += MERGE_THREADS) {            // columns of B beyond the unit's heads
        akh[g + i / KD][i % KD] = __float2bfloat16_rn(0.f);
        akl[g + i / KD][i % KD] = __float2bfloat16_rn(0.f);
    }
    asm volatile("griddepcontrol.wait;\n" ::: "memory");                 // the streaming kernel's records
    // factors of the splits: warp a < g takes head a
    if (wid < g) {
        const float mj = lane < n_splits ? rec0[((size_t)lane * g + wid) * REC] : -INFINITY;
        const float lj = lane < n_splits ? rec0[((size_t)lane * g + wid) * REC + 1] : 0.f;
        const float M = warp_max(mj);
        const float f = mj > -INFINITY ? __expf(mj - M) : 0.f;
        fs[wid][lane] = f;
        const float Lsum = warp_sum(f * lj);
        if (lane == 0) Ls[wid] = Lsum;
    }
    __syncthreads();
    // merged sums: a thread has two neighbouring elements of a record's 128 + 1024 values
    constexpr int PAIRS = (128 + KD) / 2;
    for (int i = tid; i < g * PAIRS; i += MERGE_THREADS) {
        const int a = i / PAIRS, e = (i - a * PAIRS) * 2;
        const float* src = rec0 + (size_t)a * REC + 2 + e;
        float v0, v1;
        merge_two(src, n_splits, g, fs[a], v0, v1);
        if (e < 128) { accv[a][e] = v0; accv[a][e + 1] = v1; }
        else {
            const uint32_t hi = dbf::pack_bf16(v0, v1);
            *reinterpret_cast<uint32_t*>(&akh[a][e - 128]) = hi;
            *reinterpret_cast<uint32_t*>(&akl[a][e - 128]) = dbf::pack_bf16(v0 - __uint_as_float(hi << 16), v1 - __uint_as_float(hi & 0xffff0000u));
        }
    }
    __syncthreads();
    // rows 16 (wid % 8) .. of the head's block of the map times the key sums of four input heads
    {
        const int half = wid >> 3, r0 = 16 * (wid & 7) + row;
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        map_rows_times_keys(W + ((size_t)layer * KD + (size_t)h * 128 + r0) * KD, akh, akl, half, row, quarter, d);
        // d[0], d[1]: row `row`, heads 2 quarter and 2 quarter + 1; d[2], d[3]: row `row` + 8
        if (2 * quarter < g) { pw[half][2 * quarter][r0] = d[0]; pw[half][2 * quarter][r0 + 8] = d[2]; }
        if (2 * quarter + 1 < g) { pw[half][2 * quarter + 1][r0] = d[1]; pw[half][2 * quarter + 1][r0 + 8] = d[3]; }
    }
    __syncthreads();
    for (int i = tid; i < g * 128; i += MERGE_THREADS) {
        const int a = i >> 7, c = i & 127;
        store_out(out + ((size_t)u * g + a) * 128 + c, (accv[a][c] + (pw[0][a][c] + pw[1][a][c])) / Ls[a]);
    }
}

// The same for many units: a block takes `seqs` sequences of one (layer, head), whose query heads are the product's columns.  The
// map's rows, 256 KB a block, are what most of a merge fetches from L2 where units are many and their records few.  A kernel of its
// own: as two instances of one body the other one lost 1 to 5 % (a pair of 2215 rows 34.3 -> 36.1 us a step, 40 of 349 rows 52.6 -> 55.4).
// grid (layers * HKV * ceil(batch / seqs)), 512 threads, seqs * g <= 8.
template <typename TO>
__global__ void __launch_bounds__(MERGE_THREADS)
decode_layer_merge_shared(const float* partial, const __nv_bfloat16* W, int L, int g, int batch, int seqs, Plan pl,
                       TO* __restrict__ out) {
    constexpr int KD = HKV * 128;
    __shared__ __align__(16) __nv_bfloat16 akh[8][KD], akl[8][KD];          // 32 KB
    __shared__ float accv[8][128], pw[2][8][128], fs[8][32], Ls[8];
    __shared__ int splits[8];                            // records of a sequence
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int h = blockIdx.x % HKV, layer = (blockIdx.x / HKV) % L, b0 = blockIdx.x / (HKV * L) * seqs;
    const int n_heads = min(seqs, batch - b0) * g;       // columns in use: sequence b0 + a / g, query head a % g
    const int row = lane >> 2, quarter = lane & 3;
    auto pair_of = [&](int a) { return (b0 + a / g) * L + layer; };
    auto records_of = [&](int a) { return partial + (((size_t)pair_of(a) * HKV + h) * pl.s_max * g + a % g) * REC; };      // g * REC apart
    auto splits_of = [&](int a) {
        const long long c0 = (long long)pair_of(a) * pl.weight;
        return block_of_cost(c0 + pl.weight - 1, pl) - block_of_cost(c0, pl) + 1;
    };
    for (int i = tid; i < (8 - n_heads) * KD; i += MERGE_THREADS) {      // columns of B beyond them
        akh[n_heads + i / KD][i % KD] = __float2bfloat16_rn(0.f);
        akl[n_heads + i / KD][i % KD] = __float2bfloat16_rn(0.f);
    }
    asm volatile("griddepcontrol.wait;\n" ::: "memory");                 // the streaming kernel's records
    // factors of the splits: warp a < n_heads takes column a
    if (wid < n_heads) {
        const int n_splits = splits_of(wid);
        const float* rec = records_of(wid) + (size_t)lane * g * REC;
        const float mj = lane < n_splits ? rec[0] : -INFINITY;
        const float lj = lane < n_splits ? rec[1] : 0.f;
        const float M = warp_max(mj);
        const float f = mj > -INFINITY ? __expf(mj - M) : 0.f;
        fs[wid][lane] = f;
        const float Lsum = warp_sum(f * lj);
        if (lane == 0) { Ls[wid] = Lsum; splits[wid] = n_splits; }
    }
    __syncthreads();
    // merged sums: a thread has two neighbouring elements of a record's 128 + 1024 values
    constexpr int PAIRS = (128 + KD) / 2;
    for (int i = tid; i < n_heads * PAIRS; i += MERGE_THREADS) {
        const int a = i / PAIRS, e = (i - a * PAIRS) * 2, n_splits = splits[a];
        const float* src = records_of(a) + 2 + e;
        float v0, v1;
        merge_two(src, n_splits, g, fs[a], v0, v1);
        if (e < 128) { accv[a][e] = v0; accv[a][e + 1] = v1; }
        else {
            const uint32_t hi = dbf::pack_bf16(v0, v1);
            *reinterpret_cast<uint32_t*>(&akh[a][e - 128]) = hi;
            *reinterpret_cast<uint32_t*>(&akl[a][e - 128]) = dbf::pack_bf16(v0 - __uint_as_float(hi << 16), v1 - __uint_as_float(hi & 0xffff0000u));
        }
    }
    __syncthreads();
    // rows 16 (wid % 8) .. of the head's block of the map times the key sums of four input heads
    {
        const int half = wid >> 3, r0 = 16 * (wid & 7) + row;
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        map_rows_times_keys(W + ((size_t)layer * KD + (size_t)h * 128 + r0) * KD, akh, akl, half, row, quarter, d);
        // d[0], d[1]: row `row`, heads 2 quarter and 2 quarter + 1; d[2], d[3]: row `row` + 8
        if (2 * quarter < n_heads) { pw[half][2 * quarter][r0] = d[0]; pw[half][2 * quarter][r0 + 8] = d[2]; }
        if (2 * quarter + 1 < n_heads) { pw[half][2 * quarter + 1][r0] = d[1]; pw[half][2 * quarter + 1][r0 + 8] = d[3]; }
    }
    __syncthreads();
    for (int i = tid; i < n_heads * 128; i += MERGE_THREADS) {
        const int a = i >> 7, c = i & 127;
        store_out(out + (((size_t)pair_of(a) * HKV + h) * g + a % g) * 128 + c, (accv[a][c] + (pw[0][a][c] + pw[1][a][c])) / Ls[a]);
    }
}

}  // namespace dlm
}  // namespace vec
#endif
