// Streaming half of decode attention under RoPE decoupling (bf16, head_dim 64 or 128): the tiles, slots, barriers and
// records of decode_bf16.cuh, with the work of a tile spread over a team of warps.
//
// A key-only token's logit takes the key as stored, its contribution to the key sum the key turned back by the token's
// position.  Turning a key back costs a sine, a cosine and about ten instructions per channel pair, several times the rest
// of the tile, so that warps that own whole tiles (decode_bf16.cuh) would be bound by their own instruction chains.  A
// block therefore has teams, tile i to team i % TEAMS: three of five warps, or, at 64 channels, four of three:
//   score warp   S = Q K^T and the online softmax, 64 keys a step; it leaves the weights as MMA A fragments (hi and
//                lo halves; bf16 for values, fp16 for turned keys; at 64 channels three bf16 parts for both), the factor the
//                older sums take, and the keys' positions in one of the team's two step buffers
//   sum warps    each owns 16 of the channel pairs (c, c + D/2).  It takes the rows as MMA B fragments straight from
//                the slot -- both channels of a pair lie in the same thread's fragments -- turns them in registers (fp16,
//                eleven bits: a turned key is not a bf16 number and eight bits would not keep the key sum within the
//                tolerance of the output; |k| beyond 65504 saturates; at 64 channels three bf16 parts, rope.cuh)
//                and multiplies: nothing is written back
// and one producer thread.  What bounds it: HBM once all of this overlaps, and before that the score warps (about 3000
// cycles per 64 keys, 2300 of them busy) and the sum warps (2500 busy) waiting for one another.  Measured, 128 units of 3000
// retained + 6000 key-only rows, 393 MB, with the appended row and the merge: 86 us; 104 us with warps that owned whole tiles
// and twelve helpers that turned keys back in shared memory (a fence and three block barriers per 64 keys).
// 64 channels, 512 units of 1639 + 3276 rows: 197 us a step with the appended row, bound by the sum warps' instructions (about
// 1000 for 64 key-only rows; 114 us with fp16 keys, 1139 us on CUDA cores; sum warps of eight pairs 210, five teams 203, loops
// rolled up 207).  Error of an fp32 output against fp64, median over the heads: 1.8e-7 to 4.1e-7 (fp16: 1.1e-4, CUDA cores: 2.0e-7 to 5.5e-7).
// The angle is position * theta^(-2c/D), taken as the 32-bit product of the position and the
// channel's phase (turns per position as a fraction of 2^32), which is the angle modulo one turn; 64 channels: rope.cuh.
#ifndef VECTOR_DECODE_ROPE_CUH_
#define VECTOR_DECODE_ROPE_CUH_

#include "decode_bf16.cuh"

namespace vec {
namespace dbf {

// x and y, the two channels of eight pairs (two keys to a register), turned back by pos[] * phase and left as fp16.
__device__ __forceinline__ void turn_back(uint32_t& x, uint32_t& y, uint32_t pos0, uint32_t pos1, uint32_t phase) {
    float c0, s0, c1, s1, a, b;
    rope_phase32_cos_sin(pos0, phase, c0, s0);
    rope_phase32_cos_sin(pos1, phase, c1, s1);
    // both keys at once on the packed FMA path
    const uint64_t x2 = tc::pack2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
    const uint64_t y2 = tc::pack2(__uint_as_float(y << 16), __uint_as_float(y & 0xffff0000u));
    const uint64_t c2 = tc::pack2(c0, c1);
    tc::unpack2(tc::fma2(x2, c2, tc::mul2(y2, tc::pack2(s0, s1))), a, b);
    x = pack_f16(a, b);
    tc::unpack2(tc::fma2(y2, c2, tc::mul2(x2, tc::pack2(-s0, -s1))), a, b);
    y = pack_f16(a, b);
}

// The weights of a softmax step over the 64 keys at kbase, of which nrows >= 1 are valid.  The keys fill the 16 rows of the
// MMAs and the heads their eight columns, half the MMAs of the other way round: sc[j] holds keys 16 j + gid (, + 8) of heads
// 2 tig, + 1.  m, l (this lane's keys only) and alpha, the factor what was summed up before has to take: of the same heads.
template <int D>
__device__ __forceinline__ void score_step_keys(uint32_t kbase, int nrows, float scale_log2e, const uint32_t (&qa)[D / 16][2], int lane,
                                                float (&m)[2], float (&l)[2], float (&alpha)[2], float (&sc)[4][4]) {
    const int gid = lane >> 2, mat = lane >> 3, r8 = lane & 7;
    const uint32_t row = (uint32_t)(r8 + (mat & 1) * 8) * 128u, x = (uint32_t)(((mat >> 1) ^ r8) << 4);     // (rows 0-7 | 8-15) x (chunk lo | hi)
#pragma unroll
    for (int j = 0; j < 4; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t a0, a1, a2, a3;
            ldsm_x4(kbase + (ks >> 2) * BOX_BYTES + j * 16 * 128 + row + ((((2 * ks) & 7) << 4) ^ x), a0, a1, a2, a3);
            mma_16(sc[j], a0, a1, a2, a3, qa[ks][0], qa[ks][1]);
        }
    }
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            sc[j][e] = 16 * j + 8 * (e >> 1) + gid < nrows ? sc[j][e] * scale_log2e : -INFINITY;
            mx[e & 1] = fmaxf(mx[e & 1], sc[j][e]);
        }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < 2; ++e) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], o));
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float m_new = mx[e] > m[e] + (Cfg<D, true>::EXACT ? SLACK : 0.f) ? mx[e] : m[e];       // finite: key 0 of the step is valid for every head
        alpha[e] = tc::ex2(m[e] - m_new);                              // 0 on the first step
        m[e] = m_new;
        l[e] *= alpha[e];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            sc[j][e] = tc::ex2(sc[j][e] - m[e & 1]);
            l[e & 1] += sc[j][e];
        }
}

// A sum warp's part of a softmax step, 64 channels: rows times weights over 64 rows at base (this lane's place in its column
// tiles), in three bf16 parts each way.  acc takes the sums of 32 rows at a time, which start at zero (Cfg::EXACT); alpha is the
// factor of what it held.  st: the step buffer.  Products of parts that lie below 2^-24 of the whole come along where they cost
// nothing: a fragment holds all parts of the weights.
__device__ __forceinline__ void sum_step64(uint32_t st, uint32_t base, bool retained, bool with_third, float alpha, const RopePhase (&phase)[2],
                                           float (&acc)[2][2][4], int lane) {
    using C = Cfg<64, true>;
    const int tig = lane & 3;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        float sum[2][2][4];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int p = 0; p < 2; ++p) sum[x][p][0] = sum[x][p][1] = sum[x][p][2] = sum[x][p][3] = 0.f;
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {
            const int kk = 2 * half + k2;
            uint32_t a[4], third[2] = {0u, 0u}, rx[2][2], ry[2][2];       // B fragments: low and high channels, rows 0-7 | 8-15
            ldsm_x4(st + kk * 512 + lane * 16, a[0], a[1], a[2], a[3]);
            if (with_third)
                asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n"
                             : "=r"(third[0]), "=r"(third[1]) : "r"(st + C::STEP_THIRD + kk * 256 + (lane & 15) * 16));
            const uint32_t at = base + kk * 16 * 128;
            ldsm_x4_t(at, rx[0][0], rx[0][1], rx[1][0], rx[1][1]);
            ldsm_x4_t(at ^ 64u, ry[0][0], ry[0][1], ry[1][0], ry[1][1]);
            auto add = [&](float (&s)[4], uint32_t b0, uint32_t b1) { mma_16(s, a[0], a[1], a[2], a[3], b0, b1); };
            auto add_w3 = [&](float (&s)[4], uint32_t b0, uint32_t b1) { if (with_third) mma_16(s, 0u, third[0], 0u, third[1], b0, b1); };
            if (retained) {
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    add(sum[0][p], rx[p][0], rx[p][1]);
                    add(sum[1][p], ry[p][0], ry[p][1]);
                    add_w3(sum[0][p], rx[p][0], rx[p][1]);
                    add_w3(sum[1][p], ry[p][0], ry[p][1]);
                }
            } else {
                uint32_t xp[2][2][3], yp[2][2][3];                        // [column tile][rows 0-7 | 8-15][part]
#pragma unroll
                for (int r = 0; r < 2; ++r) {                             // rows 2 tig, + 1 of the eight
                    uint32_t pos0, pos1;
                    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];\n" : "=r"(pos0), "=r"(pos1) : "r"(st + C::STEP_POS + kk * 64 + r * 32 + tig * 8));
#pragma unroll
                    for (int p = 0; p < 2; ++p) turn_back_parts(rx[p][r], ry[p][r], rope_angle((int)pos0, phase[p]), rope_angle((int)pos1, phase[p]), xp[p][r], yp[p][r]);
                }
#pragma unroll
                for (int i = 2; i >= 0; --i)                              // the small parts first
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        if (i == 0) {
                            add_w3(sum[0][p], xp[p][0][0], xp[p][1][0]);
                            add_w3(sum[1][p], yp[p][0][0], yp[p][1][0]);
                        }
                        add(sum[0][p], xp[p][0][i], xp[p][1][i]);
                        add(sum[1][p], yp[p][0][i], yp[p][1][i]);
                    }
            }
        }
        const uint64_t f = tc::pack2(alpha, alpha);
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                    const uint64_t o = tc::pack2(acc[x][p][e], acc[x][p][e + 1]), s = tc::pack2(sum[x][p][e], sum[x][p][e + 1]);
                    tc::unpack2(half == 0 ? tc::fma2(o, f, s) : tc::add2(o, s), acc[x][p][e], acc[x][p][e + 1]);
                }
    }
}

// grid, shared memory, partial, CLUSTER: as for decode_stream_bf16.  Warps 0 .. TEAMS - 1 score, the next one is the producer, then
// come the sum warps, team by team.
template <int D, bool CLUSTER>
__global__ void __launch_bounds__(Cfg<D, true>::THREADS, 1)
decode_stream_rope(const __nv_bfloat16* q, const __grid_constant__ Maps maps, Plan pl, int n_ret, int n_apx, int g,
                   int LH, float scale_log2e, float* __restrict__ partial, int* __restrict__ fault,
                   const int32_t* apx_pos, long long cap_apx, const __grid_constant__ RopePhases rope,
                   const __nv_bfloat16* W, void* __restrict__ out, int out_f32) {
    using C = Cfg<D, true>;
    constexpr int HALF_BYTES = C::HALF_BYTES, SLOT_BYTES = C::SLOT_BYTES, SLOTS = C::SLOTS, TEAMS = C::CONSUMER_WARPS, SUM_WARPS = C::SUM_WARPS;
    constexpr int REC = C::REC, CREC = C::CREC, PAIRS = 2;                    // column tiles of 8 channel pairs of a sum warp
    constexpr int STEP_THIRD = C::STEP_THIRD, STEP_POS = C::STEP_POS, STEP_ALPHA = C::STEP_ALPHA;
    const bool twice = C::EXACT && g <= 4;             // MMA rows 4-7 repeat the heads and take the third parts of the weights
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[SLOTS], empty_bar[SLOTS];
    __shared__ __align__(8) uint64_t step_full[TEAMS][2], step_empty[TEAMS][2];
    // 128B-swizzled TMA boxes want 1024-byte aligned destinations
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wq = tid >> 5;
    long long gt_lo, gt_hi;
    block_range<CLUSTER>(pl, gt_lo, gt_hi);
    const int n_my = (int)(gt_hi - gt_lo);
    const int u0 = (int)(gt_lo / pl.n_tiles), u_last = (int)((gt_hi - 1) / pl.n_tiles);
    float* const recs = reinterpret_cast<float*>(smem + SLOTS * SLOT_BYTES + C::P_BYTES);      // CLUSTER: the teams' records

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) { tma::mbar_init(&full_bar[s], 1); tma::mbar_init(&empty_bar[s], SUM_WARPS); }
#pragma unroll
        for (int w = 0; w < TEAMS; ++w)
#pragma unroll
            for (int k = 0; k < 2; ++k) { tma::mbar_init(&step_full[w][k], 1); tma::mbar_init(&step_empty[w][k], SUM_WARPS); }
        tma::mbar_fence_init();
    }
    // Launched as a programmatic dependent itself, and the merge kernel of this one: as in decode_stream_bf16.
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
            cluster_merge<D, true>(recs, smem, Wu, g, reinterpret_cast<char*>(out) + (size_t)u0 * g * D * (out_f32 ? 4 : 2),
                                   out_f32 != 0);
    };
    if (wq == TEAMS) {
        // ------------------------------------------------------------------ producer
        if (lane == 0) produce<D, true>(maps, pl, gt_lo, n_my, smem, full_bar, empty_bar, fault);
        // the sum warps wait on every tile's full barrier, so no copy outlives the block
        __syncwarp();
        merge_unit();
        return;
    }
    const bool scorer = wq < TEAMS;
    const int team = scorer ? wq : (wq - TEAMS - 1) / SUM_WARPS;
    const int gid = lane >> 2, tig = lane & 3;
    const uint32_t steps = tma::smem_u32(smem + SLOTS * SLOT_BYTES) + team * 2 * C::STEP_BYTES;
    auto record_of = [&](int unit, int head) -> float* {
        if (CLUSTER) return recs + (team * g + head) * CREC;
        int slot = b - block_of_tile((long long)unit * pl.n_tiles, pl);
        if (slot < 0 || slot >= pl.s_max) { atomicCAS(fault, 0, 5); slot = 0; }     // cannot happen; never write out of bounds
        return partial + ((((size_t)unit * pl.s_max + slot) * TEAMS + team) * g + head) * REC;
    };
    // The team's warps walk the same tiles and steps; a warp whose wait gave up walks on and touches nothing.
    int i = team;                                      // index into the block's tile sequence
    int n_step = 0;                                    // steps of the team so far: step n uses buffer n & 1
    bool ok = true;

    if (scorer) {
        // ------------------------------------------------------------------ scores and softmax
        uint32_t qa[D / 16][2];
        for (int u = u0; u <= u_last; ++u) {
            const long long unit_end = (long long)(u + 1) * pl.n_tiles - gt_lo;     // first sequence index past the unit
            bool loaded = false, keys = false;         // keys: there were key-only tiles
            float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, v_scale[2] = {1.f, 1.f};      // of heads 2 tig, + 1
            for (; i < n_my && i < unit_end; i += TEAMS) {
                const int s = i % SLOTS, t = (int)(gt_lo + i - (long long)u * pl.n_tiles);
                const bool retained = t < pl.n_rt;
                const int r0 = retained ? t * KEYS : (t - pl.n_rt) * 2 * KEYS;
                const int rows = retained ? min(KEYS, n_ret - r0) : min(2 * KEYS, n_apx - r0);
                uint32_t pos[4] = {0, 0, 0, 0};        // of rows lane + 32 k, on their way while the tile is
                if (!retained) {
                    const int32_t* pr = apx_pos + (size_t)u * cap_apx + r0 + lane;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (lane + 32 * k < rows) pos[k] = (uint32_t)pr[32 * k];
                }
                if (ok) {
                    if (!loaded) { load_queries<D>(q, u, g, lane, qa, twice); loaded = true; }
                    ok = tma::mbar_wait_warp(&full_bar[s], (i / SLOTS) & 1, fault, 2);
                }
                if (!retained && !keys) { keys = true; v_scale[0] = v_scale[1] = 1.f; }       // the value sums are parked at this maximum
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    const int nrows = min(KEYS, rows - h * KEYS);
                    if (nrows <= 0) break;
                    const int k = n_step & 1, round = n_step >> 1;
                    ++n_step;
                    if (!ok) continue;
                    float sc[4][4], alpha[2];
                    score_step_keys<D>(tma::smem_u32(smem + s * SLOT_BYTES + h * HALF_BYTES), nrows, scale_log2e, qa, lane, m, l, alpha, sc);
                    v_scale[0] *= alpha[0];
                    v_scale[1] *= alpha[1];
                    if (round > 0) ok = tma::mbar_wait_warp(&step_empty[team][k], (round - 1) & 1, fault, 3);
                    if (!ok) continue;
                    const uint32_t st = steps + k * C::STEP_BYTES;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint32_t hi[2], lo[2], third[2];         // keys gid and gid + 8 of the 16
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float p0 = sc[j][2 * e], p1 = sc[j][2 * e + 1];
                            if constexpr (C::EXACT) {
                                uint32_t part[3];
                                split_bf16(p0, p1, part);
                                const bool upper = twice && tig >= 2;
                                hi[e] = upper ? part[2] : part[0];
                                lo[e] = upper ? 0u : part[1];
                                third[e] = part[2];
                            } else if (retained) {
                                hi[e] = pack_bf16(p0, p1);
                                lo[e] = pack_bf16(p0 - __uint_as_float(hi[e] << 16), p1 - __uint_as_float(hi[e] & 0xffff0000u));
                            } else {
                                hi[e] = pack_f16(p0, p1);
                                lo[e] = pack_f16(p0 - f16_lo(hi[e]), p1 - f16_hi(hi[e]));
                            }
                        }
                        asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};\n" ::"r"(st + j * 512 + lane * 16),
                                     "r"(hi[0]), "r"(lo[0]), "r"(hi[1]), "r"(lo[1]) : "memory");
                        if (C::EXACT && !twice)
                            asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};\n"
                                         ::"r"(st + STEP_THIRD + j * 256 + (lane & 15) * 16), "r"(third[0]), "r"(third[1]) : "memory");
                    }
                    if (!retained) {
                        asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(st + STEP_POS + lane * 4), "r"(h ? pos[2] : pos[0]) : "memory");
                        asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(st + STEP_POS + 128 + lane * 4), "r"(h ? pos[3] : pos[1]) : "memory");
                    }
                    if (lane < 4) asm volatile("st.shared.v2.f32 [%0], {%1,%2};\n" ::"r"(st + STEP_ALPHA + lane * 8), "f"(alpha[0]), "f"(alpha[1]) : "memory");
                    __syncwarp();
                    if (lane == 0) tma::mbar_arrive(&step_full[team][k]);
                }
            }
            // the headers of the team's record of the unit (m = -inf if it met none of its tiles)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) l[e] += __shfl_xor_sync(0xffffffffu, l[e], o);
                if (lane < 4 && 2 * lane + e < g)
                    *reinterpret_cast<float4*>(record_of(u, 2 * lane + e)) = make_float4(m[e] * 0.69314718055994531f, l[e], keys ? v_scale[e] : 1.f, keys ? 1.f : 0.f);
            }
        }
        __syncwarp();
        merge_unit();
        return;
    }
    // ---------------------------------------------------------------------- sums
    // Warp `part` of the team: channel pairs 8 PAIRS part .. + 8 PAIRS - 1, i.e. column tiles PAIRS part + p and D/16 + PAIRS part + p.
    const int part = (wq - TEAMS - 1) % SUM_WARPS;
    const int mat = lane >> 3, r8 = lane & 7;
    RopePhase phase[PAIRS];                            // of channel pair 8 (PAIRS part + p) + gid; not EXACT: hi alone, the phase rounded to 32 bits
#pragma unroll
    for (int p = 0; p < PAIRS; ++p) phase[p] = rope_phase_words(rope.phase[8 * (PAIRS * part + p) + gid]);
    float acc[2][PAIRS][4];                            // [low | high channel of the pair][column tile][rows of first (and third) parts | of second parts]
    auto zero_acc = [&]() {
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int p = 0; p < PAIRS; ++p) acc[x][p][0] = acc[x][p][1] = acc[x][p][2] = acc[x][p][3] = 0.f;
    };
    auto add_third = [&]() {                           // the whole warp, before store_acc: the third parts' sums to their heads' rows
        if (twice) {
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
                for (int p = 0; p < PAIRS; ++p) {
                    acc[x][p][2] += __shfl_xor_sync(0xffffffffu, acc[x][p][0], 16);
                    acc[x][p][3] += __shfl_xor_sync(0xffffffffu, acc[x][p][1], 16);
                }
        }
    };
    auto store_acc = [&](float* dst) {
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int p = 0; p < PAIRS; ++p)
                *reinterpret_cast<float2*>(dst + x * (D / 2) + 8 * (PAIRS * part + p) + 2 * tig) =
                    make_float2(acc[x][p][0] + acc[x][p][2], acc[x][p][1] + acc[x][p][3]);
    };
    // Where a lane's rows of its column tiles lie within 16 rows at a multiple of 16 (ldmatrix.trans, swizzled): matrices
    // (tile | tile + 1) x (rows 0-7 | 8-15), the partner channels one box further, or half a row at 64 channels.
    const uint32_t frag = (uint32_t)(r8 + (mat & 1) * 8) * 128u + (uint32_t)(((2 * part + (mat >> 1)) ^ r8) << 4);
    zero_acc();
    for (int u = u0; u <= u_last; ++u) {
        const long long unit_end = (long long)(u + 1) * pl.n_tiles - gt_lo;
        bool any = false, parked = false;
        for (; i < n_my && i < unit_end; i += TEAMS) {
            const int s = i % SLOTS, t = (int)(gt_lo + i - (long long)u * pl.n_tiles);
            const bool retained = t < pl.n_rt;
            const int halves = !retained && n_apx - (t - pl.n_rt) * 2 * KEYS > KEYS ? 2 : 1;
            any = true;
            if (ok) ok = tma::mbar_wait_warp(&full_bar[s], (i / SLOTS) & 1, fault, 2);
            if (!retained && !parked) {                // the unit's first key-only keys: park sum p v
                add_third();
                if (gid < g) store_acc(record_of(u, gid) + 4);
                zero_acc();
                parked = true;
            }
#pragma unroll 1
            for (int h = 0; h < halves; ++h) {
                const int k = n_step & 1, round = n_step >> 1;
                ++n_step;
                if (ok) ok = tma::mbar_wait_warp(&step_full[team][k], round & 1, fault, 4);
                if (!ok) continue;
                const uint32_t st = steps + k * C::STEP_BYTES;
                const uint32_t base = tma::smem_u32(smem + s * SLOT_BYTES) + (retained ? HALF_BYTES : h * HALF_BYTES) + frag;
                float alpha;
                asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(alpha) : "r"(st + STEP_ALPHA + gid * 4));
                if constexpr (C::EXACT) {
                    sum_step64(st, base, retained, !twice, alpha, phase, acc, lane);
                } else {
#pragma unroll
                    for (int x = 0; x < 2; ++x)
#pragma unroll
                        for (int p = 0; p < PAIRS; ++p) { acc[x][p][0] *= alpha; acc[x][p][1] *= alpha; acc[x][p][2] *= alpha; acc[x][p][3] *= alpha; }
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        uint32_t a[4], rx[PAIRS][2], ry[PAIRS][2];            // B fragments: low and high channels, rows 0-7 | 8-15
                        ldsm_x4(st + kk * 512 + lane * 16, a[0], a[1], a[2], a[3]);
                        const uint32_t at = base + kk * 16 * 128;
                        ldsm_x4_t(at, rx[0][0], rx[0][1], rx[1][0], rx[1][1]);
                        ldsm_x4_t(D == 128 ? at + BOX_BYTES : at ^ 64u, ry[0][0], ry[0][1], ry[1][0], ry[1][1]);
                        if (retained) {
#pragma unroll
                            for (int p = 0; p < PAIRS; ++p) {
                                mma_16(acc[0][p], a[0], a[1], a[2], a[3], rx[p][0], rx[p][1]);
                                mma_16(acc[1][p], a[0], a[1], a[2], a[3], ry[p][0], ry[p][1]);
                            }
                        } else {
#pragma unroll
                            for (int r = 0; r < 2; ++r) {                     // rows 2 tig, + 1 of the eight
                                uint32_t pos0, pos1;
                                asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];\n" : "=r"(pos0), "=r"(pos1) : "r"(st + STEP_POS + kk * 64 + r * 32 + tig * 8));
#pragma unroll
                                for (int p = 0; p < PAIRS; ++p) turn_back(rx[p][r], ry[p][r], pos0, pos1, (uint32_t)phase[p].hi);
                            }
#pragma unroll
                            for (int p = 0; p < PAIRS; ++p) {
                                mma_16_f16(acc[0][p], a[0], a[1], a[2], a[3], rx[p][0], rx[p][1]);
                                mma_16_f16(acc[1][p], a[0], a[1], a[2], a[3], ry[p][0], ry[p][1]);
                            }
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) tma::mbar_arrive(&step_empty[team][k]);
            }
            if (ok && lane == 0) tma::mbar_arrive(&empty_bar[s]);
        }
        // the unit's sums; the cluster's merge reads no more of them than the header says
        add_third();
        if (CLUSTER) {
            // the slot that takes the key sums is the team's, and may hold its last tile
            asm volatile("bar.sync %0, %1;\n" ::"r"(2 + team), "n"(32 * SUM_WARPS) : "memory");
            if (gid < g && parked) store_acc(reinterpret_cast<float*>(smem + (SLOTS - TEAMS + team) * SLOT_BYTES) + gid * D);
            else if (gid < g && any) store_acc(record_of(u, gid) + 4);
        } else if (gid < g) {
            float* rec = record_of(u, gid);
            store_acc(rec + (parked ? 4 + D : 4));
            if (!parked) {
                zero_acc();
                store_acc(rec + 4 + D);
            }
        }
        zero_acc();
    }
    __syncwarp();
    merge_unit();
}

}  // namespace dbf
}  // namespace vec
#endif  // VECTOR_DECODE_ROPE_CUH_
