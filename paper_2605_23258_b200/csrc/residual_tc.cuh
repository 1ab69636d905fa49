// Reconstruction residual of Step 2 on the tensor cores (bf16, head_dim D = 64 or 128):
//   eps[p] = || v_i - W k~_i ||^2,  i = idx[p],  k~ = the key, or under RoPE decoupling the key
//   turned back by its position (the token index itself), channel c pairing with c + D/2.
// The gather of the listed K and V rows is what costs (64 flop per byte: HBM-bound), so the
// kernel is built around keeping row loads in flight.  Per 128-row tile the accumulator in tensor
// memory is K_tile W^T (one chain of D / 16 tcgen05.mma); the epilogue subtracts the value row,
// which it reads from the tile's copy in shared memory, squares and adds along its TMEM lane.
//
// Persistent blocks (one per SM) own equal contiguous ranges of the global tile sequence.
//   loaders     (8 warps) cp.async gathers of K and V rows into the stages, written directly
//               in the 128-byte-swizzled layout the MMA reads; row indices are fetched one tile ahead.
//               Each thread gathers, for its rows, the 16-byte chunk qc of both key halves
//               (channels 8 qc.. and D/2 + 8 qc..) and the same two chunks of V.
//   one warp    MMA issuer, TMEM owner; also TMA-loads the unit's W when the range enters a new unit
//   4 warps     epilogue: thread = row
// Without RoPE: stages of K | V (three of 64 KB at D = 128, five of 32 KB at D = 64), tiles published
// one behind the one being issued: the fence that comes before waits for the newer tiles' copies too, so that a tile held back
// longer waits for more of them.  256 lists of 9829 of 32768 tokens, routed, us: one behind 261 at D = 128 and 189 at D = 64, all
// stages but one 267 and 200.
// With RoPE: the turned key is no longer a bf16 number, so it goes to the tensor cores as a bf16
// pair hi + lo (two chains over the same W), which keeps it to 2^-17 relative; two stages of
// K hi | K lo | V (96 KB each).  At D = 64 it goes there as three bf16 parts, turned to fp32's own precision (rope.cuh): 64 KB a stage;
// residuals are then off by 1.1e-7 to 1.4e-7 (2-norm, 64 units of 2000 rows; 2.6e-6 with two parts, 1.6e-7 on CUDA cores), and four
// sequences of 8 layers of 20011 tokens take 153 us to route (137 and 942).  A loader thread takes its chunks of the keys straight into registers,
// a pass of the next tile requested as soon as that pass of this tile has been read, turns its eight channel
// pairs of each of its rows back and writes hi and lo; the values follow with cp.async and a barrier of
// their own.  With the keys landing in the stage, a tile's loads waited for the epilogue of the tile before last.
#ifndef VECTOR_RESIDUAL_TC_CUH_
#define VECTOR_RESIDUAL_TC_CUH_

#include "common.cuh"
#include "internal.h"
#include "rope.cuh"
#include "tcgen05.cuh"
#include "tma.cuh"

namespace vec {
namespace rtc {

constexpr int BOX_BYTES = 16384;                           // 128 rows x 128 bytes
constexpr int TILE = 128;
constexpr int EPI_WARPS = 4;

struct Params {
    int U, LH, n_idx, tpu;       // units, maps, rows per unit, tiles per unit
    long long N, n_tiles;        // keys per unit, U * tpu
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// One arrival on `bar` when all cp.async of this thread so far have completed.
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(tma::smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ long long range_begin(int b, long long n_tiles, int B) { return (long long)b * n_tiles / B; }
// Position in the global tile sequence: unit and tile inside it.  Stepped along, not divided out: the 64-bit divisions of
// every role and tile cost 3 % of the pass (route and compaction of 256 units of 32768 tokens: 593 -> 573 us).
struct Cursor {
    int u, t;
    __device__ __forceinline__ void next(int tpu) { if (++t == tpu) { t = 0; ++u; } }
};
__device__ __forceinline__ Cursor cursor_at(long long tile, int tpu) {
    Cursor c;
    c.u = (int)(tile / tpu);
    c.t = (int)(tile - (long long)c.u * tpu);
    return c;
}

template <int D, bool ROPE> struct RCfg {
    static constexpr int OPERAND_BYTES = (D / 64) * BOX_BYTES;     // 128 rows of D bf16 as D / 64 swizzled boxes
    static constexpr int W_BYTES = 2 * D * D;
    static constexpr int STAGES = ROPE ? 2 : D == 128 ? 3 : 5;
    static constexpr int PARTS = !ROPE ? 1 : D == 128 ? 2 : 3;     // bf16 parts of a key
    static constexpr int STAGE_BYTES = (PARTS + 1) * OPERAND_BYTES;
    static constexpr int V_OFFSET = PARTS * OPERAND_BYTES;
    static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + W_BYTES + 1024;
    static constexpr int TMEM_COLS = STAGES * D <= 128 ? 128 : STAGES * D <= 256 ? 256 : 512;   // one D-column accumulator per stage
    static constexpr int LOADER_WARPS = 8;
    static constexpr int THREADS = 32 * (LOADER_WARPS + 1 + EPI_WARPS);
};
struct RSync {
    uint64_t full[5], done[5], empty[5];
    uint64_t v_full[2];              // RoPE: the stage's values have landed
    uint64_t w_full, w_empty;
    uint32_t tmem_base;
};

// grid: min(multiprocessors, n_tiles) blocks, RCfg::THREADS threads, RCfg::SMEM_BYTES dynamic shared memory.
template <int D, bool ROPE>
__global__ void __launch_bounds__(RCfg<D, ROPE>::THREADS, 1)
residual_tc(const __nv_bfloat16* K, const __nv_bfloat16* V,
                 const __grid_constant__ CUtensorMap mapW, const int32_t* idx, const Params P,
                 const __grid_constant__ RopePhases rope, float* __restrict__ eps, int* __restrict__ fault) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ RSync sy;
    using C = RCfg<D, ROPE>;
    constexpr int STAGES = C::STAGES, R_STAGE_BYTES = C::STAGE_BYTES, TMEM_COLS = C::TMEM_COLS, R_LOADER_WARPS = C::LOADER_WARPS;
    constexpr int OPERAND_BYTES = C::OPERAND_BYTES;
    constexpr int LPR = D / 16, RPP = 32 * R_LOADER_WARPS / LPR, PASSES = TILE / RPP;    // loader threads a row, rows a pass, passes
    __shared__ unsigned long long phase_s[64];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* stage0 = smem;
    unsigned char* Ws = smem + STAGES * R_STAGE_BYTES;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long gt_lo = range_begin(blockIdx.x, P.n_tiles, gridDim.x);
    const long long gt_hi = range_begin(blockIdx.x + 1, P.n_tiles, gridDim.x);
    const int n_my = (int)(gt_hi - gt_lo);

    // A programmatic dependent of the kernel that writes idx (inside vector_route), whose other blocks may still run: the loaders,
    // the only readers of idx, wait for it below.  W is loaded ahead of that: the selection does not touch it, and what came
    // before the selection has finished, since it waits before it lets this kernel start.
    if (tid < 64) phase_s[tid] = rope.phase[tid];
    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < STAGES; ++s) {
            tma::mbar_init(&sy.full[s], 32 * R_LOADER_WARPS);
            tma::mbar_init(&sy.done[s], 1);
            tma::mbar_init(&sy.empty[s], EPI_WARPS);
            if (ROPE) tma::mbar_init(&sy.v_full[s], 32 * R_LOADER_WARPS);
        }
        tma::mbar_init(&sy.w_full, 1);
        tma::mbar_init(&sy.w_empty, 1);
        tma::mbar_fence_init();
    }
    if (warp == R_LOADER_WARPS) {
        tc::tmem_alloc(&sy.tmem_base, TMEM_COLS);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();

    if (warp < R_LOADER_WARPS) {
        // ------------------------------------------------------------------ loaders
        const int qc = tid & (LPR - 1), rsub = tid / LPR;           // chunk of each half, row inside a pass
        const uint32_t dst_thread = (uint32_t)rsub * 128u + (uint32_t)((qc ^ (rsub & 7)) << 4);   // + pass * PASS_BYTES
        // the same chunk of the other half: in the second box, or LPR chunks further in the row
        const uint32_t other = D == 128 ? (uint32_t)BOX_BYTES : (uint32_t)(((qc + LPR) ^ (rsub & 7)) << 4) - (uint32_t)((qc ^ (rsub & 7)) << 4);
        constexpr uint32_t PASS_BYTES = RPP * 128;
        uint2 fr[8];                                                 // phases of this thread's eight channel pairs; D = 64: as signed words
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            fr[e] = reinterpret_cast<const uint2*>(phase_s)[qc * 8 + e];
            if constexpr (D == 64) {
                const RopePhase w = rope_phase_words(phase_s[qc * 8 + e]);
                fr[e] = make_uint2((uint32_t)w.lo, (uint32_t)w.hi);
            }
        }
        int32_t cur[PASSES], nxt[PASSES];
        Cursor at = cursor_at(gt_lo, P.tpu), ahead = at;             // the tile at hand; the tile whose rows are fetched next
        auto fetch_idx = [&](int32_t (&out)[PASSES]) {
#pragma unroll
            for (int p = 0; p < PASSES; ++p) {
                const int row = ahead.t * TILE + p * RPP + rsub;
                out[p] = row < P.n_idx ? idx[(size_t)ahead.u * P.n_idx + row] : -1;
            }
            ahead.next(P.tpu);
        };
        // An index outside the unit reads as a row of zeros.  Checked when the rows come up, not when they are fetched: the
        // check would wait for the fetch (2 900 of 7 000 cycles a tile with RoPE).
        auto check_idx = [&](int32_t (&rows)[PASSES]) {
#pragma unroll
            for (int p = 0; p < PASSES; ++p) rows[p] = (unsigned long long)rows[p] < (unsigned long long)P.N ? rows[p] : -1;
        };
        // RoPE: this thread's key chunks of a tile: per pass, eight channels of the first half and their partners.
        uint4 kx[PASSES], ky[PASSES];
        auto request = [&](const __nv_bfloat16* Ku, int p, int32_t row) {
            kx[p] = ky[p] = make_uint4(0u, 0u, 0u, 0u);                  // zero past the end of the list
            if (row >= 0) {
                const __nv_bfloat16* kr = Ku + (size_t)row * D;
                kx[p] = *reinterpret_cast<const uint4*>(kr);
                ky[p] = *reinterpret_cast<const uint4*>(kr + D / 2);
            }
        };
        // Turns the pairs of tile i (rows listed in pos), writes them to stage s and publishes it; a pass's registers take
        // the next tile's keys (rows listed in next_rows) as soon as they have been read.
        auto turn_back = [&](int i, int s, const int32_t (&pos)[PASSES], const int32_t (&next_rows)[PASSES], const __nv_bfloat16* K_next) {
            const uint32_t hi0 = tma::smem_u32(stage0 + s * R_STAGE_BYTES) + dst_thread, lo0 = hi0 + OPERAND_BYTES;
            auto store16 = [](uint32_t at, const uint32_t (&v)[4]) {
                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};\n" ::"r"(at), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
            };
#pragma unroll
            for (int p = 0; p < PASSES; ++p) {
                uint32_t xs[4] = {kx[p].x, kx[p].y, kx[p].z, kx[p].w}, ys[4] = {ky[p].x, ky[p].y, ky[p].z, ky[p].w}, xl[4], yl[4];
                if (i + 1 < n_my) request(K_next, p, next_rows[p]);
                const uint32_t tok = pos[p] >= 0 ? (uint32_t)pos[p] : 0u;      // rows past the list are zeros
                if constexpr (D == 64) {
                    uint32_t xp[3][4], yp[3][4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint32_t angle[2], xe[3], ye[3];
#pragma unroll
                        for (int h = 0; h < 2; ++h) angle[h] = rope_angle((int)tok, RopePhase{(int)fr[2 * e + h].y, (int)fr[2 * e + h].x});
                        turn_back_parts(xs[e], ys[e], angle[0], angle[1], xe, ye);
#pragma unroll
                        for (int i = 0; i < 3; ++i) { xp[i][e] = xe[i]; yp[i][e] = ye[i]; }
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        store16(hi0 + i * OPERAND_BYTES + p * PASS_BYTES, xp[i]);
                        store16(hi0 + i * OPERAND_BYTES + other + p * PASS_BYTES, yp[i]);
                    }
                    continue;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float x[2], y[2], cs[2], sn[2], xo[2], yo[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        x[h] = __uint_as_float(h ? (xs[e] & 0xffff0000u) : (xs[e] << 16));
                        y[h] = __uint_as_float(h ? (ys[e] & 0xffff0000u) : (ys[e] << 16));
                        rope_phase_cos_sin(tok, fr[2 * e + h], cs[h], sn[h]);
                    }
                    // both pairs of the word at once on the packed FMA path
                    const uint64_t x2 = tc::pack2(x[0], x[1]), y2 = tc::pack2(y[0], y[1]);
                    const uint64_t c2 = tc::pack2(cs[0], cs[1]), s2 = tc::pack2(sn[0], sn[1]);
                    tc::unpack2(tc::fma2(x2, c2, tc::mul2(y2, s2)), xo[0], xo[1]);
                    tc::unpack2(tc::fma2(y2, c2, tc::mul2(x2, tc::pack2(-sn[0], -sn[1]))), yo[0], yo[1]);
                    // hi = the pair rounded to bf16, lo = what the rounding left, again as bf16
                    xs[e] = pack2_bf16(xo[0], xo[1]);
                    ys[e] = pack2_bf16(yo[0], yo[1]);
                    xl[e] = pack2_bf16(xo[0] - __uint_as_float(xs[e] << 16), xo[1] - __uint_as_float(xs[e] & 0xffff0000u));
                    yl[e] = pack2_bf16(yo[0] - __uint_as_float(ys[e] << 16), yo[1] - __uint_as_float(ys[e] & 0xffff0000u));
                }
                store16(hi0 + p * PASS_BYTES, xs);
                store16(hi0 + other + p * PASS_BYTES, ys);
                store16(lo0 + p * PASS_BYTES, xl);
                store16(lo0 + other + p * PASS_BYTES, yl);
            }
            fence_async_proxy();
            tma::mbar_arrive(&sy.full[s]);
        };
        bool ok = true;
        asm volatile("griddepcontrol.wait;\n" ::: "memory");      // idx is complete and visible from here on
        asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
        if (n_my > 0) fetch_idx(cur);
        if constexpr (ROPE) {
            if (n_my > 0) {
                check_idx(cur);
#pragma unroll
                for (int p = 0; p < PASSES; ++p) request(K + (size_t)at.u * P.N * D + qc * 8, p, cur[p]);
            }
            if (n_my > 1) fetch_idx(nxt);
            for (int i = 0; i < n_my && ok; ++i) {
                const int s = i % STAGES, round = i / STAGES;
                int32_t after[PASSES];
                if (i + 2 < n_my) fetch_idx(after);
                if (i + 1 < n_my) check_idx(nxt);
                if (round > 0 && !tma::mbar_wait(&sy.empty[s], (round - 1) & 1, fault, 46)) { ok = false; break; }
                const uint32_t vdst = tma::smem_u32(stage0 + s * R_STAGE_BYTES) + C::V_OFFSET + dst_thread;
                const __nv_bfloat16* Vu = V + (size_t)at.u * P.N * D + qc * 8;
#pragma unroll
                for (int p = 0; p < PASSES; ++p) {
                    const size_t ro = cur[p] >= 0 ? (size_t)cur[p] * D : 0;
                    const uint32_t nb = cur[p] >= 0 ? 16u : 0u;
                    cp_async16(vdst + p * PASS_BYTES, Vu + ro, nb);
                    cp_async16(vdst + other + p * PASS_BYTES, Vu + ro + D / 2, nb);
                }
                cp_async_arrive(&sy.v_full[s]);          // arrives once this thread's copies have landed
                at.next(P.tpu);
                turn_back(i, s, cur, nxt, K + (size_t)at.u * P.N * D + qc * 8);
#pragma unroll
                for (int p = 0; p < PASSES; ++p) { cur[p] = nxt[p]; nxt[p] = after[p]; }
            }
            cp_async_wait_all();
        } else {
            for (int i = 0; i < n_my && ok; ++i) {
                const int s = i % STAGES, round = i / STAGES;
                if (i + 1 < n_my) fetch_idx(nxt);
                check_idx(cur);
                if (round > 0 && !tma::mbar_wait(&sy.empty[s], (round - 1) & 1, fault, 46)) { ok = false; break; }
                const uint32_t kdst = tma::smem_u32(stage0 + s * R_STAGE_BYTES) + dst_thread;
                const uint32_t vdst = kdst + C::V_OFFSET;
                const __nv_bfloat16* Ku = K + (size_t)at.u * P.N * D + qc * 8;
                const __nv_bfloat16* Vu = V + (size_t)at.u * P.N * D + qc * 8;
                at.next(P.tpu);
#pragma unroll
                for (int p = 0; p < PASSES; ++p) {
                    const bool valid = cur[p] >= 0;
                    const size_t ro = valid ? (size_t)cur[p] * D : 0;
                    const uint32_t nb = valid ? 16u : 0u;                  // zero fill past the end of the list
                    cp_async16(kdst + p * PASS_BYTES, Ku + ro, nb);
                    cp_async16(kdst + other + p * PASS_BYTES, Ku + ro + D / 2, nb);
                    cp_async16(vdst + p * PASS_BYTES, Vu + ro, nb);
                    cp_async16(vdst + other + p * PASS_BYTES, Vu + ro + D / 2, nb);
                }
                cp_async_commit();
                if (i >= 1) {                            // this thread's copies of the tile before this one have landed
                    cp_async_wait<1>();
                    fence_async_proxy();
                    tma::mbar_arrive(&sy.full[(i - 1) % STAGES]);
                }
#pragma unroll
                for (int p = 0; p < PASSES; ++p) cur[p] = nxt[p];
            }
            cp_async_wait<0>();
            if (ok && n_my > 0) { fence_async_proxy(); tma::mbar_arrive(&sy.full[(n_my - 1) % STAGES]); }
        }
    } else if (warp == R_LOADER_WARPS) {
        // ------------------------------------------------------------------ W loads and MMA issue
        if (lane == 0) {
            tma::prefetch_map(&mapW);
            const uint32_t w_addr = tma::smem_u32(Ws);
            const uint32_t idesc = tc::instr_desc(128, D);
            int cur_u = -1;
            uint32_t n_units = 0;
            Cursor at = cursor_at(gt_lo, P.tpu);
            for (int i = 0; i < n_my; ++i, at.next(P.tpu)) {
                const int s = i % STAGES, round = i / STAGES;
                const int u = at.u;
                if (u != cur_u) {
                    if (n_units > 0 && !tma::mbar_wait(&sy.w_empty, (n_units - 1) & 1, fault, 47)) break;
                    tma::mbar_expect_tx(&sy.w_full, C::W_BYTES);
#pragma unroll
                    for (int x = 0; x < D / 64; ++x) tma::load_3d(Ws + x * BOX_BYTES, &mapW, 64 * x, 0, u % P.LH, &sy.w_full);
                    if (!tma::mbar_wait(&sy.w_full, n_units & 1, fault, 48)) break;
                    cur_u = u;
                    ++n_units;
                }
                // the loaders start only once the kernel that writes idx has drained: do not spend this
                // thread's bounded polls on that kernel's run time (W, loaded above, is not its output)
                if (i == 0) asm volatile("griddepcontrol.wait;\n" ::: "memory");
                if (!tma::mbar_wait(&sy.full[s], round & 1, fault, 49)) break;
                tc::fence_after_sync();
                const uint32_t k_addr = tma::smem_u32(stage0 + s * R_STAGE_BYTES), d = sy.tmem_base + s * D;
#pragma unroll
                for (int x = 0; x < C::PARTS; ++x) {
                    const uint32_t part = k_addr + (D == 64 ? C::PARTS - 1 - x : x) * OPERAND_BYTES;     // three parts: the smallest first
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint32_t o = (ks >> 2) * BOX_BYTES + (ks & 3) * 32;
                        tc::mma_bf16(d, tc::smem_desc(part + o), tc::smem_desc(w_addr + o), idesc, x > 0 || ks > 0 ? 1u : 0u);
                    }
                }
                tc::mma_commit(&sy.done[s]);
                const bool last_of_unit = i + 1 == n_my || at.t + 1 == P.tpu;
                if (last_of_unit) tc::mma_commit(&sy.w_empty);
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3;                       // TMEM lanes this warp may read: 32 (warp % 4) ..
        const int r = quarter * 32 + lane;
        const uint32_t lane_addr = sy.tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t v_thread = (uint32_t)r * 128u;
        asm volatile("griddepcontrol.wait;\n" ::: "memory");      // as in the MMA thread: the waits below time this kernel only
        Cursor at = cursor_at(gt_lo, P.tpu);
        for (int i = 0; i < n_my; ++i, at.next(P.tpu)) {
            const int s = i % STAGES, round = i / STAGES;
            // the value rows were written by the loaders: observe their barrier, then the MMA's
            if (!tma::mbar_wait_warp(ROPE ? &sy.v_full[s] : &sy.full[s], round & 1, fault, 50)) break;
            if (!tma::mbar_wait_warp(&sy.done[s], round & 1, fault, 51)) break;
            tc::fence_after_sync();
            const int u = at.u, t = at.t;
            const uint32_t v_addr = tma::smem_u32(stage0 + s * R_STAGE_BYTES) + C::V_OFFSET + v_thread;
            uint32_t ra[32], rb[32];
            const uint32_t taddr = lane_addr + s * D;
            tc::tmem_ld32(taddr, ra);
            float e0 = 0.f, e1 = 0.f, e2 = 0.f, e3 = 0.f;
#pragma unroll
            for (int ch = 0; ch < D / 32; ++ch) {
                uint32_t (&cur)[32] = (ch & 1) ? rb : ra;
                uint32_t (&nxt)[32] = (ch & 1) ? ra : rb;
                uint32_t vv[16];                           // columns 32 ch .. 32 ch + 31 of the value row
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c16 = ch * 4 + q;            // 16-byte chunk of the 256-byte row
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                                 : "=r"(vv[4 * q]), "=r"(vv[4 * q + 1]), "=r"(vv[4 * q + 2]), "=r"(vv[4 * q + 3])
                                 : "r"(v_addr + (c16 >> 3) * BOX_BYTES + (((c16 & 7) ^ (r & 7)) << 4)));
                }
                tc::tmem_ld_wait(cur);
                if (ch + 1 < D / 32) tc::tmem_ld32(taddr + (ch + 1) * 32, nxt);
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float a = __uint_as_float(cur[j]) - __uint_as_float(vv[j >> 1] << 16);
                    const float b = __uint_as_float(cur[j + 1]) - __uint_as_float(vv[j >> 1] & 0xffff0000u);
                    const float c2 = __uint_as_float(cur[j + 2]) - __uint_as_float(vv[(j >> 1) + 1] << 16);
                    const float d2 = __uint_as_float(cur[j + 3]) - __uint_as_float(vv[(j >> 1) + 1] & 0xffff0000u);
                    e0 = fmaf(a, a, e0); e1 = fmaf(b, b, e1); e2 = fmaf(c2, c2, e2); e3 = fmaf(d2, d2, e3);
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tma::mbar_arrive(&sy.empty[s]);
            const int row = t * TILE + r;
            if (row < P.n_idx) eps[(size_t)u * P.n_idx + row] = (e0 + e1) + (e2 + e3);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == R_LOADER_WARPS) {
        __syncwarp();
        tc::fence_after_sync();
        tc::tmem_dealloc(sy.tmem_base, TMEM_COLS);
    }
}

}  // namespace rtc
}  // namespace vec
#endif
