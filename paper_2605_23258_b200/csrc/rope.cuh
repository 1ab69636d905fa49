// Turning a key back to fp32's own precision, on packed pairs: for 64-channel heads, which CUDA cores with fp64 angles served
// before the tensor-core kernels took them over.
#ifndef VECTOR_ROPE_CUH_
#define VECTOR_ROPE_CUH_

#include "common.cuh"
#include "tcgen05.cuh"

namespace vec {

// The phase of a channel pair (turns per position as a 64-bit fraction) as two signed words, hi 2^32 + lo, so that
// pos hi + (pos lo >> 32) is the angle in turns modulo one, exact to 2^-32, for positions of either sign.
struct RopePhase { int32_t hi, lo; };
__device__ __forceinline__ RopePhase rope_phase_words(unsigned long long phase) {
    RopePhase p;
    p.lo = (int32_t)(uint32_t)phase;
    p.hi = (int32_t)(uint32_t)((phase + 0x80000000ull) >> 32);
    return p;
}

// The angle at a position as a 32-bit fraction of a turn.
__device__ __forceinline__ uint32_t rope_angle(int32_t pos, RopePhase ph) {
    return (uint32_t)pos * (uint32_t)ph.hi + (uint32_t)__mulhi(pos, ph.lo);
}
// Sine and cosine of two such angles.  Integer arithmetic takes an angle to the nearest quarter turn and
// what remains of it, in [-pi/4, pi/4]; there the Taylor series about zero are good to 2e-9 (sine, five terms) and 2e-10 (cosine,
// six), and a quarter turn swaps the two or changes their signs.
__device__ __forceinline__ void rope_cos_sin2(uint32_t angle0, uint32_t angle1, uint64_t& cs2, uint64_t& sn2) {
    // an eighth of a turn more: the upper two bits are the quarter turns, the rest less an eighth what remains
    const uint32_t u0 = angle0 + 0x20000000u, u1 = angle1 + 0x20000000u;
    const float r0 = (float)((int)(u0 & 0x3fffffffu) - 0x20000000), r1 = (float)((int)(u1 & 0x3fffffffu) - 0x20000000);
    const uint64_t z = tc::mul2(tc::pack2(r0, r1), tc::pack2(1.4629180792671596e-9f, 1.4629180792671596e-9f));      // 2 pi / 2^32
    const uint64_t zz = tc::mul2(z, z);
    auto both = [](float x) { return tc::pack2(x, x); };
    uint64_t s = tc::fma2(both(1.f / 362880.f), zz, both(-1.f / 5040.f));
    uint64_t c = tc::fma2(both(-1.f / 3628800.f), zz, both(1.f / 40320.f));
    s = tc::fma2(s, zz, both(1.f / 120.f));
    c = tc::fma2(c, zz, both(-1.f / 720.f));
    s = tc::fma2(s, zz, both(-1.f / 6.f));
    c = tc::fma2(c, zz, both(1.f / 24.f));
    s = tc::fma2(tc::mul2(s, zz), z, z);
    c = tc::fma2(c, zz, both(-0.5f));
    c = tc::fma2(c, zz, both(1.f));
    float s0, s1, c0, c1;
    tc::unpack2(s, s0, s1);
    tc::unpack2(c, c0, c1);
    auto turn = [](uint32_t u, float& cs, float& sn) {
        const bool odd = (u & 0x40000000u) != 0;
        const float a = odd ? sn : cs, b = odd ? cs : sn;
        cs = __uint_as_float(__float_as_uint(a) ^ ((u + 0x40000000u) & 0x80000000u));
        sn = __uint_as_float(__float_as_uint(b) ^ (u & 0x80000000u));
    };
    turn(u0, c0, s0);
    turn(u1, c1, s1);
    cs2 = tc::pack2(c0, c1);
    sn2 = tc::pack2(s0, s1);
}

// A pair of numbers as bf16 parts, each a part of what the ones before it leave.  Three are the upper halves of the words, cut off:
// together they hold all 24 bits.  Two are rounded, which halves what they lose and leaves it without a bias.
template <int PARTS>
__device__ __forceinline__ void split_bf16(float p0, float p1, uint32_t (&part)[PARTS]) {
#pragma unroll
    for (int i = 0; i < PARTS; ++i) {
        if constexpr (PARTS == 3) {
            part[i] = __byte_perm(__float_as_uint(p0), __float_as_uint(p1), 0x7632);
        } else {
            const __nv_bfloat162 v = __floats2bfloat162_rn(p0, p1);
            part[i] = *reinterpret_cast<const uint32_t*>(&v);
        }
        if (i + 1 < PARTS)
            tc::unpack2(tc::fma2(tc::pack2(part[i] << 16, part[i] & 0xffff0000u), tc::pack2(-1.f, -1.f), tc::pack2(p0, p1)), p0, p1);
    }
}

// Two channels x with their partners y (bf16, two to a register), turned back by their angles, in three parts each.
__device__ __forceinline__ void turn_back_parts(uint32_t x, uint32_t y, uint32_t angle0, uint32_t angle1, uint32_t (&xp)[3], uint32_t (&yp)[3]) {
    uint64_t cs, sn;
    rope_cos_sin2(angle0, angle1, cs, sn);
    const uint64_t x2 = tc::pack2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
    const uint64_t y2 = tc::pack2(__uint_as_float(y << 16), __uint_as_float(y & 0xffff0000u));
    float a, b;
    tc::unpack2(tc::fma2(x2, cs, tc::mul2(y2, sn)), a, b);
    split_bf16<3>(a, b, xp);
    tc::unpack2(tc::fma2(x2, tc::mul2(sn, tc::pack2(-1.f, -1.f)), tc::mul2(y2, cs)), a, b);
    split_bf16<3>(a, b, yp);
}

}  // namespace vec
#endif
