// A consumer's error head riding on the second pass of the kernel that produces its input error.
#pragma once
#include "eoq_device.cuh"
#include "eoq_internal.h"

namespace eoq {

// The error head of a layer (e1 = e * [x4 > 0], e3 = Q_e(gamma * e1), sum of e1, sum of e1 * x2) can ride on the second
// pass of the kernel that produces e: Q_e is monotonic in |.|, so max |e1| is the code of the largest masked |sum|, which
// the producer's first pass reduces beside its own maximum.  NextHead holds what the second pass needs.
struct NextHead {
    uint32_t g;         // gamma code
    float scale, rest;  // R(gamma * e1 * 2^(7 - t3)) = one fused multiply-add (see prescale_apply_kernel)
    uint32_t M3;        // max |gamma * e1|
    int t3;
};
constexpr uint32_t kHeadMagic = 0x4B400000u;  // 1.5 * 2^23

__device__ __forceinline__ NextHead next_head_setup(const int32_t *gamma_dev, uint32_t max_e1, DeviceState *dev)
{
    int gamma = __ldg(gamma_dev);
    if (gamma < -32768 || gamma > 32767) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&dev->status, EOQ_DEV_RANGE);
        gamma = gamma < 0 ? -32768 : 32767;
    }
    NextHead nh;
    nh.g = (uint32_t)gamma;
    nh.M3 = max_e1 * (uint32_t)abs(gamma);
    nh.t3 = nh.M3 ? round_log2_u32(nh.M3) : 7;
    nh.scale = __int_as_float((127 + 7 - nh.t3) << 23);
    nh.rest = 12582912.0f - 12582912.0f * nh.scale;
    return nh;
}

__device__ __forceinline__ int next_head_code(const NextHead &nh, int e1)
{
    const uint32_t biased = nh.g * (uint32_t)e1 + kHeadMagic;
    const int v = (int)(__float_as_uint(__fmaf_rn(__uint_as_float(biased), nh.scale, nh.rest)) - kHeadMagic);
    return v < -127 ? -127 : (v > 127 ? 127 : v);
}

// the codes of four errors: the subtraction of the magic number and the lower clamp are one instruction, the pack saturates
// at 127
__device__ __forceinline__ uint32_t next_head_codes(const NextHead &nh, uint32_t e1)
{
    uint32_t biased[4];
    if (nh.g < 256u) {   // gamma below 2 (codes below 256): a byte dot product takes its code out of the word and scales it
#pragma unroll
        for (int k = 0; k < 4; ++k) biased[k] = dot4_s8_u8(e1, nh.g << (8 * k), kHeadMagic);
    } else {
        const int32_t e[4] = {sbyte<0>(e1), sbyte<1>(e1), sbyte<2>(e1), sbyte<3>(e1)};
#pragma unroll
        for (int k = 0; k < 4; ++k) biased[k] = nh.g * (uint32_t)e[k] + kHeadMagic;
    }
    int32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = __viaddmax_s32((int32_t)__float_as_uint(__fmaf_rn(__uint_as_float(biased[k]), nh.scale, nh.rest)), -(int32_t)kHeadMagic, -127);
    }
    return pack4_sat(v[0], v[1], v[2], v[3]);
}

// exponent of e3 given the exponent p0 of e (the head sees e at p0 - 7 after the multiplication by gamma's grid)
__device__ __forceinline__ void next_head_exponent(const NextHead &nh, int p0, int32_t *e3_exp, DeviceState *dev)
{
    *e3_exp = nh.M3 ? p0 - 7 + nh.t3 - 7 : p0 - 7;
    if (!nh.M3) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
}


// Join of two error streams: both at the smaller exponent, added exactly; an operand more than 31 octaves below the
// other is dropped.
struct JoinShift {
    int sa, sb, p;  // left shifts of the two operands (-1: operand dropped) and the exponent of the sums
};
__device__ __forceinline__ JoinShift join_shift(int pa, int pb)
{
    JoinShift j;
    const int p = min(pa, pb);
    j.sa = pa - p;
    j.sb = pb - p;
    j.p = p;
    if (j.sa > 31) { j.sb = -1; j.sa = 0; j.p = pa; }        // b lies more than 31 octaves below a
    else if (j.sb > 31) { j.sa = -1; j.sb = 0; j.p = pb; }
    return j;
}
// The sums by one two-byte dot product each, a 16-bit factor per operand (0: dropped).  Exponents up to kJoinNear octaves apart
// give the exact sums, below 2^22.  Beyond (`far`), with |code| <= 128, the order of |sum| is that of the higher operand's |code|
// first and of the lower one's share second, for any distance of 9 or more: the maxima are taken at a distance of kJoinFar and
// brought to the true one at the end.  (A form in 64 bits for such exponents, which a diverging run meets in most of its
// joins, is gone: Q_e of 12.8 M sums with the maxima 28.7 -> 12.6 us, the join with the next head 29.8 -> 13.9.)
constexpr int kJoinNear = 14, kJoinFar = 9;
struct JoinMul {
    int gap;
    bool far, a_high;
    uint32_t pair;   // factor of a | factor of b << 16
};
__device__ __forceinline__ JoinMul join_mul(const JoinShift &j)
{
    JoinMul m;
    m.gap = max(j.sa, j.sb);
    m.far = m.gap > kJoinNear;
    m.a_high = j.sa > j.sb;
    const int up = m.far ? kJoinFar : m.gap;
    const uint32_t high = 1u << up, low = (j.sa | j.sb) < 0 ? 0u : 1u;   // (a dropped operand: the other one alone)
    m.pair = m.a_high ? high | low << 16 : low | high << 16;
    return m;
}
// four sums, each plus `bias` (codes of a and b in a word each)
__device__ __forceinline__ void join_sums(uint32_t pair, uint32_t a, uint32_t b, uint32_t bias, uint32_t (&s)[4])
{
    const uint32_t lo = __byte_perm(a, b, 0x5140), hi = __byte_perm(a, b, 0x7362);   // a0 b0 a1 b1, a2 b2 a3 b3
    s[0] = (uint32_t)__dp2a_lo((int)pair, (int)lo, (int)bias);
    s[1] = (uint32_t)__dp2a_hi((int)pair, (int)lo, (int)bias);
    s[2] = (uint32_t)__dp2a_lo((int)pair, (int)hi, (int)bias);
    s[3] = (uint32_t)__dp2a_hi((int)pair, (int)hi, (int)bias);
}
// the true |sum| behind the largest |sum| that join_sums gave
__device__ __forceinline__ unsigned long long join_magnitude(const JoinMul &m, uint32_t v)
{
    if (!m.far) return v;
    const long long high = (v + (1u << (kJoinFar - 1))) >> kJoinFar;
    return (unsigned long long)((high << m.gap) + ((long long)v - (high << kJoinFar)));
}

// Q_e of the sums under their maximum M, t = R(log2 M): factors for join_sums, and one multiply-add that rounds (see next_head_codes).
// Far operands: unless all its codes are zero (M <= 128), the higher operand's largest sets t >= gap, so the rounding is at bit 8 or
// above and the lower operand's share is at most half a unit, a half only at t = gap = 15, where the higher one's is a multiple of 128
// units and even: the code is that of the higher operand alone.
struct JoinCode {
    uint32_t pair;
    float scale, rest;
};
__device__ __forceinline__ JoinCode join_code(const JoinMul &m, unsigned long long M, int t)
{
    JoinCode c;
    int sh = t - 7;
    c.pair = m.pair;
    if (m.far) {
        const bool high = M > 128;
        c.pair = high == m.a_high ? 1u : 1u << 16;
        if (high) sh -= m.gap;
    }
    c.scale = __int_as_float((127 - sh) << 23);               // -7 <= sh <= 14
    c.rest = 12582912.0f - 12582912.0f * c.scale;             // exact
    return c;
}

}  // namespace eoq
