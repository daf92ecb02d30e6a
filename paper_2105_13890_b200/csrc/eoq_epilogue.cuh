// Pieces shared by the GEMM kernels: bounded barrier waits, and the register epilogues of the
// forward chain and of error back-propagation (arXiv 2105.13890, Sec. 3.2.1).
#pragma once
#include "eoq_device.cuh"
#include "eoq_internal.h"

namespace eoq {

struct RoleCtx {
    volatile uint32_t *abort_flag;
    DeviceState *dev;
};

// Bounded wait on an mbarrier phase.  Every polling warp takes issue slots from the warp that feeds the tensor
// core (one thread, whose scalar work between two MMAs is on the critical path), so waiters that can afford a
// few dozen nanoseconds of extra latency (loaders, epilogue) back off between polls; the MMA issuer does not.
// Only the self-test of the waits gives another `limit`.
template <int kBackoffNs = 0>
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, const RoleCtx &c, uint32_t limit = kSpinLimit)
{
    for (uint32_t i = 0; i < limit; ++i) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if (*c.abort_flag) return false;
        if (kBackoffNs > 0) __nanosleep(kBackoffNs);
    }
    *c.abort_flag = 1u;
    atomicOr(&c.dev->status, EOQ_DEV_TIMEOUT);
    return false;
}

// R(a / 2^7) with ties to even in four integer operations: adding 63 plus the parity of the quotient carries
// into bit 7 exactly when the remainder exceeds one half, or equals it with an odd quotient.
__device__ __forceinline__ int32_t rne7(int32_t a) { return (a + 63 + ((a >> 7) & 1)) >> 7; }

// The same rounding on the floating-point pipe, which the integer-heavy epilogue leaves idle.  For an integer t
// with kMagicBits + t inside [2^23, 2^24) the word kMagicBits + t read as a float is 1.5 * 2^23 + t exactly;
// one fused multiply-add forms 1.5 * 2^23 + t / 2^7, whose single rounding (nearest, ties to even, unit spacing
// in that binade) is R(t / 2^7).  Returns kMagicBits + R(t / 2^7): the low 16 bits are the two's-complement code.
constexpr uint32_t kMagicBits = 0x4B400000u;                     // 1.5 * 2^23 as a float
constexpr float kMagicRest = 12582912.0f - 12582912.0f / 128.0f;  // exact: 12484608
__device__ __forceinline__ uint32_t rne7_magic(uint32_t biased)
{
    return __float_as_uint(__fmaf_rn(__uint_as_float(biased), 0.0078125f, kMagicRest));
}

// R(x / 2^7) for an integer x in [0, 2^22) without a bias: x read as a float is the denormal x 2^-149, and one fused
// multiply-add forms x 2^-22 + 1.5 * 2^8, whose unit of rounding is 2^-15.  Returns kDenormalBits + R(x / 2^7).
constexpr uint32_t kDenormalBits = 0x43C00000u;   // 1.5 * 2^8 as a float
__device__ __forceinline__ uint32_t rne7_denormal(uint32_t x)
{
    return __float_as_uint(__fmaf_rn(__uint_as_float(x), __int_as_float((127 + 127) << 23), __uint_as_float(kDenormalBits)));
}

// Forward chain on 16 consecutive output channels of one pixel (Sec. 3.2.1: x2 = Q_a1(conv), x3 = gamma x2,
// x4 = x3 + b2 [+ shortcut], x5 = Q_a2(relu(x4)); mask = [x4 > 0]).
// The integer pipe (an instruction every two cycles and scheduler) is the busiest of this code, so clamps are moved in front of the
// roundings (both are monotonic, the clamp limits are chosen so that the rounded result is unchanged), roundings run as one
// FMA each, and the constant offsets of that trick are folded into the multiply-add that forms x4.  (The chain on floats
// alone, with conversions and saturating additions, has fewer instructions but a longer dependent sequence: 25.7 us where
// this takes 20.4 us for the 64-channel 56 x 56 layer at batch 64.)  No pipe is full: with shortcut and x2, 64 channels 56 x 56 at
// batch 512 take 133 us of which the integer pipe is busy 46% (9.4 of 26 instructions per element), the issue slots 63% and memory
// 3.6 TB/s; the largest stall is the wait for tensor memory and the shortcut.
//
// The b1 term (b1 times the sum of the weights whose taps fall inside the image, per border class and output
// channel) is read from shared memory, already multiplied by b1: the epilogue warps copy the table there once per
// kernel (kTableSmemBytes at most; larger tables are read from global memory and multiplied per use).
constexpr int kTableSmemBytes = 20 * 1024;

// One 256-bit store (sm_100): a whole 32-byte sector per lane instead of two half sectors.  ptr must be 32-byte aligned.
__device__ __forceinline__ void st_global_256(void *ptr, const uint32_t *v)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(ptr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                 "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// The three scalar codes of the forward chain as the epilogue uses them: the host values of the launch, or the
// values read from device memory when the caller keeps them there (they then change from one replay of a captured
// graph to the next without a new capture).
struct FwdScalars {
    int32_t b1, gamma, b2;
};

// Every epilogue thread calls this once per kernel.  Device-resident codes outside their range (16 bits each; b1
// also bounded by what keeps the accumulator inside int32) raise EOQ_DEV_RANGE and are clamped.
__device__ __forceinline__ FwdScalars load_fwd_scalars(const IgemmParams &p)
{
    FwdScalars s{p.b1_c, p.gamma_c, p.b2_c};
    if (p.scal_dev) {
        s.b1 = __ldg(p.scal_dev);
        s.gamma = __ldg(p.scal_dev + 1);
        s.b2 = __ldg(p.scal_dev + 2);
        // |acc| <= k_total * (127 + |b1|) * 127 must stay below 2^31 - 2^24
        const long long room = (2147483647ll - 16777216ll) / (127ll * (p.k_total > 0 ? p.k_total : 1)) - 127ll;
        const int32_t b1_lim = (int32_t)(room < 0 ? 0 : (room > 32767 ? 32767 : room));
        const bool bad = s.b1 < -b1_lim || s.b1 > b1_lim || s.gamma < -32768 || s.gamma > 32767 || s.b2 < -32768 ||
                         s.b2 > 32767 || (!p.b1_table && s.b1 != 0);
        if (bad) {
            if (blockIdx.x == 0 && (threadIdx.x & 31) == 0) atomicOr(&p.dev->status, EOQ_DEV_RANGE);
            s.b1 = p.b1_table ? clampi(s.b1, -b1_lim, b1_lim) : 0;
            s.gamma = clampi(s.gamma, -32768, 32767);
            s.b2 = clampi(s.b2, -32768, 32767);
        }
    }
    return s;
}

// Filled by the epilogue warps (`nthreads` of them, `tid` = index among them) before their first tile; they meet at
// named barrier 1 afterwards.  Returns the table's shared-memory address, or null when there is no table or it does
// not fit (uniform over the kernel).
__device__ __forceinline__ const int32_t *stage_b1_table(const IgemmParams &p, int32_t b1, uint8_t *smem_table, int tid, int nthreads)
{
    const int entries = p.b1_table ? p.b1_nrc * p.b1_ncc * p.N : 0;
    if (entries == 0 || entries * (int)sizeof(int32_t) > kTableSmemBytes) return nullptr;
    int32_t *ts = reinterpret_cast<int32_t *>(smem_table);
    for (int i = tid; i < entries; i += nthreads) ts[i] = b1 * __ldg(p.b1_table + i);
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
    return ts;
}

// The shift that brings a sum to exponent -14: 7, or what the exponent of an input behind the input quantizer asks for.
__device__ __forceinline__ int input_shift(const IgemmParams &p)
{
    if (!p.x_exp) return 7;
    const int shift = -__ldg(p.x_exp);
    if (shift <= 31 && shift >= -16) return shift;
    if (blockIdx.x == 0 && (threadIdx.x & 31) == 0) atomicOr(&p.dev->status, EOQ_DEV_RANGE);
    return max(-16, min(31, shift));
}

// The rounding of x2 = R(acc / 2^shift) for shifts 0 to 7 (7: an input at exponent -7; less behind the input quantizer).
// `unit`: gamma = 1, no shortcut, x2 not asked for: forward_unit_16, whose clamps are those of x5.
struct FwdShift {
    bool ok, unit;
    int32_t lo;           // -2^15 * 2^shift
    uint32_t hi;          // kMagicBits + 32767 * 2^shift + the part of a step that still rounds to 32767
    float scale, rest;    // 2^-shift; 1.5 * 2^23 (1 - 2^-shift), exact
};
__device__ __forceinline__ FwdShift forward_shift(const IgemmParams &p, const FwdScalars &fs, int shift)
{
    FwdShift f;
    f.ok = shift >= 0 && shift <= 7 && !p.acc_out;
    f.unit = f.ok && fs.gamma == 128 && !p.shortcut && !p.x2 && fs.b2 >= -16384 && fs.b2 <= 16384;
    const int s = clampi(shift, 0, 7);
    f.lo = f.unit ? ((p.relu ? 0 : -127) - fs.b2) * (1 << s) : -(32768 << s);
    f.hi = kMagicBits + (uint32_t)(f.unit ? (127 - fs.b2) * (1 << s) : (32767 << s) + (s ? (1 << (s - 1)) - 1 : 0));
    f.scale = __int_as_float((127 - s) << 23);
    f.rest = 12582912.0f - 12582912.0f * f.scale;
    return f;
}

__device__ __forceinline__ void store_x2(const IgemmParams &p, size_t off, const uint32_t (&h)[8])
{
    if ((reinterpret_cast<uintptr_t>(p.x2) & 31) == 0) {   // (uniform) the 16 codes of x2 are one 32-byte sector
        st_global_256(p.x2 + off, h);
    } else {
        int4 *d = reinterpret_cast<int4 *>(p.x2 + off);
        d[0] = make_int4((int)h[0], (int)h[1], (int)h[2], (int)h[3]);
        d[1] = make_int4((int)h[4], (int)h[5], (int)h[6], (int)h[7]);
    }
}

// `tb`: this pixel's 16 b1 terms in shared memory (already times b1), or null; then `tg` points at the 16 weight
// sums in global memory (or is null when the layer has no b1 term).
__device__ __forceinline__ void add_b1(int32_t (&a)[16], int32_t b1, const int32_t *tb, const int32_t *tg)
{
    if (tb) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int4 v = reinterpret_cast<const int4 *>(tb)[i];
            a[4 * i + 0] += v.x;
            a[4 * i + 1] += v.y;
            a[4 * i + 2] += v.z;
            a[4 * i + 3] += v.w;
        }
    } else if (tg) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int4 v = __ldg(reinterpret_cast<const int4 *>(tg) + i);
            a[4 * i + 0] += b1 * v.x;
            a[4 * i + 1] += b1 * v.y;
            a[4 * i + 2] += b1 * v.z;
            a[4 * i + 3] += b1 * v.w;
        }
    }
}

// `sc`: the 16 shortcut codes (zero without one).  `acc1` holds the tile's second partial sums when kTwo is set; kRelu = a
// ReLU follows.
template <bool kRelu, bool kTwo>
__device__ __forceinline__ void forward_16(const IgemmParams &p, const FwdScalars &fs, const FwdShift &sh, const uint32_t (&acc)[32],
                                           const uint32_t (&acc1)[32], size_t off, const int32_t *tb, const int32_t *tg, const int4 &sc)
{
    int32_t a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = (int32_t)acc[i];
    add_b1(a, fs.b1, tb, tg);
    // q = x2 code + kMagicBits, the code saturated to 16 bits: R(a / 2^shift) lies in [-32768, 32767] exactly when a lies
    // within half a step of those codes' multiples, and clamping a to [lo, hi - kMagicBits] first gives the same code.
    // |a| < 2^31 - 2^24 (checked on the host), so neither addition below wraps.  The lower clamp merges the second partial
    // sum (one add-max); the add of kMagicBits that follows is taken modulo 2^32, where max(A, lo) + kMagicBits is the true
    // (positive) sum for every A < 2^31 - 2^24.
    uint32_t q[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int32_t lo = kTwo ? __viaddmax_s32(a[i], (int32_t)acc1[i], sh.lo) : max(a[i], sh.lo);
        q[i] = __float_as_uint(__fmaf_rn(__uint_as_float(__viaddmin_u32((uint32_t)lo, kMagicBits, sh.hi)), sh.scale, sh.rest));
    }
    // x4 - 1 = gamma * x2 + (b2 + shortcut) * 2^7 - 1 = gamma * q + add, the bias of q folded into add (mod 2^32).
    // Forming x4 - 1 instead of x4 makes its sign bit [x4 <= 0], the complement of the mask bit, so the mask
    // costs one funnel shift per element; the + 1 rides on the add-min that clamps x4.
    const uint32_t g = (uint32_t)fs.gamma;
    const uint32_t base = ((uint32_t)fs.b2 << 7) - g * kMagicBits - 1u;
    uint32_t add[16];
    if (p.shortcut) {
        const uint32_t w[4] = {(uint32_t)sc.x, (uint32_t)sc.y, (uint32_t)sc.z, (uint32_t)sc.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) add[4 * i + k] = dot4_s8_u8(w[i], 128u << (8 * k), base);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) add[i] = base;
    }
    // Q_a2: R(x4 / 2^7) saturated to +-127 (and to 0 from below after a ReLU).  16319 / 128 = 127.49.. rounds to
    // 127 and everything above saturates to 127 too, so x4 is clamped to +-16319 before the rounding.
    uint32_t nbits = 0;  // bit i = [x4 <= 0] of channel i
    uint32_t r[16];
#pragma unroll
    for (int i = 15; i >= 0; --i) {
        const int32_t w = (int32_t)(g * q[i] + add[i]);  // x4 - 1
        nbits = __funnelshift_l((uint32_t)w, nbits, 1);
        if (kRelu) r[i] = rne7_denormal((uint32_t)__viaddmin_s32_relu(w, 1, 16319));
        else r[i] = rne7_magic((uint32_t)max(__viaddmin_s32(w, 1, 16319), -16319) + kMagicBits);
    }
    int4 o;
    if (kRelu) {
        // codes 0 to 127 above a constant: shifted and added on the multiply-add pipe, the constants taken off at the end
        constexpr uint32_t kRest = kDenormalBits * 0x01010101u;
        auto pack = [&](int i) { return (int)(((r[i + 3] * 256u + r[i + 2]) * 256u + r[i + 1]) * 256u + r[i] - kRest); };
        o = make_int4(pack(0), pack(4), pack(8), pack(12));
    } else {
        o.x = (int)__byte_perm(__byte_perm(r[0], r[1], 0x0040), __byte_perm(r[2], r[3], 0x0040), 0x5410);
        o.y = (int)__byte_perm(__byte_perm(r[4], r[5], 0x0040), __byte_perm(r[6], r[7], 0x0040), 0x5410);
        o.z = (int)__byte_perm(__byte_perm(r[8], r[9], 0x0040), __byte_perm(r[10], r[11], 0x0040), 0x5410);
        o.w = (int)__byte_perm(__byte_perm(r[12], r[13], 0x0040), __byte_perm(r[14], r[15], 0x0040), 0x5410);
    }
    *reinterpret_cast<int4 *>(p.x5 + off) = o;
    if (p.relu_mask) *reinterpret_cast<uint16_t *>(p.relu_mask + (off >> 3)) = (uint16_t)~nbits;
    if (p.x2) {
        uint32_t h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = __byte_perm(q[2 * i], q[2 * i + 1], 0x5410);
        store_x2(p, off, h);
    }
}

// The chain where gamma = 1 (unit A of a block, the first layer, projections) and x2 is not kept: x4 = x2 + b2 in whole codes, so
// Q_a2 rounds nothing and x5 = clamp(R(acc / 2^shift) + b2).  Both clamps move in front of the one rounding, where b2 shifts their
// limits (|b2| <= 2^14: the 16-bit saturation of x2 lies outside them), and mask = [x4 > 0] = [x5 > 0].  About 7 instructions per
// element, 3.5 of them on the integer pipe, the busiest of the general form (20 and 8.5): 64 channels 56 x 56,
// batch 64: 17.0 -> 15.7 us; 128 channels 28 x 28: 13.6 -> 12.3; 512 -> 256 channels 1 x 1, batch 32: 10.8 -> 9.9.
template <bool kRelu>
__device__ __forceinline__ void forward_unit_16(const IgemmParams &p, const FwdScalars &fs, const FwdShift &sh, const uint32_t (&acc)[32],
                                                const uint32_t (&acc1)[32], bool two, size_t off, const int32_t *tb, const int32_t *tg)
{
    int32_t a[16];
    if (two) {
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = (int32_t)(acc[i] + acc1[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = (int32_t)acc[i];
    }
    add_b1(a, fs.b1, tb, tg);
    uint32_t q[16];   // kMagicBits + x5 - b2
#pragma unroll
    for (int i = 0; i < 16; ++i)
        q[i] = __float_as_uint(__fmaf_rn(__uint_as_float(__viaddmin_u32((uint32_t)max(a[i], sh.lo), kMagicBits, sh.hi)), sh.scale, sh.rest));
    // four codes to a word on the multiply-add pipe; signed ones are made positive on the way
    const uint32_t rest = ((uint32_t)fs.b2 + (kRelu ? 0u : 128u) - kMagicBits) * 0x01010101u;
    uint32_t w[4], m[2] = {0u, 0u};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        w[k] = ((q[4 * k + 3] * 256u + q[4 * k + 2]) * 256u + q[4 * k + 1]) * 256u + q[4 * k] + rest;
        if (!kRelu) w[k] ^= 0x80808080u;
        const uint32_t positive = (((w[k] & 0x7f7f7f7fu) + 0x7f7f7f7fu) & ~w[k]) & 0x80808080u;
        m[k >> 1] = __dp4a(positive, (k & 1) ? 0x80402010u : 0x08040201u, m[k >> 1]);
    }
    *reinterpret_cast<int4 *>(p.x5 + off) = make_int4((int)w[0], (int)w[1], (int)w[2], (int)w[3]);
    if (p.relu_mask) *reinterpret_cast<uint16_t *>(p.relu_mask + (off >> 3)) = (uint16_t)((m[0] + m[1] * 256u) >> 7);
}

// The same for any shift, and with the accumulator dump; the partial sums are merged before.  |gamma x2| <= 2^30, so x4 fits
// 32 bits.
__device__ __forceinline__ void forward_any_16(const IgemmParams &p, const FwdScalars &fs, const uint32_t (&acc)[32], size_t off,
                                               const int32_t *tb, const int32_t *tg, const int4 &sc, int shift)
{
    int32_t a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = (int32_t)acc[i];
    add_b1(a, fs.b1, tb, tg);
    if (p.acc_out) {
        int4 *d = reinterpret_cast<int4 *>(p.acc_out + off);
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = make_int4(a[4 * i], a[4 * i + 1], a[4 * i + 2], a[4 * i + 3]);
    }
    const uint32_t w[4] = {(uint32_t)sc.x, (uint32_t)sc.y, (uint32_t)sc.z, (uint32_t)sc.w};
    const int32_t x5_lo = p.relu ? 0 : -127;
    uint32_t mask = 0, h[8] = {}, o[4] = {};
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        int32_t q;
        if (shift >= 0) {
            q = clampi(rne_shr32(a[i], shift), -32768, 32767);
        } else {
            const long long l = (long long)a[i] << (-shift);
            q = (int32_t)(l < -32768 ? -32768 : (l > 32767 ? 32767 : l));
        }
        const int32_t x4 = fs.gamma * q + (fs.b2 + ((int32_t)(w[i >> 2] << (24 - 8 * (i & 3))) >> 24)) * 128;
        mask |= (x4 > 0 ? 1u : 0u) << i;
        h[i >> 1] |= ((uint32_t)q & 0xffffu) << (16 * (i & 1));
        o[i >> 2] |= ((uint32_t)clampi(rne7(clampi(x4, -16319, 16319)), x5_lo, 127) & 0xffu) << (8 * (i & 3));
    }
    *reinterpret_cast<int4 *>(p.x5 + off) = make_int4((int)o[0], (int)o[1], (int)o[2], (int)o[3]);
    if (p.relu_mask) *reinterpret_cast<uint16_t *>(p.relu_mask + (off >> 3)) = (uint16_t)mask;
    if (p.x2) store_x2(p, off, h);
}

// One 16-channel group of the forward epilogue: the partial sums of the tile (r2 counts when nacc == 2).
__device__ __forceinline__ void forward_group(const IgemmParams &p, const FwdScalars &fs, const FwdShift &sh, uint32_t (&r)[32],
                                              uint32_t (&r2)[32], uint32_t nacc, size_t off, const int32_t *tb, const int32_t *tg,
                                              const int4 &sc, int shift)
{
    if (sh.unit) {
        if (p.relu) forward_unit_16<true>(p, fs, sh, r, r2, nacc == 2, off, tb, tg);
        else forward_unit_16<false>(p, fs, sh, r, r2, nacc == 2, off, tb, tg);
    } else if (sh.ok) {
        if (nacc == 2) {
            if (p.relu) forward_16<true, true>(p, fs, sh, r, r2, off, tb, tg, sc);
            else forward_16<false, true>(p, fs, sh, r, r2, off, tb, tg, sc);
        } else {
            if (p.relu) forward_16<true, false>(p, fs, sh, r, r2, off, tb, tg, sc);
            else forward_16<false, false>(p, fs, sh, r, r2, off, tb, tg, sc);
        }
    } else {
        if (nacc == 2) {
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] += r2[i];
        }
        forward_any_16(p, fs, r, off, tb, tg, sc, shift);
    }
}

// Error back-propagation: keep the exact sums (the scale quantizer needs the maximum over the whole tensor before any element can
// be coded) and track max |.|.  They are kept as 16-bit words that lose nothing Q_e can see (sums_pack_16), one 32-byte sector per
// lane and 16 columns: this launch is bound by its stores.  A caller who asks for the int32 sums gets those instead
// (p.sums16 == null), two 32-byte sectors at a time where the buffer allows it: with four 16-byte stores of half a sector each, 64
// channels 56 x 56 take 163 us instead of 103 at batch 512 (79 as words), 22.0 instead of 16.7 at batch 64.
__device__ __forceinline__ uint32_t dgrad_16(const IgemmParams &p, const uint32_t *acc, size_t off, uint32_t &mx_masked)
{
    uint32_t mx = 0;
    // the consumer's error head needs the maximum over the positions its ReLU lets through as well (off is the element
    // index of the error tensor and a multiple of 16: one 16-bit word of mask bits)
    const uint32_t bits = p.next_mask ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(p.next_mask) + (off >> 4)) : 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a0 = (uint32_t)abs((int)acc[4 * i]), a1 = (uint32_t)abs((int)acc[4 * i + 1]);
        const uint32_t a2 = (uint32_t)abs((int)acc[4 * i + 2]), a3 = (uint32_t)abs((int)acc[4 * i + 3]);
        mx = max(max(mx, a0), max(a1, max(a2, a3)));
        if (bits) {
            const uint32_t b4 = bits >> (4 * i);
            mx_masked = max(mx_masked, (b4 & 1u) ? a0 : 0u);
            mx_masked = max(mx_masked, (b4 & 2u) ? a1 : 0u);
            mx_masked = max(mx_masked, (b4 & 4u) ? a2 : 0u);
            mx_masked = max(mx_masked, (b4 & 8u) ? a3 : 0u);
        }
    }
    if (p.sums16) {
        uint32_t w[8];
        sums_pack_16(acc, mx, w);
        st_global_256(p.sums16 + off, w);   // (a workspace: aligned to 256 bytes)
    } else if ((reinterpret_cast<uintptr_t>(p.acc_out) & 31) == 0) {   // (off is a multiple of 16: one answer for a launch)
        st_global_256(p.acc_out + off, acc);
        st_global_256(p.acc_out + off + 8, acc + 8);
    } else {
        int4 *d = reinterpret_cast<int4 *>(p.acc_out + off);
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = make_int4((int)acc[4 * i], (int)acc[4 * i + 1], (int)acc[4 * i + 2], (int)acc[4 * i + 3]);
    }
    return mx;
}

}  // namespace eoq
