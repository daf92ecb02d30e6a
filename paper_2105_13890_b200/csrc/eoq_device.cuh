// Device-side helpers: integer rounding of the EOQ quantizers and thin wrappers over sm_100a PTX.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "eoq_internal.h"

namespace eoq {

// ------------------------------------------------------------------ integer rounding (Sec. 3.2.2)

// R(a / 2^s), nearest with ties to even, for s in [0, 31].
__device__ __forceinline__ int32_t rne_shr32(int32_t a, int s)
{
    if (s == 0) return a;
    int32_t q = a >> s;
    uint32_t r = (uint32_t)a & ((1u << s) - 1u);
    uint32_t h = 1u << (s - 1);
    return q + (int32_t)((r > h) || (r == h && (q & 1)));
}

// R(a / 2^s) for 64-bit a and s in [0, 62].
__device__ __forceinline__ long long rne_shr64(long long a, int s)
{
    if (s == 0) return a;
    long long q = a >> s;
    unsigned long long r = (unsigned long long)a & ((1ull << s) - 1ull);
    unsigned long long h = 1ull << (s - 1);
    return q + (long long)((r > h) || (r == h && (q & 1)));
}

__device__ __forceinline__ int32_t clampi(int32_t v, int32_t lo, int32_t hi) { return min(max(v, lo), hi); }

// Four int32 values saturated to int8 and packed into one word, c0 in the lowest byte: two instructions.
__device__ __forceinline__ uint32_t pack4_sat(int c0, int c1, int c2, int c3)
{
    uint32_t hi, r;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"(c3), "r"(c2), "r"(0));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(c1), "r"(c0), "r"(hi));
    return r;
}

// the same of values whose low bytes are the codes already
__device__ __forceinline__ uint32_t pack4(int a, int b, int c, int d)
{
    return (uint32_t)(a & 0xff) | ((uint32_t)(b & 0xff) << 8) | ((uint32_t)(c & 0xff) << 16) | ((uint32_t)(d & 0xff) << 24);
}

// byte k of w, sign-extended
template <int k>
__device__ __forceinline__ int32_t sbyte(uint32_t w)
{
    // prmt selector digit 8 + k replicates the sign bit of byte k (the __byte_perm intrinsic drops that bit)
    uint32_t r;
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(r) : "r"(w), "n"(((8 + k) << 12) | ((8 + k) << 8) | ((8 + k) << 4) | k));
    return (int32_t)r;
}

// sum of the products of four signed bytes with four unsigned ones, plus c: with one byte of b set to 128 it scales and adds
// one code without the byte extraction, which would go to the busier pipe
__device__ __forceinline__ uint32_t dot4_s8_u8(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("dp4a.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// R(log2 M) for M >= 1: floor(log2 M) plus one when M^2 >= 2^(2f+1).
__device__ __forceinline__ int round_log2_u32(uint32_t M)
{
    int f = 31 - __clz(M);
    unsigned long long sq = (unsigned long long)M * M;
    return f + (sq >= (1ull << (2 * f + 1)) ? 1 : 0);
}

// ... of a positive finite float given by its bit pattern
__device__ __forceinline__ int round_log2_f32bits(uint32_t bits)
{
    const int eb = (int)((bits >> 23) & 0xffu);
    const uint32_t frac = bits & 0x7fffffu;
    if (eb == 0) return round_log2_u32(frac) - 149;  // subnormal: frac * 2^-149
    const unsigned long long m = (1ull << 23) | frac;  // M = m * 2^(eb - 150), m in [2^23, 2^24)
    return (eb - 127) + ((m * m >= (1ull << 47)) ? 1 : 0);
}

__device__ __forceinline__ int round_log2_u64(unsigned long long M)
{
    if (M < (1ull << 32)) return round_log2_u32((uint32_t)M);
    int f = 63 - __clzll(M);
    unsigned long long hi = __umul64hi(M, M);  // M^2 >= 2^(2f+1) with 2f+1 >= 65
    return f + (hi >= (1ull << (2 * f + 1 - 64)) ? 1 : 0);
}

// ------------------------------------------------------------------ stochastic rounding (an extension, not in the paper)

// SplitMix64 output function (Steele, Lea, Flood 2014) as a counter hash.
__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
constexpr unsigned long long kGolden = 0x9E3779B97F4A7C15ull;
// The bits of one element: a hash of (seed, step, tensor), then of the element's index.
__device__ __forceinline__ unsigned long long rounding_key(unsigned long long seed, unsigned long long step, unsigned long long tensor)
{
    return mix64(mix64(seed + kGolden * (step + 1)) + kGolden * (tensor + 1));
}
__device__ __forceinline__ unsigned long long rounding_bits(unsigned long long key, unsigned long long element)
{
    return mix64(key + kGolden * (element + 1));
}

// Code of SQ for an integer a once t = R(log2 max) is known: sat(R(a * 2^(7-t)), -127, 127).
__device__ __forceinline__ int32_t sq_code32(int32_t a, int t)
{
    int s = t - 7;
    int32_t v = s >= 0 ? rne_shr32(a, s) : a * (1 << (-s));  // s < 0 only when |a| < 2^7.5
    return clampi(v, -127, 127);
}

// The same code for a shift s = t - 7 >= 1 known to the whole kernel, in four integer operations before the
// clamp: adding 2^(s-1) - 1 plus the parity of the quotient carries into bit s exactly when the remainder exceeds
// one half, or equals it with an odd quotient.  `half_m1` = 2^(s-1) - 1.  Needs |a| + 2^(s-1) < 2^31, which holds
// because 2^(s-1) <= max|a| / 2^7.
__device__ __forceinline__ int32_t sq_code32_shr(int32_t a, int s, int32_t half_m1)
{
    return clampi((a + half_m1 + ((a >> s) & 1)) >> s, -127, 127);
}

// Four such codes in a word: the lower clamp rides on the addition (`lo` = -127 * 2^s), the pack saturates at 127.
__device__ __forceinline__ uint32_t sq_pack4_shr(const int32_t *a, int s, int32_t half_m1, int32_t lo)
{
    int32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = (__viaddmax_s32(a[k], half_m1, lo) + ((a[k] >> s) & 1)) >> s;
    return pack4_sat(v[0], v[1], v[2], v[3]);
}

// ------------------------------------------------------------------ sums on their way to Q_e
// The sums of an error back-propagation travel from its GEMM to the kernel that codes them as 16-bit words: 16 consecutive
// channels of a pixel are 32 bytes instead of 64.  Nothing that Q_e can see is lost.  Sums below 2^14 stand as they are; in a
// group with a larger one, all 16 lose their low s bits (s = bits of the largest - 14) and what was cut off is or-ed into the
// lowest bit that stays.  Q_e rounds at bit S = R(log2 max) - 7 of the tensor's maximum, and a group's largest |sum| is at most
// that maximum, so S >= s + 6: the bit Q_e rounds at and all above it are kept, and the or-ed bit tells a remainder of exactly
// one half from one beside it.  Either way a word has 15 significant bits, so bit 15 repeats bit 14, and that is where a group
// with s > 0 is marked (word 0) and carries s (words 1 to 5): bits flipped, no space beside the sums.

// `mx` = the largest magnitude among the 16 sums
__device__ __forceinline__ void sums_pack_16(const uint32_t *acc, uint32_t mx, uint32_t (&w)[8])
{
    if (mx < (1u << 14)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = __byte_perm(acc[2 * i], acc[2 * i + 1], 0x5410);
        return;
    }
    const int s = 18 - __clz(mx);
    const uint32_t rest = (1u << s) - 1u;
    auto cut = [&](uint32_t v) { return (uint32_t)((int32_t)(v | ((v & rest) + rest)) >> s); };   // (the sum carries into bit s if any bit is lost)
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = __byte_perm(cut(acc[2 * i]), cut(acc[2 * i + 1]), 0x5410);
    w[0] ^= 0x8000u | (uint32_t)(s & 1) << 31;
    w[1] ^= (uint32_t)(s & 2) << 14 | (uint32_t)(s & 4) << 29;
    w[2] ^= (uint32_t)(s & 8) << 12 | (uint32_t)(s & 16) << 27;
}

// Was the group shortened?
__device__ __forceinline__ bool sums_shortened(uint32_t w0) { return ((w0 ^ (w0 << 1)) & 0x8000u) != 0; }

// s of a shortened group; its marked words get their bit 15 back.
__device__ __forceinline__ int sums_unmark(uint32_t (&w)[8])
{
    const uint32_t d0 = w[0] ^ (w[0] << 1), d1 = w[1] ^ (w[1] << 1), d2 = w[2] ^ (w[2] << 1);
#pragma unroll
    for (int i = 0; i < 3; ++i) w[i] = (w[i] & 0x7fff7fffu) | ((w[i] << 1) & 0x80008000u);
    return (int)((d0 >> 31) | (d1 >> 14 & 2u) | (d1 >> 29 & 4u) | (d2 >> 12 & 8u) | (d2 >> 27 & 16u));
}

// Codes of SQ for 16 sums under a shift known to the whole kernel (t = R(log2 max)), on the floating-point pipe: 2^23 + (word +
// 2^15) is a float whose bits are put together from the word, and one fused multiply-add forms 1.5 * 2^23 + word / 2^n, rounded to
// nearest even at unit spacing.  n = t - 7, less s in a shortened group.  Every constant is exact for -7 <= n <= 15; a larger n
// leaves only zeros, as 15 does (-2^14 / 2^15 is a tie and goes to 0).
__device__ __forceinline__ void sum_codes_16(int t, uint32_t (&w)[8], uint32_t (&cw)[4])
{
    int n = t - 7;
    if (sums_shortened(w[0])) n -= sums_unmark(w);
    const float scale = __int_as_float((127 - min(n, 15)) << 23), rest = 12582912.0f - 8421376.0f * scale;
    auto code = [&](uint32_t u, uint32_t sel) {
        const float f = __fmaf_rn(__uint_as_float(__byte_perm(u, 0x4B00u, sel)), scale, rest);
        return __viaddmax_s32((int32_t)__float_as_uint(f), -0x4B400000, -127);
    };
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t u0 = w[2 * q] ^ 0x80008000u, u1 = w[2 * q + 1] ^ 0x80008000u;
        cw[q] = pack4_sat(code(u0, 0x5410), code(u0, 0x5432), code(u1, 0x5410), code(u1, 0x5432));
    }
}

// Expands 4 mask bits into 4 byte masks (0x00 / 0xff).
__device__ __forceinline__ uint32_t bits_to_bytes(uint32_t nibble)
{
    return (((nibble & 0xfu) * 0x00204081u) & 0x01010101u) * 0xffu;
}

// sum of the 16 products of the codes in e with 16-bit values at x (32 bytes): below 2^26
__device__ __forceinline__ int dot16_s8_s16(const uint32_t (&e)[4], const int4 *x)
{
    const int4 lo = __ldg(x), hi = __ldg(x + 1);
    int s = __dp2a_lo(lo.x, (int)e[0], 0);
    s = __dp2a_hi(lo.y, (int)e[0], s);
    s = __dp2a_lo(lo.z, (int)e[1], s);
    s = __dp2a_hi(lo.w, (int)e[1], s);
    s = __dp2a_lo(hi.x, (int)e[2], s);
    s = __dp2a_hi(hi.y, (int)e[2], s);
    s = __dp2a_lo(hi.z, (int)e[3], s);
    return __dp2a_hi(hi.w, (int)e[3], s);
}

__device__ __forceinline__ int32_t sq_code64(long long a, int t)
{
    int s = t - 7;
    long long v = s >= 0 ? rne_shr64(a, s) : a * (1ll << (-s));
    return (int32_t)(v < -127 ? -127 : (v > 127 ? 127 : v));
}

// ------------------------------------------------------------------ border classes of the b1 term
// x1 = x0 + b1 has a zero halo, so conv(x1) = conv(x0) + b1 * (sum of the weights of the taps that fall
// inside the image).  Which taps are inside depends only on how far the output row (column) is from the
// image border: rows whose window sticks out at the top (y < nlo) or at the bottom (y >= extent - nhi) get a
// class each, all interior rows share class nlo.  When the image is so small that no interior row exists
// (ncls == extent) every row is its own class.

__device__ __forceinline__ int border_class(int y, int extent, int nlo, int nhi, int ncls)
{
    if (ncls == extent) return y;
    if (y < nlo) return y;
    if (y >= extent - nhi) return nlo + 1 + (y - (extent - nhi));
    return nlo;
}

// Is filter tap k inside the image for the rows of class `cls`?
__device__ __forceinline__ bool tap_valid(int cls, int k, int extent_out, int extent_in, int nlo, int nhi, int ncls,
                                          int stride, int pad)
{
    int y;
    if (ncls == extent_out) y = cls;
    else if (cls < nlo) y = cls;
    else if (cls == nlo) y = nlo;
    else y = extent_out - nhi + (cls - nlo - 1);
    const int src = y * stride - pad + k;
    return src >= 0 && src < extent_in;
}

// ------------------------------------------------------------------ warp reductions

__device__ __forceinline__ uint32_t warp_max_u32(uint32_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ long long warp_sum_i64(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide reductions (every thread of the block must call; the result is valid in thread 0).  Thousands of
// warps hitting one global cell with an atomic serialise at the L2, so each block sends one.
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v)   // the upper words decide, then the lower ones
{
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
    return (unsigned long long)hi << 32 | lo;
}
__device__ __forceinline__ unsigned long long block_max_u64(unsigned long long v)
{
    __shared__ unsigned long long red_max[32];
    v = warp_max_u64(v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    if (lane == 0) red_max[warp] = v;
    __syncthreads();
    if (warp == 0) v = warp_max_u64(lane < nw ? red_max[lane] : 0ull);
    __syncthreads();
    return v;
}

// The 32-bit forms use the warp-wide reduction instructions (one instead of five shuffle steps).
__device__ __forceinline__ uint32_t block_max_u32(uint32_t v)
{
    __shared__ uint32_t red_max32[32];
    v = __reduce_max_sync(0xffffffffu, v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    if (lane == 0) red_max32[warp] = v;
    __syncthreads();
    if (warp == 0) v = __reduce_max_sync(0xffffffffu, lane < nw ? red_max32[lane] : 0u);
    return v;  // (a second call in the same kernel must be separated from this one by a barrier)
}

__device__ __forceinline__ long long block_sum_i64(long long v)
{
    __shared__ long long red_sum[32];
    v = warp_sum_i64(v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    if (lane == 0) red_sum[warp] = v;
    __syncthreads();
    if (warp == 0) v = warp_sum_i64(lane < nw ? red_sum[lane] : 0ll);
    __syncthreads();
    return v;
}

// kN sums over the block behind one barrier, valid in thread 0 (and once per kernel: the cells are not free again)
template <int kN>
__device__ __forceinline__ void block_sums_i64(long long (&v)[kN])
{
    __shared__ long long red_sums[kN][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int i = 0; i < kN; ++i) {
        v[i] = warp_sum_i64(v[i]);
        if (lane == 0) red_sums[i][warp] = v[i];
    }
    __syncthreads();
    if (warp == 0)
#pragma unroll
        for (int i = 0; i < kN; ++i) v[i] = warp_sum_i64(lane < nw ? red_sums[i][lane] : 0ll);
}

// ------------------------------------------------------------------ PTX: shared-memory barriers and TMA

namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Chained launches (see launch_chained): the work of the kernels in front on the stream is complete and visible behind the
// wait; the next kernel may be brought up once every block has called grid_dep_launch or ended.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// A line that the thread will read behind a barrier: its latency runs beside that of the values the barrier waits for.
__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// Thread-block clusters: a barrier over all their threads (the writes in front of it, to shared memory of any of the blocks,
// are visible behind it), the address of a shared-memory location in another block, and a 16-byte store there.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t smem, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster_128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void st_cluster_32(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ int4 ld_shared_128(uint32_t addr)
{
    int4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

// At the start of a kernel of many small blocks: a grid of at most one block per SM leaves room for its successor at once,
// a larger one brings it up with its last blocks (or where it calls grid_dep_launch).  Brought up beside a full device, the
// successor only keeps kernels of other streams away: ResNet-18 steps took 648 us at batch 1 without, 610 with it; 1697 us
// at batch 64 without, 1730 with it in grids of any size.  (The limit is that of the whole part; on a slice of it kernels come
// up in another order, with the same results.)
__device__ __forceinline__ void grid_dep_wait_launch_small()
{
    grid_dep_wait();
    if (gridDim.x * gridDim.y <= kPartSms) grid_dep_launch();
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// the same without giving the thread up to the scheduler for a while
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Tiled TMA loads (global -> shared), completion counted in bytes on an mbarrier.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void *map, uint32_t bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void *map, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void *map, uint32_t bar, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// im2col-mode TMA load on a rank-4 (C, W, H, N) tensor: coordinates of the first pixel plus the
// filter-tap offsets (w, h).
__device__ __forceinline__ void tma_load_im2col_4d(uint32_t dst, const void *map, uint32_t bar, int c, int w, int h,
                                                   int n, uint16_t off_w, uint16_t off_h)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(off_w), "h"(off_h)
        : "memory");
}
__device__ __forceinline__ void prefetch_tensormap(const void *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// ------------------------------------------------------------------ PTX: tensor memory and tcgen05

__device__ __forceinline__ void tmem_alloc(uint32_t smem_result, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// The warp that feeds the tensor core runs its whole loop with all 32 lanes (so that every address and
// descriptor it computes is the same in all lanes and can live in the uniform datapath, which is where the MMA
// instruction takes its operands from) and only the instructions that must come from a single thread are
// predicated on one elected lane.  Issued from inside a one-lane branch instead, every operand has to be moved
// from a vector to a uniform register per MMA, which costs more cycles than a narrow MMA takes.

// 1 in exactly one lane of the (fully active) warp, 0 in the others.
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t leader;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(leader));
    return leader;
}

// Index of the calling warp in its block, in a form the compiler knows to be the same in all lanes.
__device__ __forceinline__ int warp_index_uniform() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

// D[tmem] (+)= A[smem desc] * B[smem desc], int8 x int8 -> int32, issued by the lane whose `leader` is non-zero.
// (No memory clobber: the issuing warp's scalar work between two MMAs is what limits narrow tiles, so the
// compiler must be free to keep loop state in registers.  Ordering against barrier waits and commits comes from
// those being volatile asm statements with memory clobbers.)
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate, uint32_t leader)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader));
}

// The mbarrier receives one arrival when every MMA issued so far by the leader lane has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar, uint32_t leader)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        ::"r"(bar), "r"(leader) : "memory");
}

// 32 lanes x 32 columns of 32-bit accumulators: thread t of the warp receives lane (base lane + t).
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

}  // namespace ptx

using ptx::elect_one;
using ptx::warp_index_uniform;

// 64-bit shared-memory matrix descriptor of tcgen05.mma (start address, leading and stride byte offsets
// in 16-byte units, descriptor version 1 at bit 46, swizzle mode at bits 61..63).
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes,
                                                   uint32_t layout_type)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46) | ((uint64_t)layout_type << 61);
}

// The same descriptor split in two 32-bit halves, so that an issue loop only adds byte offsets (in 16-byte
// units) to the low half: low = start address >> 4 | (leading offset >> 4) << 16, high = (stride offset >> 4) |
// version bit | swizzle mode.  Building the whole descriptor per MMA costs more cycles than a narrow MMA takes.
__device__ __forceinline__ uint32_t smem_desc_hi(uint32_t sbo_bytes, uint32_t layout_type)
{
    return ((sbo_bytes >> 4) & 0x3FFFu) | (1u << 14) | (layout_type << 29);
}
__device__ __forceinline__ uint64_t smem_desc_join(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }

// The warp that feeds the tensor core is a single in-order instruction stream: about 25 scalar instructions
// per MMA cost ~130 cycles, while a 128 x 64 x 32 MMA takes 52.  The issue helpers below are therefore fully
// unrolled with compile-time MMA indices, so that an MMA costs a handful of integer adds.
//
// Successive MMAs of a tile alternate between two partial accumulators d0 / d1 when the tile has them (an MMA
// that accumulates into the columns its predecessor is still writing waits ~97 cycles; two interleaved chains
// run at 52 cycles for 64 columns, 69 for 128).  `fresh` is 1 for the first MMAs of a tile, which overwrite.

// kSteps 32-byte K steps of one (A sub-tile, B sub-tile) pair; `parity` = index of the first MMA modulo 2.
// The B operand has its own descriptor half `b_hi` and its own K step `b_k16` (16-byte units): 2 for a K-major
// tile (32 bytes along the row), 2 * row bytes for an MN-major one (32 rows further).
template <int kSteps>
__device__ __forceinline__ void mma_k_steps(uint32_t d0, uint32_t d1, uint32_t a_lo, uint32_t b_lo, uint32_t hi,
                                            uint32_t idesc, uint32_t parity, uint32_t fresh0, uint32_t fresh1,
                                            uint32_t leader, uint32_t b_hi, uint32_t b_k16)
{
#pragma unroll
    for (int kk = 0; kk < kSteps; ++kk) {
        const bool odd = ((kk & 1) != 0) != (parity != 0);
        // the first MMA into each accumulator overwrites it
        uint32_t acc = 1u;
        if (kk < 2) acc = (odd ? fresh1 : fresh0) ? 0u : 1u;
        ptx::mma_i8(odd ? d1 : d0, smem_desc_join(a_lo + 2 * kk, hi), smem_desc_join(b_lo + kk * b_k16, b_hi), idesc, acc, leader);
    }
}

// All kDim x kDim taps of one channel chunk against resident weights: tap (a, b) reads the patch tile
// (a * row16 + b * kc16) further (16-byte units); its weights are the next sub-tile.
template <int kDim, int kSteps>
__device__ __forceinline__ void mma_patch_chunk(uint32_t d0, uint32_t d1, uint32_t a_lo, uint32_t b_lo, uint32_t row16,
                                                uint32_t kc16, uint32_t b_sub16, uint32_t hi, uint32_t idesc,
                                                bool first_chunk, bool two_acc, uint32_t leader, uint32_t b_hi,
                                                uint32_t b_k16)
{
#pragma unroll
    for (int a = 0; a < kDim; ++a)
#pragma unroll
        for (int b = 0; b < kDim; ++b)
#pragma unroll
            for (int kk = 0; kk < kSteps; ++kk) {
                const int idx = (a * kDim + b) * kSteps + kk;
                uint32_t acc = 1u;
                if (idx == 0) acc = first_chunk ? 0u : 1u;
                if (idx == 1) acc = (first_chunk && two_acc) ? 0u : 1u;
                ptx::mma_i8((idx & 1) ? d1 : d0, smem_desc_join(a_lo + a * row16 + b * kc16 + 2 * kk, hi),
                            smem_desc_join(b_lo + (a * kDim + b) * b_sub16 + kk * b_k16, b_hi), idesc, acc, leader);
            }
}
// Swizzle field of the descriptor for a sub-tile whose rows are `row_bytes` wide.
__device__ __forceinline__ uint32_t layout_type_for(int row_bytes)
{
    return row_bytes == 128 ? 2u : (row_bytes == 64 ? 4u : (row_bytes == 32 ? 6u : 0u));
}

// 32-bit instruction descriptor of tcgen05.mma kind::i8: signed 8-bit A and B, int32 accumulator, M x N.
__device__ __forceinline__ uint32_t make_idesc_i8(int m, int n, bool a_mn_major, bool b_mn_major)
{
    return (2u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

}  // namespace eoq
