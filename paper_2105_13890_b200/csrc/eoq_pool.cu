// Max-pooling of int8 codes and its backward pass with Q_e (arXiv 2105.13890, Sec. 3.2.1 chains the units of the network;
// the ImageNet networks pool behind their first layer).
#include "eoq_cells.cuh"
#include "eoq_device.cuh"
#include "eoq_internal.h"
#include "eoq_next_head.cuh"

namespace eoq {

namespace {

constexpr int kThreads = 256;

template <int kSel>
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b)
{
    uint32_t r;  // (the intrinsic __byte_perm drops the sign-replication bit of the selector digits)
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "n"(kSel));
    return r;
}

// One thread per 16 channels of an output pixel.  arg = kh * k + kw of the first maximum in scan order.  A candidate is the
// 16-bit key (code << 8) | (255 - position): the larger key is the larger code or, among equals, the earlier position, so a
// tap costs one permute and one packed maximum per two channels.  Bound by memory then (each input is read through the L1
// by the windows that cover it); with a 32-bit compare and two selects per channel and tap the 51 M codes of the
// 112 x 112 maps at batch 64 took 41 us, now 16.5 us.  kK: the window size when it is known (all loads of a thread in flight), else 0.
template <int kK>
__global__ void __launch_bounds__(kThreads)
maxpool_fwd_kernel(const int8_t *__restrict__ x, uint32_t items, int h, int w, int c, int k_rt, int s, int p, int ho, int wo,
                   int8_t *__restrict__ y, uint8_t *__restrict__ arg)
{
    ptx::grid_dep_wait_launch_small();
    const int groups = c / 16, k = kK ? kK : k_rt;
    const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= items) return;
    const uint32_t pix = i / (uint32_t)groups, row = pix / (uint32_t)wo;
    const int g = (int)(i - pix * (uint32_t)groups), ox = (int)(pix - row * (uint32_t)wo);
    const int b = (int)(row / (uint32_t)ho), oy = (int)(row - (uint32_t)b * (uint32_t)ho);
    uint32_t even[4], odd[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) even[q] = odd[q] = 0x80008000u;
    auto take = [&](const int4 &v, int pos) {
        const uint32_t at = 255u - (uint32_t)pos;
        const uint32_t word[4] = {(uint32_t)v.x, (uint32_t)v.y, (uint32_t)v.z, (uint32_t)v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            even[q] = __vmaxs2(even[q], prmt<0x2404>(word[q], at));
            odd[q] = __vmaxs2(odd[q], prmt<0x3414>(word[q], at));
        }
    };
    const int iy0 = oy * s - p, ix0 = ox * s - p;
    const int8_t *src = x + (((long long)b * h + iy0) * w + ix0) * c + g * 16;
    if (kK) {
        int4 v[kK ? kK * kK : 1];
        bool in[kK ? kK * kK : 1];
#pragma unroll
        for (int u = 0; u < kK * kK; ++u) {
            const int dy = u / (kK ? kK : 1), dx = u % (kK ? kK : 1);
            in[u] = (unsigned)(iy0 + dy) < (unsigned)h && (unsigned)(ix0 + dx) < (unsigned)w;
            v[u] = in[u] ? __ldg(reinterpret_cast<const int4 *>(src + (dy * w + dx) * (long long)c)) : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < kK * kK; ++u)
            if (in[u]) take(v[u], u);
    } else {
        for (int dy = 0; dy < k; ++dy)
            for (int dx = 0; dx < k; ++dx)
                if ((unsigned)(iy0 + dy) < (unsigned)h && (unsigned)(ix0 + dx) < (unsigned)w)
                    take(__ldg(reinterpret_cast<const int4 *>(src + (dy * w + dx) * (long long)c)), dy * k + dx);
    }
    uint32_t yo[4], ao[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        yo[q] = prmt<0x7351>(even[q], odd[q]);
        ao[q] = ~prmt<0x6240>(even[q], odd[q]);
    }
    reinterpret_cast<uint4 *>(y)[i] = make_uint4(yo[0], yo[1], yo[2], yo[3]);
    reinterpret_cast<uint4 *>(arg)[i] = make_uint4(ao[0], ao[1], ao[2], ao[3]);
}

// Backward: every output error code is added at the input position its window elected; the exact sums are then
// coded with Q_e, which needs their maximum over the whole tensor first.  So the kernel runs twice: pass 0 reduces
// max |sum| into the handle's cell, pass 1 forms the sums again and codes them (no intermediate tensor is written).
// One thread per 16 channels of an input position gathers from the windows that cover it (at most
// ceil(k / stride)^2): a window's 16 codes count where its recorded position equals this one.  Four codes are
// handled per 32-bit word: bytes are compared at once, the chosen codes are kept with an offset of 128 (others as
// 128 itself) so that they add as unsigned halves of two words without carries between them.
//
// kNext: the consumer's error head rides along (the layer in front of the pool: e1 = e_in * [x4 > 0],
// e3 = Q_e(gamma * e1), sum of e1).  Coding is monotonic in |sum|, so max |e1| is the code of the largest masked
// |sum|: pass 0 reduces that second maximum as well (into the 64-bit cell), and pass 1 knows both scales, writes
// e_in (optional) and e3 and adds up e1 - the two kernels of a separate error head and their pass over e_in are gone.
template <int kPass, bool kNext>
__global__ void __launch_bounds__(kThreads)
maxpool_bwd_kernel(const int8_t *__restrict__ e, const int32_t *e_exp, const uint8_t *__restrict__ arg, int n, int h, int w, int c,
                   int k, int s, int p, int ho, int wo, int8_t *__restrict__ e_in, int32_t *e_in_exp,
                   const uint8_t *__restrict__ next_mask, const int32_t *next_gamma, int8_t *__restrict__ e3, int32_t *e3_exp,
                   long long *sum_e1, DeviceState *dev)
{
    const int groups = c / 16;
    const uint32_t items = (uint32_t)n * h * w * groups;   // below 2^31 (checked by the caller), so i + stride cannot wrap
    int t = 7;
    NextHead nh = {};
    if (kPass == 1) {
        const uint32_t M = dev->absmax_u32;
        t = M ? round_log2_u32(M) : 7;
        const int p_in = *e_exp;
        const int p0 = M ? p_in + t - 7 : p_in;
        if (kNext) nh = next_head_setup(next_gamma, (uint32_t)abs(sq_code32((int32_t)dev->absmax_u64, t)), dev);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            if (e_in_exp) *e_in_exp = p0;
            if (!M) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
            if (kNext) next_head_exponent(nh, p0, e3_exp, dev);
        }
    }
    uint32_t mx = 0, mx_masked = 0;
    int s1 = 0;
    long long s1_total = 0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < items; i += gridDim.x * blockDim.x) {
        const uint32_t pix = i / (uint32_t)groups, row = pix / (uint32_t)w;
        const int gi = (int)(i - pix * (uint32_t)groups), ix = (int)(pix - row * (uint32_t)w);
        const int b = (int)(row / (uint32_t)h), iy = (int)(row - (uint32_t)b * (uint32_t)h);
        // windows o with o * s - p <= i <= o * s - p + k - 1
        const int oy_lo = max(0, (iy + p - k + s) / s), oy_hi = min(ho - 1, (iy + p) / s);
        const int ox_lo = max(0, (ix + p - k + s) / s), ox_hi = min(wo - 1, (ix + p) / s);
        uint32_t even[4] = {0, 0, 0, 0}, odd[4] = {0, 0, 0, 0};
        int nwin = 0;
        auto take = [&](const int4 &ev, const int4 &av, int oy, int ox) {
            const uint32_t me = (uint32_t)((iy - (oy * s - p)) * k + (ix - (ox * s - p))) * 0x01010101u;
            const uint32_t ew[4] = {(uint32_t)ev.x, (uint32_t)ev.y, (uint32_t)ev.z, (uint32_t)ev.w};
            const uint32_t aw[4] = {(uint32_t)av.x, (uint32_t)av.y, (uint32_t)av.z, (uint32_t)av.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t hit = __vcmpeq4(aw[q], me);           // 0xff in the bytes this position won
                const uint32_t v = (ew[q] & hit) ^ 0x80808080u;      // code + 128 there, 128 elsewhere
                even[q] += v & 0x00ff00ffu;
                odd[q] += (v >> 8) & 0x00ff00ffu;
            }
            ++nwin;
        };
        if (oy_hi - oy_lo <= 1 && ox_hi - ox_lo <= 1) {
            // the usual case (window at most twice the stride): at most 2 x 2 windows, all eight loads issued together
            int4 ev[4], av[4];
            bool in[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int oy = oy_lo + (u >> 1), ox = ox_lo + (u & 1);
                in[u] = oy <= oy_hi && ox <= ox_hi;
                const size_t o = (((size_t)b * ho + oy) * wo + ox) * c + gi * 16;
                ev[u] = in[u] ? __ldg(reinterpret_cast<const int4 *>(e + o)) : make_int4(0, 0, 0, 0);
                av[u] = in[u] ? __ldg(reinterpret_cast<const int4 *>(arg + o)) : make_int4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (in[u]) take(ev[u], av[u], oy_lo + (u >> 1), ox_lo + (u & 1));
        } else {
            for (int oy = oy_lo; oy <= oy_hi; ++oy)
                for (int ox = ox_lo; ox <= ox_hi; ++ox) {
                    const size_t o = (((size_t)b * ho + oy) * wo + ox) * c + gi * 16;
                    take(__ldg(reinterpret_cast<const int4 *>(e + o)), __ldg(reinterpret_cast<const int4 *>(arg + o)), oy, ox);
                }
        }
        int sum[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            sum[4 * q + 0] = (int)(even[q] & 0xffffu) - 128 * nwin;
            sum[4 * q + 1] = (int)(odd[q] & 0xffffu) - 128 * nwin;
            sum[4 * q + 2] = (int)(even[q] >> 16) - 128 * nwin;
            sum[4 * q + 3] = (int)(odd[q] >> 16) - 128 * nwin;
        }
        const uint32_t mbits = kNext ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(next_mask) + i) : 0u;
        if (kPass == 0) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const uint32_t v = (uint32_t)abs(sum[q]);
                mx = max(mx, v);
                if (kNext && ((mbits >> q) & 1u)) mx_masked = max(mx_masked, v);
            }
        } else {
            int cd[16];
            if (t >= 8) {   // a right shift by t - 7 >= 1 (sums are below 2^15, nothing can wrap)
                const int sh = t - 7, half_m1 = (1 << (sh - 1)) - 1;
#pragma unroll
                for (int q = 0; q < 16; ++q) cd[q] = sq_code32_shr(sum[q], sh, half_m1);
            } else {
#pragma unroll
                for (int q = 0; q < 16; ++q) cd[q] = sq_code32(sum[q], t);
            }
            if (e_in)
                reinterpret_cast<int4 *>(e_in)[i] =
                    make_int4((int)pack4(cd[0], cd[1], cd[2], cd[3]), (int)pack4(cd[4], cd[5], cd[6], cd[7]),
                              (int)pack4(cd[8], cd[9], cd[10], cd[11]), (int)pack4(cd[12], cd[13], cd[14], cd[15]));
            if (kNext) {
                int c3[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int e1 = ((mbits >> q) & 1u) ? cd[q] : 0;
                    s1 += e1;
                    c3[q] = next_head_code(nh, e1);
                }
                reinterpret_cast<int4 *>(e3)[i] =
                    make_int4((int)pack4(c3[0], c3[1], c3[2], c3[3]), (int)pack4(c3[4], c3[5], c3[6], c3[7]),
                              (int)pack4(c3[8], c3[9], c3[10], c3[11]), (int)pack4(c3[12], c3[13], c3[14], c3[15]));
                s1_total += s1;
                s1 = 0;
            }
        }
    }
    if (kPass == 0) {
        mx = (uint32_t)block_max_u64(mx);
        if (kNext) mx_masked = (uint32_t)block_max_u64(mx_masked);
        if (threadIdx.x == 0) {
            if (mx) atomicMax(&dev->absmax_u32, mx);
            if (kNext && mx_masked) atomicMax(&dev->absmax_u64, (unsigned long long)mx_masked);
        }
    } else {
        if (kNext && sum_e1) {
            s1_total = block_sum_i64(s1_total);
            if (threadIdx.x == 0 && s1_total) atomicAdd(reinterpret_cast<unsigned long long *>(&dev->sum0), (unsigned long long)s1_total);
        }
        if (last_block_done(dev)) {
            dev->absmax_u32 = 0;
            if (kNext) {
                dev->absmax_u64 = 0;
                if (sum_e1) *sum_e1 = (long long)atomicExch(reinterpret_cast<unsigned long long *>(&dev->sum0), 0ull);
            }
        }
    }
}

// The same for the pool of the ImageNet networks: window 3, stride 2, padding 1.  Position 2q of an axis lies in window q
// alone (as its row 1), position 2q + 1 in windows q (row 2) and q + 1 (row 0), so a thread owns the 2 x 2 positions of
// quad (qy, qx) for 16 channels and loads the four windows (qy, qx) .. (qy + 1, qx + 1) once for all nine pairs of
// position and window.  Codes are kept with an offset of 128 per window in unsigned 16-bit halves, so that they add
// without carries; a half joined with the upper half of 1.5 * 2^23 is that number plus the (offset) sum as a float, and
// one fused multiply-add takes the offset out, scales and rounds it to nearest even (see rne7_magic).
// Bound by instruction issue: about 8 instructions per code in pass 0, 14 in pass 1.  At batch 64, 51 M codes: pass 0
// 78 us, pass 1 90 us with a gather per position and 32-bit sums; now 39 and 49 us (both beside weight-gradient work).
struct PoolQuad {
    uint32_t even[4][4], odd[4][4];   // [position][word]: offset sums of channels 0, 2 / 1, 3 of the word's four
};
// offset of a position's halves: 128 per window pair, in both halves
__device__ __forceinline__ constexpr uint32_t quad_offset(int pos) { return 0x00800080u * (pos == 0 ? 1u : (pos == 3 ? 4u : 2u)); }

// adds one window to one position; kFirst: it is the position's first
template <bool kFirst>
__device__ __forceinline__ void quad_add(uint32_t (&even)[4], uint32_t (&odd)[4], const uint32_t (&e)[4], const uint32_t (&a)[4], uint32_t idx)
{
    const uint32_t me = idx * 0x01010101u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t x = a[q] ^ me;
        const uint32_t other = prmt<0xba98>(((x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | x, 0u);  // 0xff in the bytes another position won
        const uint32_t v = (e[q] & ~other) ^ 0x80808080u;
        if (kFirst) {
            even[q] = v & 0x00ff00ffu;
            odd[q] = prmt<0x4341>(v, 0u);
        } else {
            even[q] += v & 0x00ff00ffu;
            odd[q] += prmt<0x4341>(v, 0u);
        }
    }
}

__device__ __forceinline__ void quad_load(const int8_t *__restrict__ e, const uint8_t *__restrict__ arg, size_t o, bool in, uint32_t (&ew)[4],
                                          uint32_t (&aw)[4])
{
    const int4 z = make_int4(0, 0, 0, 0);
    const int4 ev = in ? __ldg(reinterpret_cast<const int4 *>(e + o)) : z, av = in ? __ldg(reinterpret_cast<const int4 *>(arg + o)) : z;
    ew[0] = (uint32_t)ev.x; ew[1] = (uint32_t)ev.y; ew[2] = (uint32_t)ev.z; ew[3] = (uint32_t)ev.w;
    aw[0] = (uint32_t)av.x; aw[1] = (uint32_t)av.y; aw[2] = (uint32_t)av.z; aw[3] = (uint32_t)av.w;
}

// Bit q of a nibble to the sign bit of byte q (the other bits are noise), for the sign-replicating permutes.
__device__ __forceinline__ uint32_t nibble_signs(uint32_t bits, int word) { return ((bits >> (4 * word)) & 0xfu) * 0x10204080u; }

template <int kPass, bool kNext>
__global__ void __launch_bounds__(kThreads)
maxpool_bwd_quad_kernel(const int8_t *__restrict__ e, const int32_t *e_exp, const uint8_t *__restrict__ arg, uint32_t items, int h, int w,
                        int c, int ho, int wo, int8_t *__restrict__ e_in, int32_t *e_in_exp, const uint8_t *__restrict__ next_mask,
                        const int32_t *next_gamma, int8_t *__restrict__ e3, int32_t *e3_exp, long long *sum_e1, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    if (kPass == 0 && kNext && blockIdx.x == 0 && threadIdx.x == 0 && sum_e1) *sum_e1 = 0;   // pass 1 adds to it
    const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
    const bool live = i < items;
    const int groups = c / 16;
    const uint32_t quad = (live ? i : 0u) / (uint32_t)groups, row = quad / (uint32_t)wo;
    const int g = (int)((live ? i : 0u) - quad * (uint32_t)groups), qx = (int)(quad - row * (uint32_t)wo);
    const int b = (int)(row / (uint32_t)ho), qy = (int)(row - (uint32_t)b * (uint32_t)ho);
    PoolQuad s;
    uint32_t mbits[4];
    bool in[4];
    const bool dn = qy + 1 < ho, rt = qx + 1 < wo;
    in[0] = live;
    in[1] = live && 2 * qx + 1 < w;
    in[2] = live && 2 * qy + 1 < h;
    in[3] = in[1] && in[2];
    const uint32_t pix = ((uint32_t)b * h + 2 * qy) * w + 2 * qx;   // 16-channel items stay below 2^31 (checked by the caller)
    const uint32_t at[4] = {pix * groups + g, (pix + 1) * groups + g, (pix + w) * groups + g, (pix + w + 1) * groups + g};
    {
        const size_t o = ((size_t)row * wo + qx) * c + g * 16;
        uint32_t e0[4], a0[4], e1[4], a1[4], e2[4], a2[4], e4[4], a4[4];
        quad_load(e, arg, o, live, e0, a0);
        quad_load(e, arg, o + c, live && rt, e1, a1);
        quad_load(e, arg, o + (size_t)wo * c, live && dn, e2, a2);
        quad_load(e, arg, o + (size_t)(wo + 1) * c, live && rt && dn, e4, a4);
#pragma unroll
        for (int p = 0; p < 4; ++p)
            mbits[p] = (kNext && in[p]) ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(next_mask) + at[p]) : 0u;
        quad_add<true>(s.even[0], s.odd[0], e0, a0, 4);
        quad_add<true>(s.even[1], s.odd[1], e0, a0, 5);
        quad_add<false>(s.even[1], s.odd[1], e1, a1, 3);
        quad_add<true>(s.even[2], s.odd[2], e0, a0, 7);
        quad_add<false>(s.even[2], s.odd[2], e2, a2, 1);
        quad_add<true>(s.even[3], s.odd[3], e0, a0, 8);
        quad_add<false>(s.even[3], s.odd[3], e1, a1, 6);
        quad_add<false>(s.even[3], s.odd[3], e2, a2, 2);
        quad_add<false>(s.even[3], s.odd[3], e4, a4, 0);
    }
    if (kPass == 0) {
        uint32_t mx = 0, mx_masked = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            if (!in[p]) continue;
            const uint32_t off = quad_offset(p);
            uint32_t hi = off, lo = off, him = off, lom = off;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                hi = __vimax3_u16x2(hi, s.even[p][q], s.odd[p][q]);
                lo = __vimin3_u16x2(lo, s.even[p][q], s.odd[p][q]);
                if (kNext) {
                    const uint32_t sg = nibble_signs(mbits[p], q);
                    const uint32_t me = prmt<0xaa88>(sg, 0u), mo = prmt<0xbb99>(sg, 0u);   // 0xffff in the halves the ReLU lets through
                    const uint32_t ev = (s.even[p][q] & me) | (off & ~me), ov = (s.odd[p][q] & mo) | (off & ~mo);
                    him = __vimax3_u16x2(him, ev, ov);
                    lom = __vimin3_u16x2(lom, ev, ov);
                }
            }
            const int o1 = (int)(off & 0xffffu);
            mx = max(mx, (uint32_t)max(max((int)(hi & 0xffffu), (int)(hi >> 16)) - o1, o1 - min((int)(lo & 0xffffu), (int)(lo >> 16))));
            if (kNext)
                mx_masked = max(mx_masked,
                                (uint32_t)max(max((int)(him & 0xffffu), (int)(him >> 16)) - o1, o1 - min((int)(lom & 0xffffu), (int)(lom >> 16))));
        }
        // both maxima are below 2^10: one reduction for the pair would need them ordered apart, so two
        __shared__ uint32_t red[2];
        if (threadIdx.x < 2) red[threadIdx.x] = 0;
        __syncthreads();
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (kNext) mx_masked = __reduce_max_sync(0xffffffffu, mx_masked);
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&red[0], mx);
            if (kNext) atomicMax(&red[1], mx_masked);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (red[0]) atomicMax(&dev->absmax_u32, red[0]);
            if (kNext && red[1]) atomicMax(&dev->absmax_u64, (unsigned long long)red[1]);
        }
    } else {
        __shared__ uint32_t m_s[2];
        __shared__ int sum_s;
        if (threadIdx.x == 0) {
            m_s[0] = *reinterpret_cast<volatile uint32_t *>(&dev->absmax_u32);
            m_s[1] = (uint32_t)*reinterpret_cast<volatile unsigned long long *>(&dev->absmax_u64);
            sum_s = 0;
        }
        __syncthreads();
        bool last = false;
        if (threadIdx.x == 0) last = last_reader(dev);   // the last block to have read the maxima clears them at its end
        const uint32_t M = m_s[0];
        const int t = M ? round_log2_u32(M) : 7;
        NextHead nh = {};
        if (kNext) nh = next_head_setup(next_gamma, (uint32_t)abs(sq_code32((int32_t)m_s[1], t)), dev);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            const int p_in = *e_exp, p0 = M ? p_in + t - 7 : p_in;
            if (e_in_exp) *e_in_exp = p0;
            if (!M) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
            if (kNext) next_head_exponent(nh, p0, e3_exp, dev);
        }
        constexpr int kLo = (int)kHeadMagic - 127, kHi = (int)kHeadMagic + 127;
        const float scale = __int_as_float((127 + 7 - t) << 23);   // 2^(7 - t), t in [0, 9]
        const uint32_t head_add = kHeadMagic - nh.g * kHeadMagic;
        int s1 = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const float rest = 12582912.0f - (12582912.0f + (float)(quad_offset(p) & 0xffffu)) * scale;  // exact
            uint32_t cw[4], hw[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t half[4] = {prmt<0x7610>(s.even[p][q], kHeadMagic), prmt<0x7610>(s.odd[p][q], kHeadMagic),
                                          prmt<0x7632>(s.even[p][q], kHeadMagic), prmt<0x7632>(s.odd[p][q], kHeadMagic)};
                int r[4], r3[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    r[k] = clampi((int)__float_as_uint(__fmaf_rn(__uint_as_float(half[k]), scale, rest)), kLo, kHi);
                    if (kNext) {
                        const uint32_t biased = nh.g * (uint32_t)r[k] + head_add;   // gamma * code + 1.5 * 2^23
                        r3[k] = __viaddmax_s32((int)__float_as_uint(__fmaf_rn(__uint_as_float(biased), nh.scale, nh.rest)), -(int)kHeadMagic, -127);
                    }
                }
                cw[q] = prmt<0x5410>(prmt<0x0040>((uint32_t)r[0], (uint32_t)r[1]), prmt<0x0040>((uint32_t)r[2], (uint32_t)r[3]));
                if (kNext) {
                    const uint32_t m = prmt<0xba98>(nibble_signs(mbits[p], q), 0u);
                    s1 = __dp4a((int)(cw[q] & m), 0x01010101, s1);
                    hw[q] = pack4_sat(r3[0], r3[1], r3[2], r3[3]) & m;   // the code of zero is zero
                }
            }
            if (in[p]) {
                if (e_in) reinterpret_cast<uint4 *>(e_in)[at[p]] = make_uint4(cw[0], cw[1], cw[2], cw[3]);
                if (kNext) reinterpret_cast<uint4 *>(e3)[at[p]] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
            }
        }
        if (kNext && sum_e1) {
            s1 = __reduce_add_sync(0xffffffffu, s1);
            if ((threadIdx.x & 31) == 0 && s1) atomicAdd(&sum_s, s1);
            __syncthreads();
            if (threadIdx.x == 0 && sum_s) atomicAdd(reinterpret_cast<unsigned long long *>(sum_e1), (unsigned long long)(long long)sum_s);
        }
        if (last) {
            dev->absmax_u32 = 0;
            if (kNext) dev->absmax_u64 = 0;
        }
    }
}

}  // namespace

cudaError_t launch_maxpool_fwd(const int8_t *x, int n, int h, int w, int c, int k, int s, int p, int8_t *y, uint8_t *arg, cudaStream_t st)
{
    const int ho = (h + 2 * p - k) / s + 1, wo = (w + 2 * p - k) / s + 1;
    const uint32_t items = (uint32_t)n * ho * wo * (c / 16);   // below 2^31 (checked by the caller)
    const unsigned blocks = (items + kThreads - 1) / kThreads;
    if (k == 3) launch_chained(maxpool_fwd_kernel<3>, blocks, kThreads, 0, st, x, items, h, w, c, k, s, p, ho, wo, y, arg);
    else launch_chained(maxpool_fwd_kernel<0>, blocks, kThreads, 0, st, x, items, h, w, c, k, s, p, ho, wo, y, arg);
    return cudaGetLastError();
}

cudaError_t launch_maxpool_bwd(const int8_t *e, const int32_t *e_exp, const uint8_t *arg, int n, int h, int w, int c, int k, int s,
                               int p, int8_t *e_in, int32_t *e_in_exp, const uint8_t *next_mask, const int32_t *next_gamma, int8_t *e3,
                               int32_t *e3_exp, long long *sum_e1, DeviceState *dev, int sm_count, cudaStream_t st,
                               const ReduceHook &hook)
{
    const int ho = (h + 2 * p - k) / s + 1, wo = (w + 2 * p - k) / s + 1;
    const bool quads = k == 3 && s == 2 && p == 1;
    const uint32_t qitems = (uint32_t)n * ho * wo * (c / 16);
    size_t blocks = ((size_t)n * h * w * (c / 16) + kThreads - 1) / kThreads;
    if (blocks > (size_t)sm_count * 32) blocks = (size_t)sm_count * 32;
    const unsigned grid = quads ? (qitems + kThreads - 1) / kThreads : (unsigned)blocks;
    auto pass = [&](auto kernel, auto quad_kernel) {
        if (quads)
            launch_chained(quad_kernel, grid, kThreads, 0, st, e, e_exp, arg, qitems, h, w, c, ho, wo, e_in, e_in_exp, next_mask, next_gamma, e3, e3_exp,
                                                   sum_e1, dev);
        else
            kernel<<<grid, kThreads, 0, st>>>(e, e_exp, arg, n, h, w, c, k, s, p, ho, wo, e_in, e_in_exp, next_mask, next_gamma, e3, e3_exp,
                                              sum_e1, dev);
    };
    if (e3) pass(maxpool_bwd_kernel<0, true>, maxpool_bwd_quad_kernel<0, true>);
    else pass(maxpool_bwd_kernel<0, false>, maxpool_bwd_quad_kernel<0, false>);
    hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, st);
    if (e3) hook(&dev->absmax_u64, 1, EOQ_REDUCE_I64, EOQ_REDUCE_MAX, st);
    if (e3) pass(maxpool_bwd_kernel<1, true>, maxpool_bwd_quad_kernel<1, true>);
    else pass(maxpool_bwd_kernel<1, false>, maxpool_bwd_quad_kernel<1, false>);
    if (e3 && sum_e1) hook(sum_e1, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, st);
    return cudaGetLastError();
}

}  // namespace eoq
