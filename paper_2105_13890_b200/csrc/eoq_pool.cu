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
// position and window.  A sum is one byte dot product of a channel's four error codes with zeros and ones, and these come out of an
// eight-byte table by one permute for all four windows: its selector is four digits, one per window, that say which of the
// quad's positions the window elected (0: (1,1), 1: (1,0), 3: (0,1), 4: (0,0); every other digit finds a zero).
// Bound by instruction issue, of the integer pipe above all.  With a compare and two additions per pair, position and code, in
// 16-bit halves, 51 M codes took 30.8 us in pass 0 and 41.6 in pass 1, now 25.5 and 32.0.

// The positions of the quad are numbered 2 * row + column, the windows likewise.
__device__ __forceinline__ uint32_t table_bytes(uint32_t lo, uint32_t hi, uint32_t digits)
{
    uint32_t r;   // (a digit of 8 or more repeats the sign of a byte: zero, as all of them are 0 or 1)
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(digits));
    return r;
}

// Sums of the four positions for the four channels of a word, each plus `bias`: e, a = the word of every window (positions 0 to 8).
__device__ __forceinline__ void quad_sums(const uint32_t (&e)[4], const uint32_t (&a)[4], uint32_t bias, uint32_t (&s)[4][4])
{
    // Digits.  8 - a, 6 - a, 2 - a and -a modulo 16 are 0 where a window elects position 3; the same differences give the others their
    // digits.  Window 1 also shows 4 and 1 for positions that are not the quad's: it is left out where it has no part.
    const uint32_t v0 = (0x18181818u - a[0]) & 0x0f0f0f0fu, v1 = (0x16161616u - a[1]) & 0x0f0f0f0fu, v2 = (0x12121212u - a[2]) & 0x0f0f0f0fu,
                   v3 = (0x10101010u - a[3]) & 0x0f0f0f0fu;
    const uint32_t lo = v1 * 16u + v0, hi = v3 * 16u + v2;
    // the codes of a channel side by side
    const uint32_t t0 = __byte_perm(e[0], e[1], 0x5140), t1 = __byte_perm(e[0], e[1], 0x7362), t2 = __byte_perm(e[2], e[3], 0x5140),
                   t3 = __byte_perm(e[2], e[3], 0x7362);
    const uint32_t codes[4] = {__byte_perm(t0, t2, 0x5410), __byte_perm(t0, t2, 0x7632), __byte_perm(t1, t3, 0x5410), __byte_perm(t1, t3, 0x7632)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t digits = __byte_perm(lo, hi, (uint32_t)((4 + k) << 4 | k)), but1 = codes[k] & 0xffff00ffu;
        s[0][k] = (uint32_t)__dp4a((int)but1, (int)table_bytes(0u, 0x00000001u, digits), (int)bias);
        s[1][k] = (uint32_t)__dp4a((int)codes[k], (int)table_bytes(0x01000000u, 0u, digits), (int)bias);
        s[2][k] = (uint32_t)__dp4a((int)but1, (int)table_bytes(0x00000100u, 0u, digits), (int)bias);
        s[3][k] = (uint32_t)__dp4a((int)codes[k], (int)table_bytes(0x00000001u, 0u, digits), (int)bias);
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
    uint32_t mbits[4];
    bool in[4];
    const bool dn = qy + 1 < ho, rt = qx + 1 < wo;
    in[0] = live;
    in[1] = live && 2 * qx + 1 < w;
    in[2] = live && 2 * qy + 1 < h;
    in[3] = in[1] && in[2];
    const uint32_t pix = ((uint32_t)b * h + 2 * qy) * w + 2 * qx;   // 16-channel items stay below 2^31 (checked by the caller)
    const uint32_t at[4] = {pix * groups + g, (pix + 1) * groups + g, (pix + w) * groups + g, (pix + w + 1) * groups + g};
    uint32_t ew[4][4], aw[4][4];   // [window][word]
    {
        const size_t o = ((size_t)row * wo + qx) * c + g * 16;
        quad_load(e, arg, o, live, ew[0], aw[0]);
        quad_load(e, arg, o + c, live && rt, ew[1], aw[1]);
        quad_load(e, arg, o + (size_t)wo * c, live && dn, ew[2], aw[2]);
        quad_load(e, arg, o + (size_t)(wo + 1) * c, live && rt && dn, ew[3], aw[3]);
#pragma unroll
        for (int p = 0; p < 4; ++p)
            mbits[p] = (kNext && in[p]) ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(next_mask) + at[p]) : 0u;
        // a byte beyond 8 elects nothing (the forward pass writes none)
        uint32_t any = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) any |= aw[u][q] | (aw[u][q] + 0x07070707u);
        if (any & 0xf0f0f0f0u) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t beyond = prmt<0xba98>(((aw[u][q] & 0x7f7f7f7fu) + 0x77777777u) | aw[u][q], 0u);
                    ew[u][q] &= ~beyond;
                    aw[u][q] &= ~beyond;
                }
        }
    }
    auto word_sums = [&](int q, uint32_t bias, uint32_t (&s)[4][4]) {
        const uint32_t e4[4] = {ew[0][q], ew[1][q], ew[2][q], ew[3][q]}, a4[4] = {aw[0][q], aw[1][q], aw[2][q], aw[3][q]};
        quad_sums(e4, a4, bias, s);
    };
    if (kPass == 0) {
        // sums plus 1024 (|sum| <= 4 * 128), two to a word
        constexpr uint32_t kOff = 0x04000400u;
        uint32_t hi = kOff, lo = kOff, him = kOff, lom = kOff;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t s[4][4];
            word_sums(q, 1024u, s);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const uint32_t s01 = s[p][1] * 65536u + s[p][0], s23 = s[p][3] * 65536u + s[p][2];
                if (in[p]) {
                    hi = __vimax3_u16x2(hi, s01, s23);
                    lo = __vimin3_u16x2(lo, s01, s23);
                }
                if (kNext) {
                    const uint32_t sg = nibble_signs(mbits[p], q);
                    const uint32_t m01 = prmt<0x9988>(sg, 0u), m23 = prmt<0xbbaa>(sg, 0u);   // 0xffff in the halves the ReLU lets through
                    const uint32_t e01 = (s01 & m01) | (kOff & ~m01), e23 = (s23 & m23) | (kOff & ~m23);
                    him = __vimax3_u16x2(him, e01, e23);
                    lom = __vimin3_u16x2(lom, e01, e23);
                }
            }
        }
        auto most = [&](uint32_t h, uint32_t l) {
            return (uint32_t)max(max((int)(h & 0xffffu), (int)(h >> 16)) - 1024, 1024 - min((int)(l & 0xffffu), (int)(l >> 16)));
        };
        uint32_t mx = most(hi, lo), mx_masked = kNext ? most(him, lom) : 0u;
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
        const float scale = __int_as_float((127 + 7 - t) << 23);   // 2^(7 - t), t in [0, 9]
        const float rest = 12582912.0f - 12582912.0f * scale;      // exact; the sums arrive plus 1.5 * 2^23 (see next_head_codes)
        int s1 = 0;
        uint32_t cw[4][4], hw[4][4];   // [position][word]
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t s[4][4];
            word_sums(q, kHeadMagic, s);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                int r[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    r[k] = __viaddmax_s32((int)__float_as_uint(__fmaf_rn(__uint_as_float(s[p][k]), scale, rest)), -(int)kHeadMagic, -127);
                cw[p][q] = pack4_sat(r[0], r[1], r[2], r[3]);
                if (kNext) {
                    const uint32_t e1 = cw[p][q] & prmt<0xba98>(nibble_signs(mbits[p], q), 0u);
                    s1 = __dp4a((int)e1, 0x01010101, s1);
                    hw[p][q] = next_head_codes(nh, e1);
                }
            }
        }
#pragma unroll
        for (int p = 0; p < 4; ++p)
            if (in[p]) {
                if (e_in) reinterpret_cast<uint4 *>(e_in)[at[p]] = make_uint4(cw[p][0], cw[p][1], cw[p][2], cw[p][3]);
                if (kNext) reinterpret_cast<uint4 *>(e3)[at[p]] = make_uint4(hw[p][0], hw[p][1], hw[p][2], hw[p][3]);
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
