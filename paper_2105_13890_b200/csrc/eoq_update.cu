// The 8-bit update (arXiv 2105.13890, Sec. 3.2.3): u = Q_u(lr g) = SQ(lr g, 8), w <- Q_w(w - u) on the int8 codes, and
// its generic-width form on master codes.  All tensors of a call go through one launch pair: a maximum per tensor, then
// the update under it; when every tensor is small, one block takes a tensor through both passes and one launch does it.
#include "eoq_cells.cuh"
#include "eoq_device.cuh"
#include "eoq_internal.h"

namespace eoq {

namespace {

constexpr int kThreads = 256;
constexpr int kUpdChunk = 64;            // tensors per launch
constexpr int kUpdElemsPerBlock = 8192;  // elements one block covers
// Tensors up to kSmallElems are updated by one block or one cluster each, in one launch: every weight tensor of the
// CIFAR-shaped networks (at most 36,864 codes).  Beyond kSmallPart codes stochastic rounding takes one block too long
// (36,864 codes: 11 us, a cluster of eight 6 us).
constexpr int kSmallThreads = 1024;
constexpr int kSmallGroups = 4;          // 16-code groups per thread
constexpr size_t kSmallElems = (size_t)kSmallThreads * kSmallGroups * 16;
constexpr size_t kSmallPart = 8192;
constexpr int kSmallMostParts = 8;
// A block of a cluster has one group per thread at most.  At 64 registers two such blocks share an SM, so that the clusters of 37
// tensors start together (blocks of 1024 threads: of 18; the 22 tensors of ResNet-20 8.9 us, with 512 threads 8.3 us).
constexpr int kSmallPartThreads = (int)(kSmallElems / kSmallMostParts / 16);

struct UpdateBatch {
    UpdateTensor t[kUpdChunk];
    int first_block[kUpdChunk + 1];
    int num;
    int tensor_base;  // index of t[0] in the whole call (cell of its maximum, counter of the hash)
    int last;         // the last launch for a step: its last block moves the step counter on
};

__device__ __forceinline__ int find_tensor(const UpdateBatch &b, int block)
{
    int lo = 0, hi = b.num - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (block >= b.first_block[mid]) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Running maximum and minimum of 16 codes as packed halves: bytes are sign-extended to 16 bits by one permute per two
// codes (selector digit 8 + k replicates the sign of byte k).
struct AbsMax16 {
    uint32_t mx = 0, mn = 0;
    __device__ __forceinline__ void add_word(uint32_t w)
    {
        uint32_t even, odd;
        asm("prmt.b32 %0, %1, %1, 0xA280;" : "=r"(even) : "r"(w));
        asm("prmt.b32 %0, %1, %1, 0xB391;" : "=r"(odd) : "r"(w));
        mx = __vimax3_s16x2(mx, even, odd);
        mn = __vimin3_s16x2(mn, even, odd);
    }
    __device__ __forceinline__ void add(const int4 &v)
    {
        add_word((uint32_t)v.x);
        add_word((uint32_t)v.y);
        add_word((uint32_t)v.z);
        add_word((uint32_t)v.w);
    }
    __device__ __forceinline__ uint32_t value() const
    {
        const int hi = max((int)(int16_t)mx, (int)mx >> 16), lo = min((int)(int16_t)mn, (int)mn >> 16);
        return (uint32_t)max(hi, -lo);
    }
};

// Bound by HBM / L2 reads (1 B per weight).  The 21 M weights of ResNet-34: 13.4 us with a 32-bit maximum per code, 7.4 us
// with packed 16-bit ones, 6.7 with both loads of a thread in flight.
__global__ void __launch_bounds__(kThreads) update_absmax_kernel(const __grid_constant__ UpdateBatch b, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    const int k = find_tensor(b, blockIdx.x);
    const UpdateTensor &T = b.t[k];
    const size_t begin = (size_t)(blockIdx.x - b.first_block[k]) * kUpdElemsPerBlock;
    const size_t end = min((size_t)T.n, begin + kUpdElemsPerBlock);
    uint32_t mx = 0;
    if (begin < end) {
        // 16-byte path when the tensor base allows it (it always does for 16-byte aligned tensors)
        const bool vec = (reinterpret_cast<uintptr_t>(T.g) & 15) == 0;
        AbsMax16 am;
        if (vec) {
            constexpr int kLoads = kUpdElemsPerBlock / (kThreads * 16);   // all in flight together
            int4 v[kLoads];
#pragma unroll
            for (int q = 0; q < kLoads; ++q) {
                const size_t i = begin + ((size_t)q * kThreads + threadIdx.x) * 16;
                v[q] = i + 16 <= end ? __ldg(reinterpret_cast<const int4 *>(T.g + i)) : make_int4(0, 0, 0, 0);
            }
#pragma unroll
            for (int q = 0; q < kLoads; ++q) am.add(v[q]);
        }
        mx = am.value();
        // remaining elements of this block's range
        const size_t tail = vec ? begin + ((end - begin) / 16) * 16 : begin;
        for (size_t j = tail + threadIdx.x; j < end; j += kThreads) mx = max(mx, (uint32_t)abs((int)T.g[j]));
    }
    mx = block_max_u32(mx);
    if (threadIdx.x == 0 && mx) atomicMax(&dev->tensor_absmax[b.tensor_base + k], mx);
}

// What the update of one tensor needs, the same for all its elements.
struct UpdateRule {
    int d;                 // exponent of u relative to the weight grid 2^-7: w - u * 2^d
    float scale;           // u = sat(R(g * scale))
    bool same, clips;      // u = g; some |g| reaches beyond 127
    unsigned long long key;
};

// `max_g`: the largest |g| of the tensor, M = lr_mant * max_g != 0
__device__ __forceinline__ UpdateRule update_rule(uint32_t max_g, int g_exp, int lr_mant, int lr_exp, int stochastic, unsigned long long seed,
                                                  unsigned long long step, int tensor)
{
    UpdateRule r;
    const int t = round_log2_u32(max_g * (uint32_t)lr_mant);
    r.scale = (float)lr_mant * __int_as_float((127 + 7 - t) << 23);   // exact, as every g * scale is
    r.clips = (float)max_g * r.scale >= 127.5f;                       // (which ties to 128)
    r.same = r.scale == 1.0f && !r.clips;
    r.d = (g_exp + lr_exp + t - 7) + 7;
    r.key = 0;
    if (stochastic) {
        r.key = rounding_key(seed, step, (unsigned long long)tensor);
    }
    return r;
}

// How w - u * 2^d is rounded; every mode is one short sequence of 32-bit operations (only kStochasticWide needs 64 bits).
enum UpdateMode {
    kShiftUp,         // d >= 0: u moves left, nothing is rounded
    kNearest,         // -7 <= d < 0, ties to even
    kKeep,            // |u| <= 127 stays below half a unit (d <= -8, nearest; d < -40, stochastic): only the clamp acts
    kStochastic,      // -30 <= d < 0
    kStochasticWide,  // -40 <= d < -30
};
__device__ __forceinline__ UpdateMode update_mode(const UpdateRule &r, int stochastic)
{
    if (r.d >= 0) return kShiftUp;
    if (stochastic) return r.d < -40 ? kKeep : (r.d < -30 ? kStochasticWide : kStochastic);
    return r.d < -7 ? kKeep : kNearest;
}

// How u comes from g: as it is (a learning rate that is a power of two, behind Q_g, whose largest code is 91 or more), by a rounded
// product, or by one that the quantizer clips.
enum UpdateCode { kSame, kScaled, kClipped };

// What the loops keep in registers.
struct UpdateLoop {
    int s;                 // -d
    uint32_t mask, one;    // 2^s - 1; 1, though the compiler does not know: a multiply-add adds it on the multiply-add pipe
    float scale;           // -scale of the rule
};
__device__ __forceinline__ UpdateLoop update_loop(const UpdateRule &r)
{
    UpdateLoop l;
    l.s = -r.d;
    l.mask = r.d < 0 && r.d >= -30 ? (1u << -r.d) - 1u : 0u;
    asm volatile("mov.u32 %0, 1;" : "=r"(l.one));
    l.scale = -r.scale;
    return l;
}

__device__ __forceinline__ uint32_t mad_lo(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// Low words of mix64 under a mask, the products on 32-bit halves.
__device__ __forceinline__ uint32_t mix64_low(unsigned long long z, uint32_t mask)
{
    constexpr uint32_t kLo1 = 0x1CE4E5B9u, kHi1 = 0xBF58476Du, kLo2 = 0x133111EBu, kHi2 = 0x94D049BBu;
    uint32_t lo = (uint32_t)z, hi = (uint32_t)(z >> 32);
    uint32_t a = lo ^ __funnelshift_r(lo, hi, 30), b = hi ^ (hi >> 30);
    unsigned long long p = (unsigned long long)a * kLo1;
    lo = (uint32_t)p;
    hi = mad_lo(b, kLo1, mad_lo(a, kHi1, (uint32_t)(p >> 32)));
    a = lo ^ __funnelshift_r(lo, hi, 27);
    b = hi ^ (hi >> 27);
    p = (unsigned long long)a * kLo2;
    lo = (uint32_t)p;
    hi = mad_lo(b, kLo2, mad_lo(a, kHi2, (uint32_t)(p >> 32)));
    return (lo ^ __funnelshift_r(lo, hi, 31)) & mask;
}

// byte k of `codes` (signed) times +-1, plus c: a byte dot product takes the code out of its word on the multiply-add pipe
template <int k, bool kMinus>
__device__ __forceinline__ int add_code(uint32_t codes, int c)
{
    int d;
    asm("dp4a.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(codes), "r"((kMinus ? 0xffu : 1u) << (8 * k)), "r"(c));
    return d;
}

constexpr uint32_t kUpdateMagic = 0x4B400000u;   // 1.5 * 2^23 as a float
// c - u of the code in byte k of `g` (`biased`: the word with its sign bits flipped).  -u = R(g * -scale) by one multiply-add: the
// byte above 2^23 is a float, 2^23 + 128 off it leaves g.
template <UpdateCode kCode, int k>
__device__ __forceinline__ int subtract_u(int c, uint32_t g, uint32_t biased, const UpdateLoop &l)
{
    if (kCode == kSame) return add_code<k, true>(g, c);
    const float x = __uint_as_float(__byte_perm(biased, 0x4B000000u, 0x7540 | k)) - 8388736.0f;
    const int bits = (int)__float_as_uint(__fmaf_rn(x, l.scale, 12582912.0f));
    if (kCode == kScaled) return c + bits - (int)kUpdateMagic;
    return c + min(__viaddmax_s32(bits, -(int)kUpdateMagic, -127), 127);
}

// New code of byte k of w; z: the element's hash counter key + (index + 1) * golden (stochastic modes).  The result still needs the
// upper clamp at 127 (the packing saturates there); the lower one at -127 is applied here.
template <UpdateMode kMode, UpdateCode kCode, int k>
__device__ __forceinline__ int update_code(uint32_t w, uint32_t g, uint32_t biased, const UpdateLoop &l, unsigned long long z)
{
    if (kMode == kKeep) return max(sbyte<k>(w), -127);
    if (kMode == kShiftUp) {
        return max(sbyte<k>(w) + subtract_u<kCode, k>(0, g, biased, l) * (1 << min(-l.s, 9)), -127);   // any |u| * 2^9 saturates, as any larger power would
    } else if (kMode == kNearest) {
        const int v = subtract_u<kCode, k>(sbyte<k>(w) * (1 << l.s), g, biased, l);
        return max((v + ((1 << (l.s - 1)) - 1) + ((v >> l.s) & 1)) >> l.s, -127);
    } else if (kMode == kStochastic) {
        // floor((w 2^s - u + rand) / 2^s) = w + floor((rand - u) / 2^s)
        return max(add_code<k, false>(w, subtract_u<kCode, k>((int)mix64_low(z, l.mask), g, biased, l) >> l.s), -127);
    } else {
        return max(sbyte<k>(w) + (int)(((long long)(mix64(z) & ((1ull << l.s) - 1ull)) + subtract_u<kCode, k>(0, g, biased, l)) >> l.s), -127);
    }
}

template <UpdateMode kMode, UpdateCode kCode>
__device__ __forceinline__ int4 update_16(const int4 &wv, const int4 &gv, const UpdateLoop &l, unsigned long long key, size_t i)
{
    const uint32_t ww[4] = {(uint32_t)wv.x, (uint32_t)wv.y, (uint32_t)wv.z, (uint32_t)wv.w};
    const uint32_t gw[4] = {(uint32_t)gv.x, (uint32_t)gv.y, (uint32_t)gv.z, (uint32_t)gv.w};
    uint32_t o[4];
    unsigned long long z = key + kGolden * ((unsigned long long)i + 1);
    auto next = [&]() {   // z, and on to the next element's: z + golden as two multiply-adds
        const unsigned long long now = z;
        if (kMode == kStochastic) {
            asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(z) : "r"(l.one), "r"((uint32_t)kGolden), "l"(now));
            z = (unsigned long long)mad_lo(l.one, (uint32_t)(kGolden >> 32), (uint32_t)(z >> 32)) << 32 | (uint32_t)z;
        } else {
            z += kGolden;
        }
        return now;
    };
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t b = gw[q] ^ 0x80808080u;
        const int c0 = update_code<kMode, kCode, 0>(ww[q], gw[q], b, l, next());
        const int c1 = update_code<kMode, kCode, 1>(ww[q], gw[q], b, l, next());
        const int c2 = update_code<kMode, kCode, 2>(ww[q], gw[q], b, l, next());
        const int c3 = update_code<kMode, kCode, 3>(ww[q], gw[q], b, l, next());
        o[q] = pack4_sat(c0, c1, c2, c3);
    }
    return make_int4((int)o[0], (int)o[1], (int)o[2], (int)o[3]);
}

// elements [begin, end) of one tensor by the calling block
template <UpdateMode kMode, UpdateCode kCode>
__device__ __forceinline__ void update_range(const UpdateTensor &T, size_t begin, size_t end, const UpdateRule &r)
{
    const UpdateLoop l = update_loop(r);
    const bool vec = ((reinterpret_cast<uintptr_t>(T.g) | reinterpret_cast<uintptr_t>(T.w)) & 15) == 0;
    if (vec)
        for (size_t i = begin + (size_t)threadIdx.x * 16; i + 16 <= end; i += (size_t)blockDim.x * 16) {
            const int4 gv = kMode == kKeep ? make_int4(0, 0, 0, 0) : __ldg(reinterpret_cast<const int4 *>(T.g + i));
            const int4 wv = *reinterpret_cast<const int4 *>(T.w + i);
            *reinterpret_cast<int4 *>(T.w + i) = update_16<kMode, kCode>(wv, gv, l, r.key, i);
        }
    const size_t tail = vec ? begin + ((end - begin) / 16) * 16 : begin;
    for (size_t j = tail + threadIdx.x; j < end; j += blockDim.x) {
        const uint32_t g = (uint8_t)T.g[j];
        T.w[j] = (int8_t)min(update_code<kMode, kCode, 0>((uint8_t)T.w[j], g, g ^ 0x80u, l, r.key + kGolden * ((unsigned long long)j + 1)), 127);
    }
}

// (Only the stochastic loop, the one that arithmetic bounds, is worth a form without the clamps or the product: the whole call for the
// 21 M weights of ResNet-34 takes 32.9 us with u = g, 35.5 with a product and 37.3 with the clamps too, 42.5 before there were forms.  To
// nearest all take the form with the clamps: 18.8 to 25.6 us, by the shift, 21.2 to 30.4 before.)
__device__ __forceinline__ void update_range(UpdateMode mode, const UpdateTensor &T, size_t begin, size_t end, const UpdateRule &r)
{
    switch (mode) {
        case kShiftUp: update_range<kShiftUp, kClipped>(T, begin, end, r); break;
        case kNearest: update_range<kNearest, kClipped>(T, begin, end, r); break;
        case kKeep: update_range<kKeep, kSame>(T, begin, end, r); break;
        case kStochastic:
            if (r.same) update_range<kStochastic, kSame>(T, begin, end, r);
            else if (!r.clips) update_range<kStochastic, kScaled>(T, begin, end, r);
            else update_range<kStochastic, kClipped>(T, begin, end, r);
            break;
        default: update_range<kStochasticWide, kClipped>(T, begin, end, r); break;
    }
}

// w <- Q_w(w - Q_u(lr * g)).  Bound by the integer pipe and by issue under stochastic rounding: 32 instructions a weight, of which the
// 64-bit hash's shifts and exclusive-ors, 10, can go nowhere else (the pipe takes an instruction every two cycles and scheduler); codes
// are taken out of their words, scaled and added on the multiply-add pipe.  The 21 M weights of ResNet-34: 37.3 us with 43
// instructions, 24 of them on that pipe, 28.6 with 15 and six blocks to an SM (31.0 with four).  Rounding to nearest is bound by its
// loads.  Every rounding mode is a loop of its own on 32-bit values.
__global__ void __launch_bounds__(kThreads, 6)
update_apply_kernel(const __grid_constant__ UpdateBatch b, int32_t lr_mant, int32_t lr_exp, int stochastic, unsigned long long seed,
                    unsigned long long step, unsigned long long *step_dev, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    __shared__ unsigned long long step_s;
    __shared__ uint32_t max_s;
    const int k = find_tensor(b, blockIdx.x);
    const UpdateTensor &T = b.t[k];
    const int g_exp = __ldg(T.g_exp);
    if (threadIdx.x == 0) {
        step_s = step_dev ? *reinterpret_cast<volatile unsigned long long *>(step_dev) : step;
        max_s = *reinterpret_cast<volatile unsigned *>(&dev->tensor_absmax[b.tensor_base + k]);
    }
    __syncthreads();
    bool last = false;
    if (threadIdx.x == 0) last = last_reader(dev);
    if (max_s != 0) {
        const UpdateRule r = update_rule(max_s, g_exp, lr_mant, lr_exp, stochastic, seed, step_s, b.tensor_base + k);
        const size_t begin = (size_t)(blockIdx.x - b.first_block[k]) * kUpdElemsPerBlock;
        update_range(update_mode(r, stochastic), T, begin, min((size_t)T.n, begin + kUpdElemsPerBlock), r);
    } else if (threadIdx.x == 0 && (int)blockIdx.x == b.first_block[k]) {
        atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);  // u = 0: the weights keep their codes
    }
    if (last) {
        for (int i = 0; i < b.num; ++i) dev->tensor_absmax[b.tensor_base + i] = 0;
        if (b.last && step_dev) *step_dev = step_s + 1ull;
    }
}

// Both passes of one small tensor in one block, or in a cluster of `parts` blocks that exchange their maxima through
// distributed shared memory (see kSmallElems and kSmallPart).  Bound by latency: one read of g, one reduction, one read and
// one write of w.  2,304 weights: 3.5 us, where a cleared cell, two passes and the step counter's own kernel took four launches
// and 8.8 us.
__global__ void __launch_bounds__(kSmallThreads)
update_small_kernel(const __grid_constant__ UpdateBatch b, int parts, int32_t lr_mant, int32_t lr_exp, int stochastic,
                    unsigned long long seed, unsigned long long step, unsigned long long *step_dev, DeviceState *dev)
{
    __shared__ unsigned long long step_s;
    __shared__ __align__(16) uint32_t max_s[kSmallMostParts];
    const int k = (int)blockIdx.x / parts, part = (int)blockIdx.x - k * parts;
    if (parts > 1) ptx::cluster_arrive();   // met below: the other blocks have started before their shared memory is written
    ptx::grid_dep_wait_launch_small();
    const UpdateTensor &T = b.t[k];
    const int g_exp = __ldg(T.g_exp);
    if (threadIdx.x == 0) step_s = step_dev ? *reinterpret_cast<volatile unsigned long long *>(step_dev) : step;
    const size_t n = (size_t)T.n, slice = ((n + parts - 1) / parts + 15) / 16 * 16;
    const size_t begin = min(n, part * slice), end = min(n, begin + slice);
    const bool vec = (reinterpret_cast<uintptr_t>(T.g) & 15) == 0;
    AbsMax16 am;
    if (vec) {
#pragma unroll
        for (int q = 0; q < kSmallGroups; ++q) {
            const size_t i = begin + ((size_t)q * blockDim.x + threadIdx.x) * 16;
            if (i + 16 <= end) am.add(__ldg(reinterpret_cast<const int4 *>(T.g + i)));
        }
    }
    uint32_t mx = am.value();
    for (size_t j = (vec ? begin + (end - begin) / 16 * 16 : begin) + threadIdx.x; j < end; j += blockDim.x)
        mx = max(mx, (uint32_t)abs((int)T.g[j]));
    mx = block_max_u32(mx);
    if (parts > 1) {
        ptx::cluster_wait();
        if (threadIdx.x < 32) {
            mx = __shfl_sync(0xffffffffu, mx, 0);
            if ((int)threadIdx.x < parts) ptx::st_cluster_32(ptx::cluster_addr(ptx::smem_u32(&max_s[part]), threadIdx.x), mx);
        }
        ptx::cluster_sync();
        mx = 0;
        for (int i = 0; i < parts; ++i) mx = max(mx, max_s[i]);
    } else {
        if (threadIdx.x == 0) max_s[0] = mx;
        __syncthreads();
        mx = max_s[0];
    }
    bool last = false;
    if (threadIdx.x == 0) last = last_reader(dev);
    if (mx != 0) {
        const UpdateRule r = update_rule(mx, g_exp, lr_mant, lr_exp, stochastic, seed, step_s, b.tensor_base + k);
        update_range(update_mode(r, stochastic), T, begin, end, r);
    } else if (threadIdx.x == 0 && part == 0) {
        atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
    }
    if (last && b.last && step_dev) *step_dev = step_s + 1ull;
}

// The update with a k_u-bit update quantizer and k_m-bit master codes (Sec. 3.2.3 compares the 8-bit update with a
// 24-bit one): u = SQ(lr g, k_u), master <- CQ(master - u, k_m) on the grid 2^-(k_m - 1), w = Q_w(master).
__global__ void update_wide_apply_kernel(const __grid_constant__ UpdateBatch b, int32_t lr_mant, int32_t lr_exp, int k_u, int k_m,
                                         int stochastic, unsigned long long seed, unsigned long long step,
                                         unsigned long long *step_dev, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    __shared__ unsigned long long step_s;
    __shared__ uint32_t max_s;
    const int k = find_tensor(b, blockIdx.x);
    const UpdateTensor &T = b.t[k];
    if (threadIdx.x == 0) {
        step_s = step_dev ? *reinterpret_cast<volatile unsigned long long *>(step_dev) : step;
        max_s = *reinterpret_cast<volatile unsigned *>(&dev->tensor_absmax[b.tensor_base + k]);
    }
    __syncthreads();
    bool last = false;
    if (threadIdx.x == 0) last = last_reader(dev);
    step = step_s;
    const uint32_t M = max_s * (uint32_t)lr_mant;
    if (M != 0) {
        const int t = round_log2_u32(M);
        const int su = t - (k_u - 1);                                  // u code = R(lr_mant g / 2^su)
        const int d = (__ldg(T.g_exp) + lr_exp + su) + (k_m - 1);      // exponent of u relative to the master grid
        const long long lim_u = (1ll << (k_u - 1)) - 1, lim_m = (1ll << (k_m - 1)) - 1;
        unsigned long long key = 0;
        if (stochastic) key = rounding_key(seed, step, (unsigned long long)(b.tensor_base + k));
        const size_t begin = (size_t)(blockIdx.x - b.first_block[k]) * kUpdElemsPerBlock;
        const size_t end = min((size_t)T.n, begin + kUpdElemsPerBlock);
        for (size_t j = begin + threadIdx.x; j < end; j += blockDim.x) {
            const long long a = (long long)lr_mant * T.g[j];
            long long u = su >= 0 ? rne_shr64(a, su) : a * (1ll << (-su));
            u = u < -lim_u ? -lim_u : (u > lim_u ? lim_u : u);
            const long long th = T.master[j];
            long long next;
            if (d >= 0) {
                next = th - u * (1ll << min(d, 38));
            } else if (-d > 38) {
                next = th;
            } else {
                const int s = -d;
                const long long v = th * (1ll << s) - u;
                if (!stochastic) {
                    next = rne_shr64(v, s);
                } else {
                    const unsigned long long r = rounding_bits(key, j) & ((1ull << s) - 1ull);
                    next = (v + (long long)r) >> s;
                }
            }
            next = next < -lim_m ? -lim_m : (next > lim_m ? lim_m : next);
            T.master[j] = (int32_t)next;
            const long long w8 = rne_shr64(next, k_m - 8);
            T.w[j] = (int8_t)(w8 < -127 ? -127 : (w8 > 127 ? 127 : w8));
        }
    } else if (threadIdx.x == 0 && (int)blockIdx.x == b.first_block[k]) {
        atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
    }
    if (last) {
        for (int i = 0; i < b.num; ++i) dev->tensor_absmax[b.tensor_base + i] = 0;
        if (b.last && step_dev) *step_dev = step_s + 1ull;
    }
}

// The tensors [base, base + kUpdChunk) of a call as one launch's batch; returns its block count.
// `first`: index of t[0] in the list that the rounding counts by; `last`: the call ends a step.
int fill_batch(UpdateBatch &b, const UpdateTensor *t, int num, int base, int first, bool last)
{
    b.num = num - base < kUpdChunk ? num - base : kUpdChunk;
    b.tensor_base = first + base;
    b.last = last && base + b.num == num;
    int blocks = 0;
    for (int k = 0; k < b.num; ++k) {
        b.t[k] = t[base + k];
        b.first_block[k] = blocks;
        blocks += (int)((t[base + k].n + kUpdElemsPerBlock - 1) / kUpdElemsPerBlock);
    }
    b.first_block[b.num] = blocks;
    return blocks;
}

}  // namespace

int update_launches(const UpdateTensor *t, int num, bool wide)
{
    const int chunks = (num + kUpdChunk - 1) / kUpdChunk;
    for (int i = 0; i < num && !wide; ++i) wide = t[i].n > kSmallElems;
    return wide ? 2 * chunks : chunks;
}

cudaError_t launch_update(const UpdateTensor *t, int num, int32_t lr_mant, int32_t lr_exp, int stochastic, uint64_t seed,
                          uint64_t step, unsigned long long *step_dev, DeviceState *dev, cudaStream_t s, int first, bool last)
{
    const int chunks = (num + kUpdChunk - 1) / kUpdChunk;
    const bool small = update_launches(t, num, false) == chunks;
    int parts = 1;
    for (int i = 0; i < num; ++i)
        if (stochastic && t[i].n > kSmallPart) parts = kSmallMostParts;   // (the hash is what takes the time)
    const int threads = parts > 1 ? kSmallPartThreads : kSmallThreads;
    UpdateBatch b;
    if (!small)
        for (int base = 0; base < num; base += kUpdChunk) {
            const int blocks = fill_batch(b, t, num, base, first, last);
            launch_chained(update_absmax_kernel, blocks, kThreads, 0, s, b, dev);
        }
    for (int base = 0; base < num; base += kUpdChunk) {
        const int blocks = fill_batch(b, t, num, base, first, last);
        if (small) launch_chained_clusters(parts, update_small_kernel, b.num * parts, threads, 0, s, b, parts, lr_mant, lr_exp, stochastic, seed, step, step_dev, dev);
        else launch_chained(update_apply_kernel, blocks, kThreads, 0, s, b, lr_mant, lr_exp, stochastic, seed, step, step_dev, dev);
    }
    return cudaGetLastError();
}

cudaError_t launch_update_wide(const UpdateTensor *t, int num, int32_t lr_mant, int32_t lr_exp, int k_u, int k_m, int stochastic,
                               uint64_t seed, uint64_t step, unsigned long long *step_dev, DeviceState *dev, cudaStream_t s)
{
    UpdateBatch b;
    for (int pass = 0; pass < 2; ++pass)
        for (int base = 0; base < num; base += kUpdChunk) {
            const int blocks = fill_batch(b, t, num, base, 0, true);
            if (pass == 0) launch_chained(update_absmax_kernel, blocks, kThreads, 0, s, b, dev);
            else launch_chained(update_wide_apply_kernel, blocks, kThreads, 0, s, b, lr_mant, lr_exp, k_u, k_m, stochastic, seed, step, step_dev, dev);
        }
    return cudaGetLastError();
}

}  // namespace eoq
