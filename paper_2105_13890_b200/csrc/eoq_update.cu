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
constexpr size_t kSmallPart = 8192;
constexpr int kSmallMostParts = 8;
constexpr size_t kSmallElems = (size_t)kSmallThreads * kSmallGroups * 16;

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
// with packed 16-bit ones.
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
            for (size_t i = begin + (size_t)threadIdx.x * 16; i + 16 <= end; i += (size_t)kThreads * 16)
                am.add(__ldg(reinterpret_cast<const int4 *>(T.g + i)));
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
    int mul, sh, half_m1;  // u = sat(R(mul * g / 2^sh))
    int d;                 // exponent of u relative to the weight grid 2^-7: w - u * 2^d
    unsigned long long key;
};

__device__ __forceinline__ UpdateRule update_rule(uint32_t M, int g_exp, int lr_mant, int lr_exp, int stochastic, unsigned long long seed,
                                                  unsigned long long step, int tensor)
{
    UpdateRule r;
    const int t = round_log2_u32(M);
    r.mul = t < 7 ? lr_mant << (7 - t) : lr_mant;
    r.sh = t < 7 ? 0 : t - 7;
    r.half_m1 = r.sh ? (1 << (r.sh - 1)) - 1 : 0;
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

// One code; z: the element's hash counter key + (index + 1) * golden (stochastic modes).  The result still needs the
// upper clamp at 127 (the packing saturates there); the lower one at -127 is applied here.
template <UpdateMode kMode>
__device__ __forceinline__ int update_code(int w, int g, const UpdateRule &r, unsigned long long z)
{
    if (kMode == kKeep) return max(w, -127);
    int u = r.mul * g;
    if (r.sh) u = (u + r.half_m1 + ((u >> r.sh) & 1)) >> r.sh;
    u = clampi(u, -127, 127);
    int next;
    if (kMode == kShiftUp) {
        next = w - u * (1 << min(r.d, 9));  // any |u| * 2^9 saturates, as any larger power would
    } else if (kMode == kNearest) {
        const int s = -r.d, v = w * (1 << s) - u;
        next = (v + ((1 << (s - 1)) - 1) + ((v >> s) & 1)) >> s;
    } else if (kMode == kStochastic) {
        // floor((w 2^s - u + rand) / 2^s) = w + floor((rand - u) / 2^s)
        const int s = -r.d;
        next = w + (((int)((uint32_t)mix64(z) & ((1u << s) - 1u)) - u) >> s);
    } else {
        const int s = -r.d;
        next = w + (int)(((long long)(mix64(z) & ((1ull << s) - 1ull)) - u) >> s);
    }
    return max(next, -127);
}

template <UpdateMode kMode>
__device__ __forceinline__ int4 update_16(const int4 &wv, const int4 &gv, const UpdateRule &r, size_t i)
{
    const uint32_t ww[4] = {(uint32_t)wv.x, (uint32_t)wv.y, (uint32_t)wv.z, (uint32_t)wv.w};
    const uint32_t gw[4] = {(uint32_t)gv.x, (uint32_t)gv.y, (uint32_t)gv.z, (uint32_t)gv.w};
    uint32_t o[4];
    unsigned long long z = r.key + kGolden * ((unsigned long long)i + 1);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int c[4];
#pragma unroll
        for (int k = 0; k < 4; ++k, z += kGolden)
            c[k] = update_code<kMode>((int)(int8_t)(ww[q] >> (8 * k)), (int)(int8_t)(gw[q] >> (8 * k)), r, z);
        o[q] = pack4_sat(c[0], c[1], c[2], c[3]);
    }
    return make_int4((int)o[0], (int)o[1], (int)o[2], (int)o[3]);
}

// elements [begin, end) of one tensor by the calling block
template <UpdateMode kMode>
__device__ __forceinline__ void update_range(const UpdateTensor &T, size_t begin, size_t end, const UpdateRule &r)
{
    const bool vec = ((reinterpret_cast<uintptr_t>(T.g) | reinterpret_cast<uintptr_t>(T.w)) & 15) == 0;
    if (vec)
        for (size_t i = begin + (size_t)threadIdx.x * 16; i + 16 <= end; i += (size_t)blockDim.x * 16) {
            const int4 gv = kMode == kKeep ? make_int4(0, 0, 0, 0) : __ldg(reinterpret_cast<const int4 *>(T.g + i));
            const int4 wv = *reinterpret_cast<const int4 *>(T.w + i);
            *reinterpret_cast<int4 *>(T.w + i) = update_16<kMode>(wv, gv, r, i);
        }
    const size_t tail = vec ? begin + ((end - begin) / 16) * 16 : begin;
    for (size_t j = tail + threadIdx.x; j < end; j += blockDim.x)
        T.w[j] = (int8_t)min(update_code<kMode>(T.w[j], T.g[j], r, r.key + kGolden * ((unsigned long long)j + 1)), 127);
}

__device__ __forceinline__ void update_range(UpdateMode mode, const UpdateTensor &T, size_t begin, size_t end, const UpdateRule &r)
{
    switch (mode) {
        case kShiftUp: update_range<kShiftUp>(T, begin, end, r); break;
        case kNearest: update_range<kNearest>(T, begin, end, r); break;
        case kKeep: update_range<kKeep>(T, begin, end, r); break;
        case kStochastic: update_range<kStochastic>(T, begin, end, r); break;
        default: update_range<kStochasticWide>(T, begin, end, r); break;
    }
}

// w <- Q_w(w - Q_u(lr * g)).  Bound by the integer pipe under stochastic rounding: 43 instructions a weight, most of them the 64-bit
// hash's, 24 of which go to the pipe that takes one every two cycles and scheduler: 27.5 of the 37 us that the 21 M weights of
// ResNet-34 take (the pipe is 79% busy while an SM has work).  Rounding to nearest takes 14 instructions and 15 us; its largest stall
// is that of its loads.  Every rounding mode is a loop of its own on 32-bit values: one 64-bit sequence for all modes took 58 us.
__global__ void __launch_bounds__(kThreads)
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
    const uint32_t M = max_s * (uint32_t)lr_mant;  // max |lr_mant * g| < 2^15
    if (M != 0) {
        const UpdateRule r = update_rule(M, g_exp, lr_mant, lr_exp, stochastic, seed, step_s, b.tensor_base + k);
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
            const size_t i = begin + ((size_t)q * kSmallThreads + threadIdx.x) * 16;
            if (i + 16 <= end) am.add(__ldg(reinterpret_cast<const int4 *>(T.g + i)));
        }
    }
    uint32_t mx = am.value();
    for (size_t j = (vec ? begin + (end - begin) / 16 * 16 : begin) + threadIdx.x; j < end; j += kSmallThreads)
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
    const uint32_t M = mx * (uint32_t)lr_mant;
    if (M != 0) {
        const UpdateRule r = update_rule(M, g_exp, lr_mant, lr_exp, stochastic, seed, step_s, b.tensor_base + k);
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
    UpdateBatch b;
    if (!small)
        for (int base = 0; base < num; base += kUpdChunk) {
            const int blocks = fill_batch(b, t, num, base, first, last);
            launch_chained(update_absmax_kernel, blocks, kThreads, 0, s, b, dev);
        }
    for (int base = 0; base < num; base += kUpdChunk) {
        const int blocks = fill_batch(b, t, num, base, first, last);
        if (small) launch_chained_clusters(parts, update_small_kernel, b.num * parts, kSmallThreads, 0, s, b, parts, lr_mant, lr_exp, stochastic, seed, step, step_dev, dev);
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
