// Bandwidth-bound kernels of the EOQ layer (arXiv 2105.13890): the standalone quantizers Q / CQ / SQ
// (Sec. 3.2.2), the second phase of the scale quantizer after a convolution, the head of the error
// chain (Sec. 3.2.1) and small layout helpers.
// Reductions run warp-shuffle -> shared memory -> one atomic per block; 16 elements per thread with 128-bit accesses.
#include <algorithm>
#include <cooperative_groups.h>

#include "eoq_cells.cuh"
#include "eoq_device.cuh"
#include "eoq_epilogue.cuh"
#include "eoq_internal.h"
#include "eoq_next_head.cuh"

namespace eoq {

namespace {

constexpr int kThreads = 256;

inline int grid_for(size_t work_items, int sm_count, int per_sm = 8)
{
    size_t blocks = (work_items + kThreads - 1) / kThreads;
    size_t cap = (size_t)sm_count * per_sm;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

// ------------------------------------------------------------------ fp32 -> Q / CQ / SQ

// x * 2^up, exact wherever the code depends on it (a result too small for a normal number codes to 0 either way).
// 2^up itself may exceed the float range for a tensor of subnormal size, hence two factors.
struct Pow2Scale {
    float f1, f2;
    // nearest, ties to even; NaN gives 0 and an infinity the largest or smallest int, as the conversion defines
    __device__ __forceinline__ int code(float x) const { return __float2int_rn(__fmul_rn(__fmul_rn(x, f1), f2)); }
};
__device__ __forceinline__ Pow2Scale pow2_scale(int up)
{
    return Pow2Scale{__int_as_float((clampi(up, -126, 127) + 127) << 23), up > 127 ? __int_as_float(up << 23) : 1.0f};
}

// Shift of SQ under the maximum `mbits` (bit pattern of max |x|): codes = R(x * 2^up), exponent -up.
__device__ __forceinline__ int sq_up(uint32_t mbits) { return (mbits != 0 && mbits < 0x7f800000u) ? 7 - round_log2_f32bits(mbits) : 7; }

template <int kMode>
__device__ __forceinline__ int quantize_code(const Pow2Scale &sc, float x)
{
    return clampi(sc.code(x), kMode == 0 ? -32768 : -127, kMode == 0 ? 32767 : 127);
}

// four codes at element index 4 i
template <int kMode>
__device__ __forceinline__ void quantize_store4(void *dst, size_t i, const Pow2Scale &sc, const float4 &v)
{
    const int a = quantize_code<kMode>(sc, v.x), b = quantize_code<kMode>(sc, v.y), c = quantize_code<kMode>(sc, v.z),
              d = quantize_code<kMode>(sc, v.w);
    if (kMode == 0) reinterpret_cast<uint2 *>(dst)[i] = make_uint2((a & 0xffff) | (b << 16), (c & 0xffff) | (d << 16));
    else reinterpret_cast<uint32_t *>(dst)[i] = pack4_sat(a, b, c, d);
}

__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t max_abs(uint32_t mx, const float4 &v)
{
    return max(max(mx, max(abs_bits(v.x), abs_bits(v.y))), max(abs_bits(v.z), abs_bits(v.w)));
}

// A block takes one tile of kQuantTile float4, eight independent, coalesced loads per thread.
constexpr int kQuantLoads = 8, kQuantTile = kThreads * kQuantLoads;
__device__ __forceinline__ void load_tile(const float *__restrict__ src, size_t n4, size_t tile, float4 (&v)[kQuantLoads])
{
#pragma unroll
    for (int u = 0; u < kQuantLoads; ++u) {
        const size_t i = tile * kQuantTile + (size_t)u * kThreads + threadIdx.x;
        v[u] = i < n4 ? __ldg(reinterpret_cast<const float4 *>(src) + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// ------------------------------------------------------------------ SQ of a tensor beyond one cluster, and of images
// Two passes: the maximum, then the codes, the second read out of the L2.  Whole tiles of loads are in flight in both, and the second
// pass's blocks read theirs while the first pass ends.  Floats from memory, what a row of calls on other tensors takes each: 1 M 4.8 us, 4 M
// 7.2, 8 M 12.6 (of one tensor again and again 4.0, 5.7 and 8.3).  A pass for the maximum with one load of a thread in flight: 5.6, 9.3 and
// 16.0.  Codes formed in the first pass under a guess, and again where the guess was wrong: 5.0, 8.8 and 13.3 where it never is, 6.2, 10.9
// and 15.3 under one element beyond all others; 64 images 224 x 224 18.5 and 25.9, so 19.9 whatever they hold.

// First pass: the largest |x|.  Bound by memory (4 B in).
__global__ void __launch_bounds__(kThreads) absmax_f32_kernel(const float *__restrict__ src, size_t n, DeviceState *dev)
{
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    float4 v[kQuantLoads];
    load_tile(src, n / 4, blockIdx.x, v);
    uint32_t mx = 0;
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) mx = abs_bits(src[n / 4 * 4 + threadIdx.x]);
#pragma unroll
    for (int u = 0; u < kQuantLoads; ++u) mx = max_abs(mx, v[u]);
    mx = block_max_u32(mx);
    if (threadIdx.x == 0) {
        if (mx) atomicMax(&dev->absmax_u32, mx);
        if (mx >= 0x7f800000u) atomicOr(&dev->status, EOQ_DEV_NONFINITE);
    }
}

// What a block of SQ's second pass does with the maximum once its operands are on their way: the shift, and the exponent (one block).
// All threads; `tid` in the block.  True in one thread of the grid, which clears the cell when its block is done.
__device__ __forceinline__ bool sq_shift(int tid, int32_t *dst_exp, DeviceState *dev, int *up)
{
    __shared__ uint32_t max_s;
    if (tid == 0) max_s = *reinterpret_cast<volatile uint32_t *>(&dev->absmax_u32);
    __syncthreads();
    *up = sq_up(max_s);
    if (tid != 0) return false;
    if (blockIdx.x == 0) {
        *dst_exp = -*up;
        if (max_s == 0) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
    }
    return last_reader(dev);
}

// Codes of a tile whose values are at hand, kMode 0: Q -> int16, 1: CQ -> int8, 2: SQ -> int8; block 0 also those of the up to three
// elements behind the last float4.
template <int kMode>
__device__ __forceinline__ void store_tile(void *dst, const float *src, size_t n, size_t tile, const Pow2Scale &sc, const float4 (&v)[kQuantLoads])
{
    const size_t n4 = n / 4;
#pragma unroll
    for (int u = 0; u < kQuantLoads; ++u) {
        const size_t i = tile * kQuantTile + (size_t)u * kThreads + threadIdx.x;
        if (i < n4) quantize_store4<kMode>(dst, i, sc, v[u]);
    }
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) {
        const size_t i = n4 * 4 + threadIdx.x;
        const int c = quantize_code<kMode>(sc, src[i]);
        if (kMode == 0) reinterpret_cast<int16_t *>(dst)[i] = (int16_t)c;
        else reinterpret_cast<int8_t *>(dst)[i] = (int8_t)c;
    }
}

// Q and CQ.  Bound by memory: 4 B in, 1 or 2 B out; up to some 2 M floats by the rate of launches: 3.0 us a call in a row of calls, 3.4 as
// instances of SQ's second pass, with its two more parameters and a wait that goes by one of them.
template <int kMode>
__global__ void __launch_bounds__(kThreads) quantize_f32_kernel(const float *__restrict__ src, size_t n, void *dst, int32_t *dst_exp)
{
    ptx::grid_dep_wait_launch_small();
    float4 v[kQuantLoads];
    load_tile(src, n / 4, blockIdx.x, v);
    constexpr int up = 7;
    if (blockIdx.x == 0 && threadIdx.x == 0 && dst_exp) *dst_exp = -up;
    store_tile<kMode>(dst, src, n, blockIdx.x, pow2_scale(up), v);
}

// SQ under the reduced maximum (tiles backwards: the first pass read the last ones last).  Bound by memory: 4 B in, from L2 where it holds
// the tensor, 1 B out.
// early: the first pass is the launch in front and lets this one in once the source is complete, so its tiles are read ahead of the wait.
__global__ void __launch_bounds__(kThreads)
quantize_sq_second_kernel(const float *__restrict__ src, size_t n, int8_t *dst, int32_t *dst_exp, DeviceState *dev, int early)
{
    const size_t tile = gridDim.x - 1 - blockIdx.x;
    if (!early) ptx::grid_dep_wait_launch_small();
    float4 v[kQuantLoads];
    load_tile(src, n / 4, tile, v);
    if (early) ptx::grid_dep_wait_launch_small();
    int up;
    const bool last = sq_shift(threadIdx.x, dst_exp, dev, &up);
    store_tile<2>(dst, src, n, tile, pow2_scale(up), v);
    if (last) dev->absmax_u32 = 0;
}

// ------------------------------------------------------------------ SQ of a tensor much of which a second read takes from memory
// The codes depend on the tensor's maximum through R(log2 max) alone, and a tile of a few thousand elements often has the tensor's
// R(log2 max) already.  So the first pass codes every tile under the larger of its own maximum and what other blocks have reduced by
// then, and leaves the shift it used; the second pass, under the whole maximum, codes again the tiles whose shift was another one, and
// returns where there are none.  Bound by memory; times at kSqResident.

// shift of a tile: what its codes were formed under, or one of
constexpr int kTileAny = 0x7fff;     // all of it is zero: codes 0 under any shift
constexpr int kTileMixed = 0x7ffe;   // parts under different shifts
constexpr int kAgainPerSm = 5;       // blocks of the second pass on an SM

// The block's guess for one part of its tile (all threads, `tid` in the block; one barrier): `mx` is the thread's maximum.
struct TileGuess {
    uint32_t own = 0;        // largest |x| of the tile so far (bit pattern)
    int shift = kTileAny;    // of the tile so far
    int turn = 0;
    __device__ __forceinline__ int part(uint32_t mx, int tid, DeviceState *dev)
    {
        __shared__ __align__(16) uint32_t warp_s[2][kThreads / 32];
        __shared__ uint32_t seen_s;
        uint32_t *w = warp_s[turn & 1];
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (turn == 0 && tid == 0) seen_s = *reinterpret_cast<volatile uint32_t *>(&dev->absmax_u32);
        if ((tid & 31) == 0) w[tid >> 5] = mx;
        __syncthreads();
        uint32_t m = 0;
#pragma unroll
        for (int i = 0; i < kThreads / 32; ++i) m = max(m, w[i]);
        own = max(own, m);
        const int up = sq_up(max(own, seen_s));
        if (m) shift = shift == kTileAny || shift == up ? up : kTileMixed;
        ++turn;
        return up;
    }
    __device__ __forceinline__ void publish(int tid, int16_t *tile_shift, DeviceState *dev) const
    {
        if (tid != 0) return;
        *tile_shift = (int16_t)shift;
        if (own) atomicMax(&dev->absmax_u32, own);
        if (own >= 0x7f800000u) atomicOr(&dev->status, EOQ_DEV_NONFINITE);
    }
};

// Second pass: calls again(tile, scale) in all threads of a block for those of its tiles that need it; tiles are dealt out from the
// tensor's end, which the first pass read last.  Thread 0 of block 0 writes the exponent.
template <typename Again>
__device__ __forceinline__ void recode_tiles(const int16_t *tile_shift, int tiles, int tid, int32_t *dst_exp, DeviceState *dev, Again again)
{
    __shared__ uint32_t max_s;
    __shared__ uint8_t wrong_s[kThreads];
    bool last = false;
    if (tid == 0) max_s = *reinterpret_cast<volatile uint32_t *>(&dev->absmax_u32);
    for (int first = blockIdx.x; first < tiles; first += gridDim.x * kThreads) {   // (one round)
        const int t = first + tid * (int)gridDim.x, used = t < tiles ? tile_shift[tiles - 1 - t] : kTileAny;
        __syncthreads();
        const int up = sq_up(max_s);
        const bool wrong = used != kTileAny && used != up;
        wrong_s[tid] = wrong;
        if (first == (int)blockIdx.x && tid == 0) {
            last = last_reader(dev);
            if (blockIdx.x == 0) {
                *dst_exp = -up;
                if (max_s == 0) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
            }
        }
        if (!__syncthreads_or(wrong)) continue;
        const Pow2Scale sc = pow2_scale(up);
        for (int k = 0, t = first; k < kThreads && t < tiles; ++k, t += gridDim.x)
            if (wrong_s[k]) again(tiles - 1 - t, sc);
    }
    if (last) dev->absmax_u32 = 0;
}

// Part `p` of the tensor is a tile of load_tile; a tile here is `reps` of them.
__device__ __forceinline__ void store_part(int8_t *dst, size_t n4, size_t p, const Pow2Scale &sc, const float4 (&v)[kQuantLoads])
{
#pragma unroll
    for (int u = 0; u < kQuantLoads; ++u) {
        const size_t i = p * kQuantTile + (size_t)u * kThreads + threadIdx.x;
        if (i < n4) quantize_store4<2>(dst, i, sc, v[u]);
    }
}

__global__ void __launch_bounds__(kThreads)
quantize_sq_kernel(const float *__restrict__ src, size_t n, int8_t *dst, int16_t *tile_shift, int reps, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    const size_t n4 = n / 4;
    TileGuess guess;
    for (int r = 0; r < reps; ++r) {
        const size_t p = (size_t)blockIdx.x * reps + r;
        float4 v[kQuantLoads];
        load_tile(src, n4, p, v);
        uint32_t mx = 0;
        // (the up to three elements behind the last float4 are coded by the second pass)
        if (blockIdx.x == 0 && r == 0 && threadIdx.x < (n & 3)) mx = abs_bits(src[n4 * 4 + threadIdx.x]);
#pragma unroll
        for (int u = 0; u < kQuantLoads; ++u) mx = max_abs(mx, v[u]);
        store_part(dst, n4, p, pow2_scale(guess.part(mx, threadIdx.x, dev)), v);
    }
    guess.publish(threadIdx.x, tile_shift + blockIdx.x, dev);
}

__global__ void __launch_bounds__(kThreads, kAgainPerSm)
quantize_sq_again_kernel(const float *__restrict__ src, size_t n, int8_t *dst, int32_t *dst_exp, const int16_t *tile_shift, int tiles, int reps,
                         DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    const size_t n4 = n / 4;
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) {
        const size_t i = n4 * 4 + threadIdx.x;
        dst[i] = (int8_t)quantize_code<2>(pow2_scale(sq_up(*reinterpret_cast<volatile uint32_t *>(&dev->absmax_u32))), src[i]);
    }
    recode_tiles(tile_shift, tiles, threadIdx.x, dst_exp, dev, [&](int tile, const Pow2Scale &sc) {
        for (int r = 0; r < reps; ++r) {
            float4 v[kQuantLoads];
            load_tile(src, n4, (size_t)tile * reps + r, v);
            store_part(dst, n4, (size_t)tile * reps + r, sc, v);
        }
    });
}

// SQ in one launch for tensors that one cluster can hold in registers (kSmallElems codes per block, up to
// kSmallCluster blocks): every block reduces its part, the maxima meet in distributed shared memory, no cell and no
// second read is needed.  Bound by latency.
constexpr int kSmallThreads = 1024, kSmallLoads = 8, kSmallCluster = 8;
constexpr size_t kSmallElems = (size_t)kSmallThreads * kSmallLoads * 4;
__global__ void __launch_bounds__(kSmallThreads)
quantize_sq_small_kernel(const float *__restrict__ src, size_t n, int8_t *dst, int32_t *dst_exp, DeviceState *dev)
{
    namespace cg = cooperative_groups;
    __shared__ uint32_t max_s;
    cg::cluster_group cluster = cg::this_cluster();
    const size_t n4 = n / 4, base = (size_t)blockIdx.x * kSmallThreads + threadIdx.x, step = (size_t)gridDim.x * kSmallThreads;
    float4 v[kSmallLoads];
    uint32_t mx = 0;
#pragma unroll
    for (int u = 0; u < kSmallLoads; ++u) {
        const size_t i = base + u * step;
        v[u] = i < n4 ? __ldg(reinterpret_cast<const float4 *>(src) + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float tail = 0.0f;
    const size_t ti = n4 * 4 + threadIdx.x;
    if (blockIdx.x == 0 && ti < n) tail = src[ti];
#pragma unroll
    for (int u = 0; u < kSmallLoads; ++u)
        mx = max(max(mx, max(__float_as_uint(v[u].x) & 0x7fffffffu, __float_as_uint(v[u].y) & 0x7fffffffu)),
                 max(__float_as_uint(v[u].z) & 0x7fffffffu, __float_as_uint(v[u].w) & 0x7fffffffu));
    mx = max(mx, __float_as_uint(tail) & 0x7fffffffu);
    mx = block_max_u32(mx);
    if (threadIdx.x == 0) max_s = mx;
    cluster.sync();
    mx = 0;
    for (unsigned r = 0; r < gridDim.x; ++r) mx = max(mx, *cluster.map_shared_rank(&max_s, r));
    const int up = sq_up(mx);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *dst_exp = -up;
        if (mx == 0) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
        if (mx >= 0x7f800000u) atomicOr(&dev->status, EOQ_DEV_NONFINITE);
    }
    const Pow2Scale sc = pow2_scale(up);
#pragma unroll
    for (int u = 0; u < kSmallLoads; ++u) {
        const size_t i = base + u * step;
        if (i < n4) quantize_store4<2>(dst, i, sc, v[u]);
    }
    if (blockIdx.x == 0 && ti < n) dst[ti] = (int8_t)quantize_code<2>(sc, tail);
    cluster.sync();  // no block leaves while another may still read its maximum
}

// SQ of an fp32 image under the reduced maximum: c_src channels in, c_dst (zero-padded) channels out, rows widened by `wmargin` zero
// pixels at both ends.  A thread writes kG = 16 or 8 channels of a pixel.  Bound by memory (12 B in, 8 or 16 B out per RGB pixel).  A block is
// tx pixels x ty rows and a thread takes its pixel in kImageRows rows, all loads issued before the maximum is needed, no divisions.
constexpr int kImageRows = 4;
struct ImageShape {
    int rows, w, c_src, c_dst, wmargin;
};
// 16 or 8 codes of an output pixel from the values of its channels (`more`: those beyond the first four, read here)
template <int kG>
__device__ __forceinline__ void image_store(int8_t *dst, size_t o, const Pow2Scale &sc, const float (&v)[4], const float *more, int nch)
{
    int c[kG];
#pragma unroll
    for (int k = 0; k < kG; ++k) c[k] = k < 4 ? quantize_code<2>(sc, v[k & 3]) : (more && k < nch ? quantize_code<2>(sc, __ldg(more + k)) : 0);
    if (kG == 16)
        reinterpret_cast<uint4 *>(dst)[o] = make_uint4(pack4_sat(c[0], c[1], c[2], c[3]), pack4_sat(c[4], c[5], c[6], c[7]),
                                                       pack4_sat(c[8 % kG], c[9 % kG], c[10 % kG], c[11 % kG]),
                                                       pack4_sat(c[12 % kG], c[13 % kG], c[14 % kG], c[15 % kG]));
    else
        reinterpret_cast<uint2 *>(dst)[o] = make_uint2(pack4_sat(c[0], c[1], c[2], c[3]), pack4_sat(c[4], c[5], c[6], c[7]));
}

// kStaged: images of up to four channels in one group, no row wider than the block: a block's rows are then a run of at most 4 * kThreads
// pixels, read as float4 and handed out through shared memory.
template <int kG, bool kStaged>
__global__ void __launch_bounds__(kThreads)
quantize_image_kernel(const float *__restrict__ src, ImageShape s, int8_t *dst, int32_t *dst_exp, DeviceState *dev, int early)
{
    if (!early) ptx::grid_dep_wait_launch_small();   // (see quantize_sq_second_kernel)
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, block = (int)(gridDim.x - 1 - blockIdx.x);
    const int row0 = block * kImageRows * (int)blockDim.y, w_mem = s.w + 2 * s.wmargin;
    int up = 7;
    bool last = false;
    if (kStaged) {
        __shared__ __align__(16) float stage[4 * kImageRows * kThreads];
        const int rows = min(kImageRows * (int)blockDim.y, s.rows - row0), count = rows * s.w * s.c_src;
        const float *p = src + (size_t)row0 * s.w * s.c_src;   // (16-byte aligned: row0 is a multiple of 4)
        float4 v[kImageRows];
#pragma unroll
        for (int u = 0; u < kImageRows; ++u) {
            const int i = u * kThreads + tid;
            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (4 * i + 3 < count) v[u] = __ldg(reinterpret_cast<const float4 *>(p) + i);
            else if (4 * i < count) {
                v[u].x = __ldg(p + 4 * i);
                if (4 * i + 1 < count) v[u].y = __ldg(p + 4 * i + 1);
                if (4 * i + 2 < count) v[u].z = __ldg(p + 4 * i + 2);
            }
        }
        if (early) ptx::grid_dep_wait_launch_small();
#pragma unroll
        for (int u = 0; u < kImageRows; ++u) reinterpret_cast<float4 *>(stage)[u * kThreads + tid] = v[u];
        last = sq_shift(tid, dst_exp, dev, &up);   // (its barrier also publishes the stage)
        const Pow2Scale sc = pow2_scale(up);
        const int xm = (int)threadIdx.x - s.wmargin;
        const bool in = xm >= 0 && xm < s.w;
#pragma unroll
        for (int u = 0; u < kImageRows; ++u) {
            const int r = threadIdx.y + u * blockDim.y;
            if ((int)threadIdx.x >= w_mem || r >= rows) continue;
            const float *q = stage + (r * s.w + xm) * s.c_src;
            float f[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) f[k] = in && k < s.c_src ? q[k] : 0.0f;
            image_store<kG>(dst, (size_t)(row0 + r) * w_mem + threadIdx.x, sc, f, nullptr, 0);
        }
    } else {
        const int groups = s.c_dst / kG, items = w_mem * groups;
        for (int x0 = 0; x0 < items; x0 += blockDim.x) {   // one round unless a row is wider than the block
            const int it = x0 + threadIdx.x;
            const int xp = groups == 1 ? it : it / groups, g = groups == 1 ? 0 : it - xp * groups, xm = xp - s.wmargin;
            const int nch = min(kG, s.c_src - g * kG);       // real channels of this group (none or fewer beyond c_src)
            const bool in = it < items && xm >= 0 && xm < s.w;
            float v[kImageRows][4];                          // the first four channels; more are read when they are coded
#pragma unroll
            for (int u = 0; u < kImageRows; ++u) {
                const int row = row0 + threadIdx.y + u * blockDim.y;
                const float *p = src + ((size_t)row * s.w + xm) * s.c_src + g * kG;
#pragma unroll
                for (int k = 0; k < 4; ++k) v[u][k] = (in && row < s.rows && k < nch) ? __ldg(p + k) : 0.0f;
            }
            if (x0 == 0) {
                if (early) ptx::grid_dep_wait_launch_small();
                last = sq_shift(tid, dst_exp, dev, &up);
            }
            const Pow2Scale sc = pow2_scale(up);
#pragma unroll
            for (int u = 0; u < kImageRows; ++u) {
                const int row = row0 + threadIdx.y + u * blockDim.y;
                if (it >= items || row >= s.rows) continue;
                image_store<kG>(dst, (size_t)row * items + it, sc, v[u], in && nch > 4 ? src + ((size_t)row * s.w + xm) * s.c_src + g * kG : nullptr, nch);
            }
        }
    }
    if (last) dev->absmax_u32 = 0;
}

// w[oc][kh][kw][c] -> wp[oc][kh][8][c] with zeros in the unused taps; c = 16 (Pixel = int4) or 8 (int2)
template <typename Pixel>
__global__ void weight_pad_rows_kernel(const int8_t *__restrict__ w, int8_t *__restrict__ wp, int rows, int kw)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;  // one pixel of the padded layout
    if (i >= rows * 8) return;
    const int r = i >> 3, t = i & 7;
    Pixel v = Pixel();
    if (t < kw) v = __ldg(reinterpret_cast<const Pixel *>(w) + (size_t)r * kw + t);
    reinterpret_cast<Pixel *>(wp)[i] = v;
}

// ------------------------------------------------------------------ int32 -> SQ (phase 2 of Q_e after dgrad)

__global__ void absmax_i32_kernel(const int32_t *__restrict__ src, size_t n, DeviceState *dev)
{
    uint32_t mx = 0;
    const size_t n4 = n / 4;
    const int4 *s4 = reinterpret_cast<const int4 *>(src);
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        int4 v = __ldg(s4 + i);
        mx = max(max(mx, (uint32_t)abs(v.x)), max((uint32_t)abs(v.y), max((uint32_t)abs(v.z), (uint32_t)abs(v.w))));
    }
    for (size_t i = n4 * 4 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        mx = max(mx, (uint32_t)abs(src[i]));
    mx = (uint32_t)block_max_u64(mx);
    if (threadIdx.x == 0 && mx) atomicMax(&dev->absmax_u32, mx);
}

// One 256-bit streaming load (sm_100); ptr must be 32-byte aligned.
__device__ __forceinline__ void ld_global_256_stream(const void *ptr, uint32_t *v)
{
    asm volatile("ld.global.cs.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(ptr));
}

// kNext: the error head of the layer that consumes dst rides along (see NextHead): the masked maximum sits in the
// handle's 64-bit cell (the GEMM epilogue reduced it beside the plain one), so the codes of e3 and the head's sums
// come out of the same pass.  n must then be a multiple of 16.
// kJoin: dst is the first operand of an error join; the join's first pass rides along: max |dst * 2^sa + b * 2^sb|
// over all positions (64-bit cell) and over those the consumer's ReLU lets through (second 64-bit cell).
// kPacked: src holds the sums of an error back-propagation as 16-bit words (sums_pack_16; 32-byte aligned, n a multiple of 16);
// int32 otherwise.
template <bool kPacked, bool kNext, bool kJoin>
__global__ void sq_i32_kernel(const void *__restrict__ src_any, const int32_t *src_exp, int exp_bias, size_t n,
                              int8_t *dst, int32_t *dst_exp, long long *sum_codes, NextHeadArgs next, JoinStatArgs join,
                              DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    // The maxima go through one thread per block and shared memory; that thread counts the block as a reader, and the last
    // one puts the cells back to zero at its end.  The sums are added to where the caller wants them (cleared by the kernel
    // in front): with a ticket, a fence and the publication of the sums by the last block, these kernels took about 2 us more
    // on the few hundred KB of a small batch.
    __shared__ uint32_t cell_s[2];
    const size_t n16 = n / 16;
    const int32_t *const src = static_cast<const int32_t *>(src_any);
    // a group of 16 sums, and what a join wants beside it
    struct Group {
        uint32_t raw[kPacked ? 8 : 16];
        int4 b;
        uint32_t gate, nm;
    } cur = {};
    const bool wide_in = (reinterpret_cast<uintptr_t>(src) & 31) == 0;
    auto load16 = [&](size_t i, Group &to) {
        if constexpr (kPacked) {
            ld_global_256_stream(static_cast<const uint16_t *>(src_any) + i * 16, to.raw);
        } else if (wide_in) {   // two 256-bit loads: whole 32-byte sectors per lane
            ld_global_256_stream(src + i * 16, to.raw);
            ld_global_256_stream(src + i * 16 + 8, to.raw + 8);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int4 v = __ldcs(reinterpret_cast<const int4 *>(src) + i * 4 + k);
                to.raw[4 * k + 0] = v.x;
                to.raw[4 * k + 1] = v.y;
                to.raw[4 * k + 2] = v.z;
                to.raw[4 * k + 3] = v.w;
            }
        }
        if (kJoin) {
            to.b = __ldg(reinterpret_cast<const int4 *>(join.b) + i);
            to.gate = join.mask_b ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(join.mask_b) + i) : 0xffffu;
            to.nm = join.next_mask ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(join.next_mask) + i) : 0u;
        }
        if (kNext) to.nm = (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(next.mask) + i);
    };
    // the first group of every thread is on its way while the maxima are read
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n16) {
        load16(i, cur);
        if (kNext && next.x2) ptx::prefetch_l1(next.x2 + i * 16);
    }
    bool last = false;
    if (threadIdx.x == 0) {
        cell_s[0] = *(volatile unsigned *)&dev->absmax_u32;
        if (kNext) cell_s[1] = (uint32_t)*(volatile unsigned long long *)&dev->absmax_u64;
    }
    const int p_in = (src_exp ? __ldg(src_exp) : 0) + exp_bias;
    __syncthreads();
    if (threadIdx.x == 0) last = last_reader(dev);
    const uint32_t M = cell_s[0];
    const int t = M ? round_log2_u32(M) : 7;
    const int p0 = M ? p_in + t - 7 : p_in;
    NextHead nh = {};
    if (kNext) nh = next_head_setup(next.gamma, (uint32_t)abs(sq_code32((int32_t)cell_s[1], t)), dev);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *dst_exp = p0;
        if (!M) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
        if (kNext) next_head_exponent(nh, p0, next.e3_exp, dev);
    }
    long long sum = 0, s1 = 0, s2 = 0;
    const int sh = t - 7;
    JoinMul jm = {};
    if (kJoin) jm = join_mul(join_shift(p0, __ldg(join.b_exp)));
    // the maximum bounds every element, so |a| + 2^(sh-1) cannot wrap as long as M + M / 2^7 < 2^31
    const bool fast = sh >= 1 && M < 0x7e000000u;
    const int32_t half_m1 = fast ? (1 << (sh - 1)) - 1 : 0, lo = fast ? -(127 << sh) : 0;
    uint32_t jm32 = 0, jmm32 = 0;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    while (i < n16) {
        Group ahead = {};   // the thread's next group travels while this one is worked on
        if (i + stride < n16) {
            load16(i + stride, ahead);
            if (kNext && next.x2) ptx::prefetch_l1(next.x2 + (i + stride) * 16);
        }
        uint32_t cw[4];   // four codes per word
        if constexpr (kPacked) {
            sum_codes_16(t, cur.raw, cw);
        } else {
            const int32_t *a = reinterpret_cast<const int32_t *>(cur.raw);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                cw[q] = fast ? sq_pack4_shr(a + 4 * q, sh, half_m1, lo)
                             : pack4_sat(sq_code32(a[4 * q], t), sq_code32(a[4 * q + 1], t), sq_code32(a[4 * q + 2], t), sq_code32(a[4 * q + 3], t));
        }
        int sum16 = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) sum16 = __dp4a((int)cw[q], 0x01010101, sum16);
        sum += sum16;
        reinterpret_cast<int4 *>(dst)[i] = make_int4((int)cw[0], (int)cw[1], (int)cw[2], (int)cw[3]);
        if (kJoin) {
            const uint32_t bw[4] = {(uint32_t)cur.b.x, (uint32_t)cur.b.y, (uint32_t)cur.b.z, (uint32_t)cur.b.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t g = bw[q] & bits_to_bytes(cur.gate >> (4 * q)), m = cur.nm >> (4 * q);
                uint32_t u[4];
                join_sums(jm.pair, cw[q], g, 0u, u);
                const uint32_t u0 = (uint32_t)abs((int32_t)u[0]), u1 = (uint32_t)abs((int32_t)u[1]), u2 = (uint32_t)abs((int32_t)u[2]),
                               u3 = (uint32_t)abs((int32_t)u[3]);
                jm32 = max(max(jm32, u0), max(u1, max(u2, u3)));
                if (m & 1u) jmm32 = max(jmm32, u0);
                if (m & 2u) jmm32 = max(jmm32, u1);
                if (m & 4u) jmm32 = max(jmm32, u2);
                if (m & 8u) jmm32 = max(jmm32, u3);
            }
        }
        if (kNext) {
            const uint32_t bits = cur.nm;
            uint32_t e1[4], c3[4];
            int a1 = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                e1[q] = cw[q] & bits_to_bytes(bits >> (4 * q));
                a1 = __dp4a((int)e1[q], 0x01010101, a1);
                c3[q] = next_head_codes(nh, e1[q]);
            }
            s1 += a1;
            if (next.x2) s2 += dot16_s8_s16(e1, reinterpret_cast<const int4 *>(next.x2) + 2 * i);
            reinterpret_cast<int4 *>(next.e3)[i] = make_int4((int)c3[0], (int)c3[1], (int)c3[2], (int)c3[3]);
        }
        i += stride;
        cur = ahead;
    }
    ptx::grid_dep_launch();
    if (!kPacked)
        for (size_t i = n16 * 16 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
            const int c = sq_code32(src[i], t);
            sum += c;
            dst[i] = (int8_t)c;
        }
    {
        long long v[kNext ? 3 : 1];
        v[0] = sum;
        if (kNext) {
            v[kNext ? 1 : 0] = s1;
            v[kNext ? 2 : 0] = s2;
        }
        if (kNext || sum_codes) block_sums_i64(v);
        if (threadIdx.x == 0) {
            auto add = [](long long *dst, long long x) {
                if (dst && x) atomicAdd(reinterpret_cast<unsigned long long *>(dst), (unsigned long long)x);
            };
            add(sum_codes, v[0]);
            if (kNext) {
                add(next.sum_e1, v[kNext ? 1 : 0]);
                add(next.sum_e1x2, v[kNext ? 2 : 0]);
            }
        }
    }
    if (kJoin) {
        // the join's second pass (the next kernel on the stream) reads these cells and puts them back to zero
        jm32 = block_max_u32(jm32);
        __syncthreads();
        jmm32 = block_max_u32(jmm32);
        if (threadIdx.x == 0) {
            if (jm32) atomicMax(&dev->absmax_u64, join_magnitude(jm, jm32));
            if (jmm32) atomicMax(&dev->absmax2_u64, join_magnitude(jm, jmm32));
        }
    }
    if (last) {
        dev->absmax_u32 = 0;
        if (kNext) dev->absmax_u64 = 0;
    }
}

// n / d for n below 2^31 by one multiplication (Granlund and Montgomery: m = ceil(2^(31 + s) / d) with s = ceil(log2 d)).
struct Divider {
    uint32_t d, m, s;
    Divider(uint32_t d_) : d(d_), m(0), s(0)
    {
        while ((1ull << s) < d) ++s;
        if (d > 1) m = (uint32_t)(((1ull << (31 + s)) + d - 1) / d);
    }
    __device__ __forceinline__ uint32_t quotient(uint32_t n) const { return d == 1 ? n : __umulhi(n, m) >> (s - 1); }
};
// items are [image][row][column][group of 16 channels]
struct ScatterShape {
    Divider groups, ww, hh, stride;
};

// Q_e for a strided 1x1 filter: only the pixels (y, x) with y and x multiples of the stride receive an error, the
// others are exactly zero.  The GEMM leaves its sums (16-bit words) compact, [n][hq][wq][c]; this kernel writes the full tensor
// [n][h][w][c], codes on the grid and zeros elsewhere, so neither a cleared full-size tensor of sums nor a pass over
// it is needed.  A thread writes 16 channels of one pixel.  Bound by the latency of its first loads and by its
// stores.  12.8 M codes behind a GEMM, from launch to end: 10.8 us with five divisions an item and one load in flight, 8.8 now.
__global__ void __launch_bounds__(kThreads)
sq_sums_scatter_kernel(const uint16_t *__restrict__ src, const int32_t *src_exp, int exp_bias, uint32_t items,
                       uint32_t first_row, int last_part, const __grid_constant__ ScatterShape sh, int hq, int wq, int8_t *dst, int32_t *dst_exp,
                       long long *sum_codes, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    __shared__ uint32_t cell_s;   // (the protocol of sq_i32_kernel)
    bool last = false;
    if (threadIdx.x == 0) cell_s = *(volatile unsigned *)&dev->absmax_u32;
    __syncthreads();
    if (threadIdx.x == 0) last = last_reader(dev);
    const uint32_t M = cell_s;
    const int t = M ? round_log2_u32(M) : 7;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int p_in = (src_exp ? *src_exp : 0) + exp_bias;
        *dst_exp = M ? p_in + t - 7 : p_in;
        if (!M) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
    }
    long long sum = 0;
    const uint32_t c = sh.groups.d * 16u, step = gridDim.x * kThreads;
    dst += (size_t)first_row * sh.ww.d * c;
    constexpr int kAtOnce = 2;   // loads in flight together
    for (uint32_t i0 = blockIdx.x * kThreads + threadIdx.x; i0 < items; i0 += kAtOnce * step) {   // (items stay below 2^30: it cannot wrap)
        uint32_t raw[kAtOnce][8];
        bool on[kAtOnce];
#pragma unroll
        for (int u = 0; u < kAtOnce; ++u) {
            const uint32_t i = i0 + u * step;
            const uint32_t pix = sh.groups.quotient(i), g = i - pix * sh.groups.d;
            const uint32_t local = sh.ww.quotient(pix), x = pix - local * sh.ww.d, row = first_row + local;
            const uint32_t img = sh.hh.quotient(row), y = row - img * sh.hh.d;
            const uint32_t yq = sh.stride.quotient(y), xq = sh.stride.quotient(x);
            on[u] = i < items && yq * sh.stride.d == y && xq * sh.stride.d == x;
            if (on[u]) ld_global_256_stream(src + (((size_t)img * hq + yq) * wq + xq) * c + g * 16u, raw[u]);
        }
#pragma unroll
        for (int u = 0; u < kAtOnce; ++u) {
            const uint32_t i = i0 + u * step;
            if (i >= items) break;
            int4 out = make_int4(0, 0, 0, 0);
            if (on[u]) {
                uint32_t cw[4];
                sum_codes_16(t, raw[u], cw);
                int sc = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) sc = __dp4a((int)cw[k], 0x01010101, sc);
                sum += sc;
                out = make_int4((int)cw[0], (int)cw[1], (int)cw[2], (int)cw[3]);
            }
            reinterpret_cast<int4 *>(dst)[i] = out;
        }
    }
    if (sum_codes) {
        long long v[1] = {sum};
        block_sums_i64(v);
        if (threadIdx.x == 0 && v[0]) atomicAdd(reinterpret_cast<unsigned long long *>(sum_codes), (unsigned long long)v[0]);
    }
    if (last && last_part) dev->absmax_u32 = 0;
}

// ------------------------------------------------------------------ head of the error chain

// Two chained passes over e0 and the mask, the second out of the L2.  Bound by launch latency up to a million codes, then by the
// latency of the loads: a thread's next group travels while it works on one.  One cooperative kernel that kept e1 in registers read
// everything once, but cannot be chained to its predecessor: 0.26, 1.6, 6.4 and 12.8 M codes with x2 took it 8.1, 8.2, 9.6 and 13.4
// us in a row of calls, the two 4.1, 4.8, 7.7 and 11.2 (backward of 512 channels 7 x 7 at batch 64 58.6 -> 52.2 us).

// largest |code| of a byte word, running (a code of -128 counts as 127)
struct HeadMax {
    uint32_t mx = 0, mn = 0;   // packed 16-bit halves
    __device__ __forceinline__ void add(uint32_t w)
    {
        uint32_t even, odd;   // sign-extended by one permute per two codes
        asm("prmt.b32 %0, %1, %1, 0xA280;" : "=r"(even) : "r"(w));
        asm("prmt.b32 %0, %1, %1, 0xB391;" : "=r"(odd) : "r"(w));
        mx = __vimax3_s16x2(mx, even, odd);
        mn = __vimin3_s16x2(mn, even, odd);
    }
    __device__ __forceinline__ uint32_t value() const
    {
        const int hi = max((int)(int16_t)mx, (int)mx >> 16), lo = min((int)(int16_t)mn, (int)mn >> 16);
        return (uint32_t)min(max(hi, -lo), 127);
    }
};

// Pass 1: max |e1| and the sums behind g_b2 and g_gamma, with e1 = e0 * [x4 > 0].
__global__ void __launch_bounds__(kThreads)
prescale_reduce_kernel(const int8_t *__restrict__ e0, const uint8_t *__restrict__ mask, const int16_t *__restrict__ x2, size_t n16,
                       DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    HeadMax most;
    long long v[2] = {0, 0};
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    struct Group {
        int4 e;
        uint32_t m;
    } cur = {};
    auto load = [&](size_t i) {
        if (x2) ptx::prefetch_l1(x2 + i * 16);
        return Group{__ldg(reinterpret_cast<const int4 *>(e0) + i), mask ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(mask) + i) : 0xffffu};
    };
    if (i < n16) cur = load(i);
    for (; i < n16; i += stride) {
        Group ahead = {};
        if (i + stride < n16) ahead = load(i + stride);
        const uint32_t w[4] = {(uint32_t)cur.e.x, (uint32_t)cur.e.y, (uint32_t)cur.e.z, (uint32_t)cur.e.w};
        uint32_t e1[4];
        int a1 = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            e1[q] = w[q] & bits_to_bytes(cur.m >> (4 * q));
            most.add(e1[q]);
            a1 = __dp4a((int)e1[q], 0x01010101, a1);
        }
        v[0] += a1;
        if (x2) v[1] += dot16_s8_s16(e1, reinterpret_cast<const int4 *>(x2) + 2 * i);
        cur = ahead;
    }
    ptx::grid_dep_launch();
    const uint32_t mx = block_max_u32(most.value());
    block_sums_i64(v);
    if (threadIdx.x == 0) {
        if (mx) atomicMax(&dev->absmax_u32, mx);
        if (v[0]) atomicAdd(reinterpret_cast<unsigned long long *>(&dev->sum0), (unsigned long long)v[0]);
        if (v[1]) atomicAdd(reinterpret_cast<unsigned long long *>(&dev->sum1), (unsigned long long)v[1]);
    }
}

// gamma of a launch: the host value, or the code read from device memory (clamped to 16 bits, EOQ_DEV_RANGE raised)
__device__ __forceinline__ int32_t load_gamma(int32_t gamma_c, const int32_t *gamma_dev, DeviceState *dev)
{
    if (!gamma_dev) return gamma_c;
    int32_t g = __ldg(gamma_dev);
    if (g < -32768 || g > 32767) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&dev->status, EOQ_DEV_RANGE);
        g = clampi(g, -32768, 32767);
    }
    return g;
}

// Pass 2: e3 = Q_e(gamma * e1) under the reduced maximum.
__global__ void __launch_bounds__(kThreads)
prescale_apply_kernel(const int8_t *__restrict__ e0, const int32_t *e0_exp, const uint8_t *__restrict__ mask, size_t n16, int32_t gamma_c,
                      const int32_t *gamma_dev, int8_t *e3, int32_t *e3_exp, long long *sum_e1, long long *sum_e1x2, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    __shared__ uint32_t max_s;   // (the protocol of sq_i32_kernel)
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    struct Group {
        int4 e;
        uint32_t m;
    } cur = {};
    auto load = [&](size_t i) {
        return Group{__ldg(reinterpret_cast<const int4 *>(e0) + i), mask ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(mask) + i) : 0xffffu};
    };
    if (i < n16) cur = load(i);
    if (threadIdx.x == 0) max_s = *reinterpret_cast<volatile unsigned *>(&dev->absmax_u32);
    gamma_c = load_gamma(gamma_c, gamma_dev, dev);
    __syncthreads();
    const uint32_t M = max_s * (uint32_t)abs(gamma_c);  // max |gamma * e1| < 2^7 * 2^15
    const int t = M ? round_log2_u32(M) : 7;
    bool last = false;
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) {
            const int p_in = *e0_exp - 7;
            *e3_exp = M ? p_in + t - 7 : p_in;
            if (!M) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
            if (sum_e1) *sum_e1 = *reinterpret_cast<volatile long long *>(&dev->sum0);
            if (sum_e1x2) *sum_e1x2 = *reinterpret_cast<volatile long long *>(&dev->sum1);
            __threadfence();   // read before the block counts as a reader
        }
        last = last_reader(dev);
    }
    // R(v * 2^(7-t)) for v = gamma * e1 (|v| < 2^22) on the floating-point pipe: kHeadMagic + v read as a float is
    // 1.5 * 2^23 + v exactly; one fused multiply-add forms 1.5 * 2^23 + v * 2^(7-t) (the products are exact, the sum
    // is rounded once, to nearest even at unit spacing), so the low bits of the result are the rounded quotient.
    // For t < 7 the scaling is a left shift and nothing is rounded; either way |result| < 2^22 keeps the binade.
    NextHead nh;
    nh.g = (uint32_t)gamma_c;
    nh.scale = __int_as_float((127 + 7 - t) << 23);   // 2^(7-t), t in [0, 22]
    nh.rest = 12582912.0f - 12582912.0f * nh.scale;   // exact: a multiple of a power of two below 2^31
    for (; i < n16; i += stride) {
        Group ahead = {};
        if (i + stride < n16) ahead = load(i + stride);
        const uint32_t w[4] = {(uint32_t)cur.e.x, (uint32_t)cur.e.y, (uint32_t)cur.e.z, (uint32_t)cur.e.w};
        uint32_t c3[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) c3[q] = next_head_codes(nh, w[q] & bits_to_bytes(cur.m >> (4 * q)));
        reinterpret_cast<int4 *>(e3)[i] = make_int4((int)c3[0], (int)c3[1], (int)c3[2], (int)c3[3]);
        cur = ahead;
    }
    ptx::grid_dep_launch();
    if (last) {
        dev->absmax_u32 = 0;
        dev->sum0 = 0;
        dev->sum1 = 0;
    }
}

// Self-test of the bounded waits (eoq_debug_force_wait_timeout), in the place of the call's passes: an mbarrier of two arrivals gets one.
// Warp 0 waits as the GEMM kernels' MMA issuer does, runs into `limit`, raises the abort flag and flags the handle; warp 1 waits as their
// loaders and epilogues do, sixteen times as long, and leaves by the abort flag.  Behind them the reduction cells are what a kernel that gave
// up may leave behind.  Writes nothing else.
__global__ void __launch_bounds__(64) wait_self_test_kernel(DeviceState *dev, uint32_t limit)
{
    __shared__ __align__(8) uint64_t bar_s;
    __shared__ volatile uint32_t abort_s;
    const uint32_t bar = ptx::smem_u32(&bar_s);
    if (threadIdx.x == 0) {
        abort_s = 0;
        ptx::mbar_init(bar, 2);
        ptx::fence_barrier_init();
    }
    __syncthreads();
    const RoleCtx ctx{&abort_s, dev};
    bool met;
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) ptx::mbar_arrive(bar);
        met = __all_sync(0xffffffffu, wait_bar(bar, 0, ctx, limit));
    } else {
        met = __all_sync(0xffffffffu, wait_bar<64>(bar, 0, ctx, 16 * limit));
    }
    if (__syncthreads_or(met) || threadIdx.x != 0) return;
    dev->absmax_u32 = 0x7f000000u;
    dev->absmax_u64 = dev->absmax2_u64 = 1ull << 40;
    dev->sum0 = dev->sum1 = -1;
    dev->ticket = 1;
}

// The same in one cluster of up to kHeadCluster blocks, for tensors of that many blocks' shares: every thread keeps its share of e1 (up to
// kHeadGroups groups of 16 codes) in registers between the passes, the maxima and sums meet in distributed shared memory, and one launch
// does it.  Bound by latency: 4.6 us for 65,536 codes with x2, as long as the two passes take; at 196,608 codes, six groups a thread,
// 6.3 us and they 4.6.  (It is one launch less where calls are issued one by one.)
constexpr int kHeadCluster = 8, kHeadGroups = 2;
__global__ void __launch_bounds__(kThreads)
prescale_cluster_kernel(const int8_t *__restrict__ e0, const int32_t *e0_exp, const uint8_t *__restrict__ mask,
                        const int16_t *__restrict__ x2, size_t n16, int32_t gamma_c, const int32_t *gamma_dev, int8_t *e3,
                        int32_t *e3_exp, long long *sum_e1, long long *sum_e1x2, DeviceState *dev)
{
    __shared__ __align__(16) uint32_t cells[kHeadCluster][8];   // of each block: maximum, -, sum of e1 (2 words), of e1 * x2 (2 words)
    ptx::cluster_arrive();   // (met before the first write to another block's shared memory)
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    gamma_c = load_gamma(gamma_c, gamma_dev, dev);
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t e1w[kHeadGroups][4];
    uint32_t mx4 = 0;
    long long s1 = 0, s2 = 0;
    {
        int4 ev[kHeadGroups];
        uint32_t mv[kHeadGroups];
#pragma unroll
        for (int u = 0; u < kHeadGroups; ++u) {
            const size_t i = i0 + u * stride;
            const bool in = i < n16;
            ev[u] = in ? __ldg(reinterpret_cast<const int4 *>(e0) + i) : make_int4(0, 0, 0, 0);
            mv[u] = (in && mask) ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(mask) + i) : 0xffffu;
        }
#pragma unroll
        for (int u = 0; u < kHeadGroups; ++u) {
            const uint32_t w[4] = {(uint32_t)ev[u].x, (uint32_t)ev[u].y, (uint32_t)ev[u].z, (uint32_t)ev[u].w};
            int a1 = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                e1w[u][q] = w[q] & bits_to_bytes(mv[u] >> (4 * q));
                mx4 = __vmaxu4(mx4, __vabsss4(e1w[u][q]));
                a1 = __dp4a((int)e1w[u][q], 0x01010101, a1);
            }
            s1 += a1;
            const size_t i = i0 + u * stride;
            if (x2 && i < n16) s2 += dot16_s8_s16(e1w[u], reinterpret_cast<const int4 *>(x2) + 2 * i);
        }
    }
    uint32_t mx = max(max(mx4 & 0xffu, (mx4 >> 8) & 0xffu), max((mx4 >> 16) & 0xffu, mx4 >> 24));
    mx = block_max_u32(mx);
    long long sums[2] = {s1, s2};
    block_sums_i64(sums);   // valid in warp 0's first lane, as the maximum
    ptx::cluster_wait();
    if (threadIdx.x < 32) {
        mx = __shfl_sync(0xffffffffu, mx, 0);
        s1 = __shfl_sync(0xffffffffu, sums[0], 0);
        s2 = __shfl_sync(0xffffffffu, sums[1], 0);
        if (threadIdx.x < gridDim.x) {
            const uint32_t dst = ptx::cluster_addr(ptx::smem_u32(&cells[blockIdx.x][0]), threadIdx.x);
            ptx::st_cluster_128(dst, mx, 0u, (uint32_t)s1, (uint32_t)(s1 >> 32));
            ptx::st_cluster_128(dst + 16, (uint32_t)s2, (uint32_t)(s2 >> 32), 0u, 0u);
        }
    }
    ptx::cluster_sync();
    uint32_t M = 0;
    for (int r = 0; r < (int)gridDim.x; ++r) M = max(M, cells[r][0]);
    M *= (uint32_t)abs(gamma_c);
    const int t = M ? round_log2_u32(M) : 7;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int p_in = *e0_exp - 7;
        *e3_exp = M ? p_in + t - 7 : p_in;
        if (!M) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
        long long t1 = 0, t2 = 0;
        for (int r = 0; r < (int)gridDim.x; ++r) {
            t1 += (long long)((unsigned long long)cells[r][3] << 32 | cells[r][2]);
            t2 += (long long)((unsigned long long)cells[r][5] << 32 | cells[r][4]);
        }
        if (sum_e1) *sum_e1 = t1;
        if (sum_e1x2) *sum_e1x2 = t2;
    }
    NextHead nh;   // (the rounding of prescale_apply_kernel)
    nh.g = (uint32_t)gamma_c;
    nh.scale = __int_as_float((127 + 7 - t) << 23);
    nh.rest = 12582912.0f - 12582912.0f * nh.scale;
#pragma unroll
    for (int u = 0; u < kHeadGroups; ++u) {
        const size_t i = i0 + u * stride;
        if (i >= n16) continue;
        uint32_t c3[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) c3[q] = next_head_codes(nh, e1w[u][q]);
        reinterpret_cast<int4 *>(e3)[i] = make_int4((int)c3[0], (int)c3[1], (int)c3[2], (int)c3[3]);
    }
}

// ------------------------------------------------------------------ layout helpers

// [n][rows][cols] -> [n][cols][rows] on bytes, 32 x 32 tiles through shared memory.
__global__ void transpose_bytes_kernel(const int8_t *__restrict__ src, int8_t *__restrict__ dst, int rows, int cols)
{
    __shared__ int8_t tile[32][33];
    const size_t img = (size_t)blockIdx.z * rows * cols;
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int rr = r0 + r, cc = c0 + threadIdx.x;
        if (rr < rows && cc < cols) tile[r][threadIdx.x] = src[img + (size_t)rr * cols + cc];
    }
    __syncthreads();
    for (int c = threadIdx.y; c < 32; c += blockDim.y) {
        const int cc = c0 + c, rr = r0 + threadIdx.x;
        if (rr < rows && cc < cols) dst[img + (size_t)cc * rows + rr] = tile[threadIdx.x][c];
    }
}

// ------------------------------------------------------------------ b1 support

// table[class][oc] = sum over the taps valid for the class, and over ic, of w[oc][tap][ic]  (the forward
// pass adds b1 times this: conv(x0 + b1) = conv(x0) + b1 * conv(indicator of the image)).
// One block per output channel: warps reduce the taps' channel sums, then threads combine them per class.
__global__ void b1_weight_table_kernel(const int8_t *__restrict__ w, int32_t *table, eoq_conv_desc_t d, int ho, int wo,
                                       BorderClasses bc)
{
    __shared__ int32_t tap_sum[kMaxTaps];
    const int oc = blockIdx.x;
    const int taps = d.kh * d.kw;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    for (int t = warp; t < taps; t += nwarps) {
        const int4 *p = reinterpret_cast<const int4 *>(w + ((size_t)oc * taps + t) * d.c_in);
        int sum = 0;
        for (int i = lane; i < d.c_in / 16; i += 32) {
            const int4 v = __ldg(p + i);
            sum = __dp4a(v.x, 0x01010101, sum);
            sum = __dp4a(v.y, 0x01010101, sum);
            sum = __dp4a(v.z, 0x01010101, sum);
            sum = __dp4a(v.w, 0x01010101, sum);
        }
        if (d.c_in == 8 && lane == 0) {  // the 8-channel first layer: one 8-byte pixel per tap
            const int2 v = __ldg(reinterpret_cast<const int2 *>(p));
            sum = __dp4a(v.x, 0x01010101, sum);
            sum = __dp4a(v.y, 0x01010101, sum);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) tap_sum[t] = sum;
    }
    __syncthreads();
    for (int cls = threadIdx.x; cls < bc.nrc * bc.ncc; cls += blockDim.x) {
        const int rc = cls / bc.ncc, cc = cls % bc.ncc;
        int32_t sum = 0;
        for (int kh = 0; kh < d.kh; ++kh) {
            if (!tap_valid(rc, kh, ho, d.h, bc.nlo_h, bc.nhi_h, bc.nrc, d.stride, d.pad)) continue;
            for (int kw = 0; kw < d.kw; ++kw)
                if (tap_valid(cc, kw, wo, d.w, bc.nlo_w, bc.nhi_w, bc.ncc, d.stride, d.pad)) sum += tap_sum[kh * d.kw + kw];
        }
        table[(size_t)cls * d.c_out + oc] = sum;
    }
}

// What eoq_weight_prep derives from the weights of several layers in one launch: the b1 table of every layer
// (as b1_weight_table_kernel builds it) and, for a first layer on the filter-row path, the weights re-packed as
// [oc][kh][8][c_in] with zero taps.  One block per (layer, output channel), bound by latency: the taps that each
// border class takes are worked out while the kernel in front runs, all chunks of a channel are loaded at once and added to their tap's
// cell (a single 16-channel layer's calls 35.0 -> 34.0 us with the former in front of the wait).
__global__ void weight_prep_kernel(const __grid_constant__ PrepBatch b)
{
    __shared__ int32_t tap_sum[kMaxTaps];
    int k = 0;
    for (int hi = b.num - 1; k < hi;) {
        const int mid = (k + hi + 1) >> 1;
        if ((int)blockIdx.x >= b.first_block[mid]) k = mid;
        else hi = mid - 1;
    }
    const PrepItem &it = b.item[k];
    const eoq_conv_desc_t &d = it.d;
    const BorderClasses &bc = it.bc;
    const int oc = blockIdx.x - b.first_block[k];
    const int taps = d.kh * d.kw, width = d.c_in == 8 ? 8 : 16, per_tap = d.c_in / width, chunks = taps * per_tap;
    const int8_t *w = it.w + (size_t)oc * taps * d.c_in;
    // what the launch's parameters give, while the kernels in front still run
    for (int t = threadIdx.x; t < taps; t += blockDim.x) tap_sum[t] = 0;
    const int classes = bc.nrc * bc.ncc;   // at most kMaxBorderClasses, fewer than threads
    unsigned long long takes = 0;          // the taps of this thread's class that fall inside the image
    if ((int)threadIdx.x < classes) {
        const int rc = threadIdx.x / bc.ncc, cc = threadIdx.x - rc * bc.ncc;
        unsigned long long row = 0;
        for (int kw = 0; kw < d.kw; ++kw)
            if (tap_valid(cc, kw, it.wo, d.w, bc.nlo_w, bc.nhi_w, bc.ncc, d.stride, d.pad)) row |= 1ull << kw;
        for (int kh = 0; kh < d.kh; ++kh)
            if (tap_valid(rc, kh, it.ho, d.h, bc.nlo_h, bc.nhi_h, bc.nrc, d.stride, d.pad)) takes |= row << (kh * d.kw);
    }
    ptx::grid_dep_wait_launch_small();
    auto load = [&](int i) {
        if (width == 16) return __ldg(reinterpret_cast<const int4 *>(w) + i);
        const int2 v = __ldg(reinterpret_cast<const int2 *>(w) + i);   // the 8-channel first layer: one 8-byte pixel per tap
        return make_int4(v.x, v.y, 0, 0);
    };
    constexpr int kAhead = 3;   // 3 x 3 filters of up to 640 channels in one round
    int4 v[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
        const int i = threadIdx.x + u * blockDim.x;
        if (i < chunks) v[u] = load(i);
    }
    if (it.w_rows) {
        // this output channel's filter rows, each widened to 8 taps (c_in is 16 or 8: 4 or 2 words per tap)
        const int words = d.c_in / 4;
        const int32_t *src = reinterpret_cast<const int32_t *>(it.w) + (size_t)oc * taps * words;
        int32_t *dst = reinterpret_cast<int32_t *>(it.w_rows) + (size_t)oc * d.kh * 8 * words;
        for (int i = threadIdx.x; i < d.kh * 8 * words; i += blockDim.x) {
            const int r = i / (8 * words), t = (i / words) % 8, wd = i % words;
            dst[i] = t < d.kw ? __ldg(src + (r * d.kw + t) * words + wd) : 0;
        }
    }
    __syncthreads();
    auto add = [&](int i, const int4 &q) {
        const int s = __dp4a(q.x, 0x01010101, __dp4a(q.y, 0x01010101, __dp4a(q.z, 0x01010101, __dp4a(q.w, 0x01010101, 0))));
        if (per_tap % 32 == 0) {   // a warp's chunks belong to one tap (and `chunks` is a multiple of 32)
            const int sum = __reduce_add_sync(0xffffffffu, s);
            if ((threadIdx.x & 31) == 0) atomicAdd(&tap_sum[i / per_tap], sum);
        } else {
            atomicAdd(&tap_sum[i / per_tap], s);
        }
    };
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
        const int i = threadIdx.x + u * blockDim.x;
        if (i < chunks) add(i, v[u]);
    }
    for (int i = threadIdx.x + kAhead * blockDim.x; i < chunks; i += blockDim.x) add(i, load(i));
    __syncthreads();
    if ((int)threadIdx.x < classes) {
        int32_t sum = 0;
        for (unsigned long long m = takes; m; m &= m - 1) sum += tap_sum[__ffsll((long long)m) - 1];
        it.table[(size_t)threadIdx.x * d.c_out + oc] = sum;
    }
}

}  // namespace

// ------------------------------------------------------------------ launchers

cudaError_t launch_reset_cells(DeviceState *dev, cudaStream_t s)
{
    // every cell after the status word
    return cudaMemsetAsync(reinterpret_cast<char *>(dev) + offsetof(DeviceState, absmax_u32), 0,
                           offsetof(DeviceState, tensor_absmax) - offsetof(DeviceState, absmax_u32), s);
}

bool quantize_is_small(int mode, size_t n, const ReduceHook &hook) { return mode == 2 && !hook.fn && n <= kSmallElems * kSmallCluster; }

// Largest tensor whose codes wait for the maximum (see quantize_sq_kernel).  Normal numbers / one element beyond all others / tiles of
// unequal size, us, tensors from memory: 8 M floats 13.3 / 15.3 / 15.1 under the guess, 12.6 read twice; 10.5 M 15.3 / 16.8 / 17.1 and 15.3, the
// line; 12.8 M 17.4 / 18.6 / 18.4 and 17.4 (in a row of calls on three tensors 16.4 or 17.7 from process to process, and 17.5); 21 M 23.0 /
// 27.5 / 26.7 and 27.9; 34 M 39.1 / 36.7 / 37.3 and 44.0.  The worst of them is no slower than a maximum's pass with one load of a thread in
// flight was (17.7, 21.3, 32.4, 50.4); below the line it is (4 M: 12.0 and 10.2).
constexpr size_t kSqResident = 10u << 20;

static unsigned quantize_tiles(size_t n) { return n / 4 > kQuantTile ? (unsigned)((n / 4 + kQuantTile - 1) / kQuantTile) : 1u; }

// Tiles of the SQ that guesses: `reps` parts each, more than one only where the handle has no cell for every part; the second pass's
// blocks look after at most kThreads tiles each.
struct TileSplit {
    int reps, tiles, again_blocks;
};
static TileSplit split_tiles(size_t parts, int sm_count)
{
    TileSplit t;
    t.reps = (int)((parts + kSqTiles - 1) / kSqTiles);
    t.tiles = (int)((parts + t.reps - 1) / t.reps);
    const int least = (t.tiles + kThreads - 1) / kThreads, most = kAgainPerSm * sm_count;
    t.again_blocks = t.tiles < most ? t.tiles : (least > most ? least : most);
    return t;
}

// The largest |x| into the cell (and its exchange: float bit patterns of |x| order like integers).
static void launch_sq_maximum(const float *src, size_t n, DeviceState *dev, cudaStream_t s, const ReduceHook &hook)
{
    launch_chained(absmax_f32_kernel, quantize_tiles(n), kThreads, 0, s, src, n, dev);
    hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, s);
}

cudaError_t launch_quantize_f32(int mode, const float *src, size_t n, void *dst, int32_t *dst_exp, int16_t *tile_shift, DeviceState *dev,
                                int sm_count, cudaStream_t s, const ReduceHook &hook)
{
    if (quantize_is_small(mode, n, hook)) {
        int blocks = 1;
        while ((size_t)blocks * kSmallElems < n) blocks *= 2;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim = {(unsigned)blocks, 1, 1};
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(kSmallThreads);
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, quantize_sq_small_kernel, src, n, static_cast<int8_t *>(dst), dst_exp, dev);
    }
    const unsigned tiles = quantize_tiles(n);
    if (mode == 2 && n > kSqResident) {
        const TileSplit t = split_tiles(tiles, sm_count);
        launch_chained(quantize_sq_kernel, t.tiles, kThreads, 0, s, src, n, static_cast<int8_t *>(dst), tile_shift, t.reps, dev);
        hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, s);
        launch_chained(quantize_sq_again_kernel, t.again_blocks, kThreads, 0, s, src, n, static_cast<int8_t *>(dst), dst_exp,
                       (const int16_t *)tile_shift, t.tiles, t.reps, dev);
        return cudaGetLastError();
    }
    if (mode == 2) {
        launch_sq_maximum(src, n, dev, s, hook);
        launch_chained(quantize_sq_second_kernel, tiles, kThreads, 0, s, src, n, static_cast<int8_t *>(dst), dst_exp, dev, (int)!hook.fn);
    } else if (mode == 0) {
        launch_chained(quantize_f32_kernel<0>, tiles, kThreads, 0, s, src, n, dst, dst_exp);
    } else {
        launch_chained(quantize_f32_kernel<1>, tiles, kThreads, 0, s, src, n, dst, dst_exp);
    }
    return cudaGetLastError();
}

cudaError_t launch_quantize_image(const float *src, int n, int h, int w, int c_src, int c_dst, int wmargin, int8_t *dst, int32_t *dst_exp,
                                  DeviceState *dev, cudaStream_t s, const ReduceHook &hook)
{
    launch_sq_maximum(src, (size_t)n * h * w * c_src, dev, s, hook);
    const int g = c_dst % 16 == 0 ? 16 : 8, items = (w + 2 * wmargin) * (c_dst / g);
    const ImageShape shape{n * h, w, c_src, c_dst, wmargin};
    int tx = 32;
    while (tx < items && tx < kThreads) tx *= 2;
    const dim3 block(tx, kThreads / tx);
    const int block_rows = kImageRows * (int)block.y;
    const bool staged = c_src <= 4 && c_dst == g && items <= kThreads;
    const auto kernel = staged ? (g == 16 ? quantize_image_kernel<16, true> : quantize_image_kernel<8, true>)
                               : (g == 16 ? quantize_image_kernel<16, false> : quantize_image_kernel<8, false>);
    launch_chained(kernel, (unsigned)((shape.rows + block_rows - 1) / block_rows), block, 0, s, src, shape, dst, dst_exp, dev, (int)!hook.fn);
    return cudaGetLastError();
}

cudaError_t launch_weight_pad_rows(const int8_t *w, int8_t *wp, int c_out, int kh, int kw, int c_in, cudaStream_t s)
{
    const int rows = c_out * kh;
    if (c_in == 16) weight_pad_rows_kernel<int4><<<(rows * 8 + 255) / 256, 256, 0, s>>>(w, wp, rows, kw);
    else weight_pad_rows_kernel<int2><<<(rows * 8 + 255) / 256, 256, 0, s>>>(w, wp, rows, kw);
    return cudaGetLastError();
}

cudaError_t launch_sq_i32(const int32_t *src, const int32_t *src_exp, int exp_bias, size_t n, int8_t *dst,
                          int32_t *dst_exp, long long *sum_codes, bool max_already_reduced, DeviceState *dev,
                          int sm_count, cudaStream_t s, const ReduceHook &hook)
{
    if (!max_already_reduced) absmax_i32_kernel<<<grid_for(n / 4 + 1, sm_count), kThreads, 0, s>>>(src, n, dev);
    hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, s);
    launch_chained(sq_i32_kernel<false, false, false>, grid_for(n / 16 + 1, sm_count), kThreads, 0, s, src, src_exp, exp_bias, n, dst, dst_exp,
                   sum_codes, NextHeadArgs{}, JoinStatArgs{}, dev);
    if (sum_codes) hook(sum_codes, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, s);
    return cudaGetLastError();
}

cudaError_t launch_sq_sums(const uint16_t *src, const int32_t *src_exp, int exp_bias, size_t n, int8_t *dst, int32_t *dst_exp,
                           long long *sum_codes, DeviceState *dev, int sm_count, cudaStream_t s, const ReduceHook &hook,
                           const NextHeadArgs *next, const JoinStatArgs *join)
{
    hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, s);
    const int grid = grid_for(n / 16 + 1, sm_count);
    if (join) {
        // (no hook in this form: callers with replicas take the separate calls)
        launch_chained(sq_i32_kernel<true, false, true>, grid, kThreads, 0, s, src, src_exp, exp_bias, n, dst, dst_exp, sum_codes, NextHeadArgs{}, *join, dev);
    } else if (next) {
        // (only behind a GEMM whose epilogue reduced the masked maximum)
        hook(&dev->absmax_u64, 1, EOQ_REDUCE_I64, EOQ_REDUCE_MAX, s);
        launch_chained(sq_i32_kernel<true, true, false>, grid, kThreads, 0, s, src, src_exp, exp_bias, n, dst, dst_exp, sum_codes, *next, JoinStatArgs{}, dev);
        if (next->sum_e1) hook(next->sum_e1, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, s);
        if (next->sum_e1x2) hook(next->sum_e1x2, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, s);
    } else {
        launch_chained(sq_i32_kernel<true, false, false>, grid, kThreads, 0, s, src, src_exp, exp_bias, n, dst, dst_exp, sum_codes, NextHeadArgs{},
                       JoinStatArgs{}, dev);
    }
    if (sum_codes) hook(sum_codes, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, s);
    return cudaGetLastError();
}

cudaError_t launch_sq_sums_scatter(const uint16_t *src, const int32_t *src_exp, int exp_bias, int n_img, int hh, int ww, int c,
                                   int stride, int hq, int wq, int8_t *dst, int32_t *dst_exp, long long *sum_codes,
                                   DeviceState *dev, int sm_count, cudaStream_t s, const ReduceHook &hook)
{
    const ScatterShape shape{Divider(c / 16), Divider(ww), Divider(hh), Divider(stride)};
    hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, s);
    const size_t row_items = (size_t)ww * (c / 16), rows = (size_t)n_img * hh, most = std::max<size_t>(1, (1u << 30) / row_items);
    for (size_t r = 0; r < rows; r += most) {   // (one launch below 2^30 items)
        const size_t items = std::min(most, rows - r) * row_items;
        launch_chained(sq_sums_scatter_kernel, grid_for(items, sm_count, 5), kThreads, 0, s, src, src_exp, exp_bias, (uint32_t)items, (uint32_t)r,
                       r + most >= rows ? 1 : 0, shape, hq, wq, dst, dst_exp, sum_codes, dev);
    }
    if (sum_codes) hook(sum_codes, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, s);
    return cudaGetLastError();
}

cudaError_t launch_err_prescale(const int8_t *e0, const int32_t *e0_exp, const uint8_t *mask, const int16_t *x2,
                                size_t n_el, int32_t gamma_c, const int32_t *gamma_dev, int8_t *e3, int32_t *e3_exp,
                                long long *sum_e1, long long *sum_e1x2, DeviceState *dev, int sm_count, cudaStream_t s,
                                int *kernels, bool force_timeout, const ReduceHook &hook)
{
    const size_t n16 = n_el / 16;
    *kernels = 2;
    const size_t share = (size_t)kThreads * kHeadGroups;
    if (force_timeout) {
        *kernels = 1;
        wait_self_test_kernel<<<1, 64, 0, s>>>(dev, 256u);
        return cudaGetLastError();
    }
    if (!hook.fn && n16 > 0 && n16 <= kHeadCluster * share) {
        // one cluster, of the fewest blocks that hold the tensor
        int blocks = 1;
        while ((size_t)blocks * share < n16) blocks *= 2;
        *kernels = 1;
        return launch_chained_clusters(blocks, prescale_cluster_kernel, blocks, kThreads, 0, s, e0, e0_exp, mask, x2, n16, gamma_c, gamma_dev, e3,
                                       e3_exp, sum_e1, sum_e1x2, dev);
    }
    const int grid = grid_for(n16, sm_count, 5);
    launch_chained(prescale_reduce_kernel, grid, kThreads, 0, s, e0, mask, x2, n16, dev);
    hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, s);
    hook(&dev->sum0, 2, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, s);  // sum0 and sum1 are adjacent
    launch_chained(prescale_apply_kernel, grid, kThreads, 0, s, e0, e0_exp, mask, n16, gamma_c, gamma_dev, e3, e3_exp, sum_e1, sum_e1x2, dev);
    return cudaGetLastError();
}

cudaError_t launch_layout_convert(const int8_t *src, int8_t *dst, int n, int c, int h, int w, int to_nhwc,
                                  cudaStream_t s)
{
    // NCHW is [n][c][hw]; NHWC is [n][hw][c]
    const int rows = to_nhwc ? c : h * w, cols = to_nhwc ? h * w : c;
    dim3 grid((cols + 31) / 32, (rows + 31) / 32, n), block(32, 8);
    transpose_bytes_kernel<<<grid, block, 0, s>>>(src, dst, rows, cols);
    return cudaGetLastError();
}

cudaError_t launch_b1_weight_table(const int8_t *w, int32_t *table, const eoq_conv_desc_t &d, const BorderClasses &bc,
                                   cudaStream_t s)
{
    const int ho = (d.h + 2 * d.pad - d.kh) / d.stride + 1, wo = (d.w + 2 * d.pad - d.kw) / d.stride + 1;
    b1_weight_table_kernel<<<d.c_out, 128, 0, s>>>(w, table, d, ho, wo, bc);
    return cudaGetLastError();
}

cudaError_t launch_weight_prep(const PrepBatch &b, cudaStream_t s)
{
    launch_chained(weight_prep_kernel, b.first_block[b.num], 128, 0, s, b);
    return cudaGetLastError();
}

}  // namespace eoq
