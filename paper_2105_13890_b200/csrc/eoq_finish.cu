// What follows the weight-gradient GEMM (arXiv 2105.13890, Sec. 3.2.1: g_w = Q_g(e3 * x1) with x1 = x0 + Q_b(b1)), for one
// layer or for many layers in the same three launches: the b1 error sums (one pass over e3), the exact sums (split-K slices
// plus the b1 term) reduced to their maximum, and Q_g.  Blocks find their layer by their index.
// The maximum's cell is cleared by the GEMM kernel, as are the b1 error sums' cells where these are added up (FinishItem::tap_add).
#include "eoq_device.cuh"
#include "eoq_internal.h"

namespace eoq {

namespace {

constexpr int kThreads = 256;
constexpr int kTapSlab = 32;      // channels one block of the error sums covers: a 32-byte sector of a pixel
constexpr int kTapThreads = 512;

__device__ __forceinline__ int finish_item_of(const int *first, int num, int block)
{
    int k = 0;
    while (k + 1 < num && block >= first[k + 1]) ++k;
    return k;
}

__device__ __forceinline__ int finish_b1(const FinishItem &it)
{
    return it.b1_dev ? clampi(__ldg(it.b1_dev), -32768, 32767) : it.b1_c;
}

// Do the layer's sums fit 32 bits?  |G| <= pixels * 127 * (127 + |b1|).
__device__ __forceinline__ bool finish_narrow(const FinishItem &it, int b1)
{
    return it.pixels < (1ull << 31) && (double)it.pixels * 127.0 * (127.0 + (double)abs(b1)) < 2147483647.0;
}

// ------------------------------------------------------------------ b1 error sums
// tap_sums[oc][tap] = sum of e3[n,y,x,oc] over the pixels for which the tap falls inside the image (the weight gradient
// adds b1 times this to every input channel).  Only border rows and columns ever fall outside a tap, so with T the sum over
// all pixels, R_i and C_j those over the i-th border row and the j-th border column, and P_ij those over their crossings,
//   tap sum = T - sum of R_i - sum of C_j + sum of P_ij   over the border rows and columns the tap does not take.
// Every term is a plain sum over a regular set of pixels.  A block covers a range of rows and a slab of channels; a lane
// keeps the sums of 16 channels (one 128-bit load per pixel, several in flight).  All warps sum T, then share out the border sets.
// A slab's rows are dealt to its blocks.  Up to kTapReplicas blocks store a copy of the cells each; more of them add to the copies, which
// the GEMM has cleared.
// Bound by the latency of a few dependent rounds of loads.  A single layer's sums run beside its GEMM, which lets them in once it has seen
// e3 complete; they wait for its end before they add, or before they end.  Up to kTapsFirstBytes of errors they go in front and let the GEMM
// in, which waits for them at its end: they would be the last to end behind it (48 -> 80 channels, stride 2, 37 x 29 at batch 5: 12.4 us for the
// weight gradient, 11.6 so; 64 channels 56 x 56 at batch 4, 0.8 M errors, 15.6 beside, 17.2 in front).  Whichever comes second finds
// room because the first asks its SMs for all the shared memory there is: an SM divides its memory between L1 and shared memory when it is
// idle.  All sums in front of the GEMM, in clusters of up to eight blocks that stored what they had summed through distributed shared
// memory, left few slabs too few blocks, and the GEMM waited for many: 16 -> 32 channels 56 x 56 at batch 512 68.3 us for the weight
// gradient, 58.2 so, 64 -> 64 99 and 82, 16 -> 240 by 1 x 1, 64 x 64 at batch 40, 35.5 and 28.3; 64 -> 128 channels 56 x 56, stride 2, batch 64
// 19.9 and 19.5, 1024 -> 256 by 1 x 1, 14 x 14, batch 32 14.8 and 14.0.  Sums of four pixels by dot products and no divisions in front of the
// first load: the kernel 7.5 -> 5.5 us for the 48 -> 80 channel strided layer.
struct PixelSum {
    int v[16] = {};
    // adds four pixels: the codes of a channel side by side, then one byte dot product
    __device__ __forceinline__ void add4(const int4 &p0, const int4 &p1, const int4 &p2, const int4 &p3)
    {
        const uint32_t w0[4] = {(uint32_t)p0.x, (uint32_t)p0.y, (uint32_t)p0.z, (uint32_t)p0.w};
        const uint32_t w1[4] = {(uint32_t)p1.x, (uint32_t)p1.y, (uint32_t)p1.z, (uint32_t)p1.w};
        const uint32_t w2[4] = {(uint32_t)p2.x, (uint32_t)p2.y, (uint32_t)p2.z, (uint32_t)p2.w};
        const uint32_t w3[4] = {(uint32_t)p3.x, (uint32_t)p3.y, (uint32_t)p3.z, (uint32_t)p3.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t t0 = __byte_perm(w0[q], w1[q], 0x5140), t1 = __byte_perm(w0[q], w1[q], 0x7362), t2 = __byte_perm(w2[q], w3[q], 0x5140),
                           t3 = __byte_perm(w2[q], w3[q], 0x7362);
            v[4 * q] = __dp4a((int)__byte_perm(t0, t2, 0x5410), 0x01010101, v[4 * q]);
            v[4 * q + 1] = __dp4a((int)__byte_perm(t0, t2, 0x7632), 0x01010101, v[4 * q + 1]);
            v[4 * q + 2] = __dp4a((int)__byte_perm(t1, t3, 0x5410), 0x01010101, v[4 * q + 2]);
            v[4 * q + 3] = __dp4a((int)__byte_perm(t1, t3, 0x7632), 0x01010101, v[4 * q + 3]);
        }
    }
    // Adds the warp's sums to the cells of a set: `dst` is the lane's first channel, `lanes` (1 or 2) the lanes of a pixel.  Lanes
    // that hold the same channels would queue at the cells (32 of them for 16 channels), so they first halve their channels among
    // each other, pairwise, and every channel is added once per warp.
    __device__ __forceinline__ void flush(int32_t *dst, int lanes)
    {
        const int lane = threadIdx.x & 31;
        int off = 0;
#pragma unroll
        for (int m = 16, half = 8; half >= 1; m >>= 1, half >>= 1) {
            const bool up = (lane & m) != 0;
#pragma unroll
            for (int c = 0; c < half; ++c) {
                const int keep = up ? v[c + half] : v[c], send = up ? v[c] : v[c + half];
                v[c] = keep + __shfl_xor_sync(0xffffffffu, send, m);
            }
            off += up ? half : 0;
        }
        if (lanes == 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if (lanes > 1 || !(lane & 1)) atomicAdd(dst + off, v[0]);
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = 0;
    }
};

// the i-th border row (column) of `extent` rows, and how many there are: all of them when no interior class exists
__device__ __forceinline__ int border_count(int extent, int nlo, int nhi, int ncls) { return ncls == extent ? extent : nlo + nhi; }
__device__ __forceinline__ int border_at(int i, int extent, int nlo, int nhi, int ncls)
{
    return (ncls == extent || i < nlo) ? i : extent - nhi + (i - nlo);
}
__device__ __forceinline__ bool tap_takes(int y, int k, int stride, int pad, int extent_in)
{
    const int src = y * stride - pad + k;
    return src >= 0 && src < extent_in;
}

// Border rows / columns of the item that a filter row / column does not take, as bits.
struct TapMasks {
    unsigned long long rows[16], cols[16];
};
__device__ __forceinline__ void tap_masks(const FinishItem &it, int nr, int nc, TapMasks &m)
{
    const eoq_conv_desc_t &d = it.d;
    const BorderClasses &bc = it.bc;
    if (threadIdx.x < d.kh) {
        unsigned long long out = 0;
        for (int i = 0; i < nr; ++i)
            if (!tap_takes(border_at(i, it.ho, bc.nlo_h, bc.nhi_h, bc.nrc), threadIdx.x, d.stride, d.pad, d.h)) out |= 1ull << i;
        m.rows[threadIdx.x] = out;
    } else if (threadIdx.x >= 32 && threadIdx.x < 32 + d.kw) {
        unsigned long long out = 0;
        for (int i = 0; i < nc; ++i)
            if (!tap_takes(border_at(i, it.wo, bc.nlo_w, bc.nhi_w, bc.ncc), threadIdx.x - 32, d.stride, d.pad, d.w)) out |= 1ull << i;
        m.cols[threadIdx.x - 32] = out;
    }
}

// Rows [r_begin, r_end) of a slab into sets[1 + border rows][1 + border columns][kTapSlab]; index 0 = all rows / columns.
template <int kT>   // threads of the block
__device__ __forceinline__ void tap_sets(const FinishItem &it, int slab, int slab_ch, int r_begin, int r_end, int nr, int nc, int32_t *sets)
{
    const eoq_conv_desc_t &d = it.d;
    const BorderClasses &bc = it.bc;
    const int ho = it.ho, wo = it.wo, c_out = d.c_out, nsets = (1 + nr) * (1 + nc);
    for (int i = threadIdx.x; i < nsets * kTapSlab; i += kT) sets[i] = 0;
    __syncthreads();
    const int two = slab_ch >> 5, lanes_per_pix = 1 + two, pix_per_step = 32 >> two;   // (a slab has 16 or 32 channels)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lane_ch = (lane & two) * 16, slot = lane >> two;
    const int8_t *base = it.e3 + slab * kTapSlab + lane_ch;
    const int4 zero = make_int4(0, 0, 0, 0);
    PixelSum acc;
    {   // T
        constexpr int kUnroll = 8;
        const size_t p_end = (size_t)r_end * wo;
        const int step = (kT / 32) * pix_per_step;
        for (size_t p0 = (size_t)r_begin * wo + warp * pix_per_step; p0 < p_end; p0 += kUnroll * step) {   // the same in all lanes
            int4 v[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const size_t p = p0 + slot + u * step;
                v[u] = p < p_end ? __ldcg(reinterpret_cast<const int4 *>(base + p * c_out)) : zero;
            }
            acc.add4(v[0], v[1], v[2], v[3]);
            acc.add4(v[4], v[5], v[6], v[7]);
        }
        acc.flush(sets + lane_ch, lanes_per_pix);
    }
    if (nsets > 1) {
        // the border sets, each by as many warps as there are for one
        const int share = max(1, (kT / 32) / (nsets - 1)), r_at = r_begin % ho;
        const float per_row = 1.0f / (float)wo;
        for (int turn = warp; turn < (nsets - 1) * share; turn += kT / 32) {
            constexpr int kUnroll = 4;
            const int set = 1 + turn / share, part = turn % share;
            const int i = set / (1 + nc), j = set - i * (1 + nc);
            int32_t *dst = sets + set * kTapSlab + lane_ch;
            // rows first + q * row_step of the range, columns x0 .. x0 + cols - 1
            int first = r_begin, row_step = 1, x0 = 0, cols = wo;
            if (i > 0) {
                const int y = border_at(i - 1, ho, bc.nlo_h, bc.nhi_h, bc.nrc);
                row_step = ho;
                first = r_begin + y - r_at + (y < r_at ? ho : 0);
            }
            if (j > 0) {
                x0 = border_at(j - 1, wo, bc.nlo_w, bc.nhi_w, bc.ncc);
                cols = 1;
            }
            const int rows = first < r_end ? (r_end - first + row_step - 1) / row_step : 0;
            const int pixels = rows * cols, step = share * pix_per_step;
            for (int q0 = part * pix_per_step; q0 < pixels; q0 += kUnroll * step) {
                int4 v[kUnroll];
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) {
                    // (q / wo: below 2^20 the product is off by less than the half that is added)
                    const int q = q0 + slot + u * step, rq = cols == 1 ? q : (pixels < (1 << 20) ? (int)(((float)q + 0.5f) * per_row) : q / wo);
                    const int r = first + rq * row_step, x = x0 + (q - rq * cols);
                    v[u] = q < pixels ? __ldcg(reinterpret_cast<const int4 *>(base + ((size_t)r * wo + x) * c_out)) : zero;
                }
                acc.add4(v[0], v[1], v[2], v[3]);
            }
            acc.flush(dst, lanes_per_pix);
        }
    }
    __syncthreads();
}

// Range `range` (of `ranges`, each of rows_here rows) of a slab's rows into its tap sums, by the calling block.  sets: shared memory of
// tap_set_bytes.  kMayAdd: false where no item adds (tap_add); kBeside: the layer's GEMM is the launch in front and may still run.
template <int kT, bool kMayAdd, bool kBeside>
__device__ __forceinline__ void finish_taps_slab(const FinishItem &it, int slab, int range, int ranges, int rows_here, int32_t *sets)
{
    __shared__ TapMasks masks;
    const eoq_conv_desc_t &d = it.d;
    const BorderClasses &bc = it.bc;
    const int nr = border_count(it.ho, bc.nlo_h, bc.nhi_h, bc.nrc), nc = border_count(it.wo, bc.nlo_w, bc.nhi_w, bc.ncc);
    tap_masks(it, nr, nc, masks);   // (published by the barriers of tap_sets)
    const int slab_ch = min(kTapSlab, d.c_out - slab * kTapSlab);  // channels of this slab (16 or 32)
    const int taps = d.kh * d.kw, items = taps * slab_ch;
    const int rows = d.n * it.ho;   // (sums below: ranges * rows_here is less than rows + ranges)
    const int begin = (int)min((uint32_t)rows, (uint32_t)range * rows_here), end = (int)min((uint32_t)rows, (uint32_t)begin + rows_here);
    const int chunk = (long long)rows_here * it.wo <= (1 << 23) ? max(1, rows_here) : max(1, (1 << 23) / it.wo);   // keeps the int32 sets exact
    const int ch_shift = 31 - __clz(slab_ch), per_kw = 65536 / d.kw + 1;   // tap / kw = tap * per_kw >> 16 for the few taps there are
    const bool add = kMayAdd && it.tap_add;
    for (int at = 0; at < rows_here; at += chunk) {
        const int r0 = min(end, begin + at), r1 = min(end, r0 + min(chunk, rows_here - at));
        tap_sets<kT>(it, slab, slab_ch, r0, r1, nr, nc, sets);
        if (kBeside && add) ptx::grid_dep_wait();   // (the GEMM has cleared the cells)
        for (int i = threadIdx.x; i < items; i += kT) {   // [tap][channel], stored at [oc][tap]
            const int tap = i >> ch_shift, c = i & (slab_ch - 1), kh = tap * per_kw >> 16, kw = tap - kh * d.kw;
            const unsigned long long rm = masks.rows[kh], cm = masks.cols[kw];
            const int32_t *cell = sets + c;
            auto over_columns = [&](const int32_t *row) {
                int v = row[0];
                for (unsigned long long m = cm; m; m &= m - 1) v -= row[__ffsll((long long)m) * kTapSlab];
                return v;
            };
            int sum = over_columns(cell);
            for (unsigned long long m = rm; m; m &= m - 1) sum -= over_columns(cell + __ffsll((long long)m) * (1 + nc) * kTapSlab);
            long long *copies = it.tap_sums + ((size_t)(slab * kTapSlab + c) * taps + tap) * kTapReplicas;
            if (add) {
                if (sum) atomicAdd(reinterpret_cast<unsigned long long *>(copies + range % kTapReplicas), (unsigned long long)(long long)sum);
                continue;
            }
            copies[range] = at == 0 ? sum : copies[range] + sum;   // (its own copy)
            if (range == 0 && at == 0)
                for (int r = ranges; r < kTapReplicas; ++r) copies[r] = 0;
        }
        __syncthreads();
    }
}

__host__ __device__ inline int tap_slabs(const FinishItem &it) { return (it.d.c_out + kTapSlab - 1) / kTapSlab; }

template <TapsOrder kOrder>
// (at most 64 registers: a block and a CTA of the GEMM share an SM)
__global__ void __launch_bounds__(kTapThreads, 2) finish_taps_kernel(const __grid_constant__ FinishBatch b)
{
    if (kOrder != kTapsBeside) ptx::grid_dep_wait();
    if (kOrder == kTapsFirst) ptx::grid_dep_launch();
    extern __shared__ __align__(16) int32_t sets[];
    const int k = finish_item_of(b.tap_first, b.num, (int)blockIdx.x);
    const int local = (int)blockIdx.x - b.tap_first[k], ranges = b.item[k].tap_ranges, slab = local / ranges;
    finish_taps_slab<kTapThreads, kOrder != kTapsFirst, kOrder == kTapsBeside>(b.item[k], slab, local - slab * ranges, ranges, b.item[k].tap_rows,
                                                                             sets);
    if (kOrder == kTapsBeside) ptx::grid_dep_wait();   // (what comes behind this launch waits for it alone)
}

__device__ __forceinline__ void clear_tap_cell(const FinishItem &it, uint32_t i)
{
    longlong2 *cell = reinterpret_cast<longlong2 *>(it.tap_sums) + (size_t)i * (kTapReplicas / 2);
    cell[0] = cell[1] = make_longlong2(0, 0);
}

// ------------------------------------------------------------------ exact sums and their maximum
// A thread owns four neighbouring weights (c_in is a multiple of 4: they share their (oc, tap)); a block is (256 / groups) such
// quads x `groups` slice groups that meet in shared memory.  The sums are written once, as int32 where they provably fit.
// Bound by the latency of a round of loads, so the launch for one layer is one wave (kSumBlocks blocks of 48 registers to an SM) whose
// threads keep up to four slices in flight, the last and incomplete round too.  In a launch for several layers each of them has up to
// four blocks per SM for itself, several waves in all (plan_finish_item).  With a serial remainder, more blocks than an SM holds and
// 64-bit sums throughout: the layer of 512 channels with three slices 11.1 us, 256 channels with eleven 11.4, 128 with 43 8.6;
// now 6.6, 7.0 and 6.1.  The coding pass reads the written sums: forming them again from one or two slices costs it 6.4 us
// instead of 4.5 at 512 channels and saves this pass 0.1.
constexpr int kSumBlocks = 5;

// b1 term of the quad at weight index 4 q; the copies of a cell are neighbours (one 32-byte sector)
__device__ __forceinline__ long long finish_b1_term(const FinishItem &it, int b1, uint32_t q)
{
    static_assert(kTapReplicas == 4, "two 16-byte loads hold a cell's copies");
    const longlong2 *t = reinterpret_cast<const longlong2 *>(it.tap_sums) + (size_t)((4u * q) / (uint32_t)it.d.c_in) * 2;
    const longlong2 lo = __ldg(t), hi = __ldg(t + 1);
    return (long long)b1 * (lo.x + lo.y + hi.x + hi.y);
}

// Adds slices s, s + groups, ... of quad q, four of them (or what is left) in flight together.  Sum: long long, or int where the
// layer's sums provably fit 32 bits (the slices' sums and the b1 term then fit by themselves).
template <typename Sum>
__device__ __forceinline__ void finish_add_slices(const FinishItem &it, uint32_t q, uint32_t quads, int s, int groups, Sum (&v)[4])
{
    const int4 *p = reinterpret_cast<const int4 *>(it.parts) + q;
    for (; s < it.num_parts; s += 4 * groups) {
        int4 a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            a[u] = s + u * groups < it.num_parts ? __ldg(p + (size_t)(s + u * groups) * quads) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[0] += a[u].x;
            v[1] += a[u].y;
            v[2] += a[u].z;
            v[3] += a[u].w;
        }
    }
}

// Sums of the block's quads, written where the coding pass will read them; returns the thread's maximum.
template <typename Sum>
__device__ __forceinline__ unsigned long long finish_sums_block(const FinishItem &it, int block, int b1, Sum (*part)[4])
{
    constexpr bool kNarrow = sizeof(Sum) == 4;
    const int groups = it.groups, bw = kThreads / groups, tx = threadIdx.x % bw, ty = threadIdx.x / bw;
    const uint32_t quads = (uint32_t)(it.n / 4);
    unsigned long long mx = 0;
    for (uint32_t base = (uint32_t)block * bw; base < quads; base += (uint32_t)it.fin_blocks * bw) {
        const uint32_t q = base + tx;
        const bool in = q < quads;
        Sum v[4] = {0, 0, 0, 0};
        if (in) {
            finish_add_slices(it, q, quads, ty, groups, v);
            if (ty == 0 && it.use_b1) {
                const Sum t = (Sum)finish_b1_term(it, b1, q);
#pragma unroll
                for (int c = 0; c < 4; ++c) v[c] += t;
            }
        }
        if (groups > 1) {
#pragma unroll
            for (int c = 0; c < 4; ++c) part[threadIdx.x][c] = v[c];
            __syncthreads();
            if (ty == 0)
                for (int u = 1; u < groups; ++u)
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[c] += part[u * bw + tx][c];
            __syncthreads();
        }
        if (ty == 0 && in) {
            if (kNarrow) {
                reinterpret_cast<int4 *>(it.acc)[q] = make_int4((int)v[0], (int)v[1], (int)v[2], (int)v[3]);
            } else {
                longlong2 *o = reinterpret_cast<longlong2 *>(it.acc) + 2 * (size_t)q;
                o[0] = make_longlong2(v[0], v[1]);
                o[1] = make_longlong2(v[2], v[3]);
            }
            if (it.copy_out)
#pragma unroll
                for (int c = 0; c < 4; ++c) it.copy_out[4 * (size_t)q + c] = v[c];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (kNarrow) {
                    mx = max((uint32_t)mx, (uint32_t)abs((int)v[c]));
                } else {
                    const unsigned long long a = (unsigned long long)(v[c] < 0 ? -v[c] : v[c]);
                    mx = a > mx ? a : mx;
                }
            }
        }
    }
    return mx;
}

__global__ void __launch_bounds__(kThreads, kSumBlocks) finish_sums_kernel(const __grid_constant__ FinishBatch b)
{
    ptx::grid_dep_wait();
    __shared__ __align__(16) long long part[kThreads][4];
    const int k = finish_item_of(b.fin_first, b.num, (int)blockIdx.x);
    const FinishItem &it = b.item[k];
    const int b1 = it.use_b1 ? finish_b1(it) : 0, block = (int)blockIdx.x - b.fin_first[k];
    unsigned long long mx;
    if (finish_narrow(it, b1) && !it.keep_sums) mx = finish_sums_block<int>(it, block, b1, reinterpret_cast<int (*)[4]>(part));
    else mx = finish_sums_block<long long>(it, block, b1, part);
    mx = block_max_u64(mx);
    if (threadIdx.x == 0 && mx && !it.keep_sums) atomicMax(it.max_cell, mx);
}

// max |.| of 64-bit sums that an all-reduce over replicas completed (keep_sums)
__global__ void __launch_bounds__(kThreads) finish_max_kernel(const long long *__restrict__ src, size_t n, unsigned long long *max_cell)
{
    ptx::grid_dep_wait();
    unsigned long long mx = 0;
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kThreads) {
        const long long v = src[i];
        const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
        mx = a > mx ? a : mx;
    }
    mx = block_max_u64(mx);
    if (threadIdx.x == 0 && mx) atomicMax(max_cell, mx);
}

// ------------------------------------------------------------------ Q_g

__global__ void __launch_bounds__(kThreads) finish_code_kernel(const __grid_constant__ FinishBatch b, unsigned *status)
{
    ptx::grid_dep_wait();
    const int k = finish_item_of(b.sq_first, b.num, (int)blockIdx.x);
    const FinishItem &it = b.item[k];
    const int bx = (int)blockIdx.x - b.sq_first[k];
    const unsigned long long M = *it.max_cell;
    const bool narrow = finish_narrow(it, it.use_b1 ? finish_b1(it) : 0) && !it.keep_sums;   // how the sums were written
    const int t = M ? round_log2_u64(M) : 7;
    if (bx == 0 && threadIdx.x == 0) {
        const int p_in = __ldg(it.e3_exp) - 7;
        *it.g_exp = M ? p_in + t - 7 : p_in;
        if (!M) atomicOr(status, EOQ_DEV_SQ_ZERO);
    }
    if (it.tap_clear)
        for (uint32_t i = (uint32_t)bx * kThreads + threadIdx.x; i < (uint32_t)(it.d.c_out * it.d.kh * it.d.kw); i += (uint32_t)it.sq_blocks * kThreads)
            clear_tap_cell(it, i);
    // sums below 2^31 - 2^(t - 8): a right shift in four 32-bit operations (see sq_code32_shr)
    const bool fast = t >= 8 && M < 0x7e000000ull;
    const int sh = t - 7, half_m1 = fast ? (1 << (sh - 1)) - 1 : 0;
    const uint32_t quads = (uint32_t)(it.n / 4);
    for (uint32_t q = (uint32_t)bx * kThreads + threadIdx.x; q < quads; q += (uint32_t)it.sq_blocks * kThreads) {
        long long v[4];
        if (narrow) {
            const int4 a = __ldg(reinterpret_cast<const int4 *>(it.acc) + q);
            v[0] = a.x;
            v[1] = a.y;
            v[2] = a.z;
            v[3] = a.w;
        } else {
            const longlong2 lo = __ldg(reinterpret_cast<const longlong2 *>(it.acc) + 2 * (size_t)q);
            const longlong2 hi = __ldg(reinterpret_cast<const longlong2 *>(it.acc) + 2 * (size_t)q + 1);
            v[0] = lo.x;
            v[1] = lo.y;
            v[2] = hi.x;
            v[3] = hi.y;
        }
        int cd[4];
        if (fast) {
#pragma unroll
            for (int c = 0; c < 4; ++c) cd[c] = sq_code32_shr((int32_t)v[c], sh, half_m1);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) cd[c] = sq_code64(v[c], t);
        }
        reinterpret_cast<uint32_t *>(it.g)[q] = pack4_sat(cd[0], cd[1], cd[2], cd[3]);
    }
}

// ------------------------------------------------------------------ all of it in one cluster
// The three steps for one small layer in one launch of a cluster: tap sums into the cells, slice sums into shared memory, their
// maximum through distributed shared memory, codes.  Bound by latency, so a layer has to be small: one pass over a CTA's weights and
// four rounds of loads (34,560 weights of a 48 -> 80 layer in 17 passes took 39 us where the three launches take 14).  The 16-channel
// layer at batch 8 called by itself 42.2 -> 39.3 us with it and the error head in a cluster, the backward of the 16-channel layer
// 32 x 32 at batch 2 29.7 -> 24.8, of a 256 -> 64 1 x 1 layer 28.2 -> 23.5.
// The block shares an SM with a CTA of the GEMM, beside which it comes up: launch bounds of more threads than it has keep it at 80 registers,
// so that 24,576 of an SM's are left, a quarter of them in each of its four parts (the GEMMs take 13,824 or 16,384); without them it took 103
// and left 12,288.  The single 16-channel layer takes the same time with either (33.4 and 33.3 us), as its GEMM leaves some SMs alone.
constexpr int kSmallCtas = 8, kSmallThreads = 512, kSmallBounds = kSmallThreads + 160;
constexpr size_t kSmallErrorBytes = 256 * 1024;

__device__ __forceinline__ long long finish_b1_term_fresh(const FinishItem &it, int b1, uint32_t q)   // (cells written in this launch)
{
    const longlong2 *t = reinterpret_cast<const longlong2 *>(it.tap_sums) + (size_t)((4u * q) / (uint32_t)it.d.c_in) * 2;
    const longlong2 lo = __ldcg(t), hi = __ldcg(t + 1);
    return (long long)b1 * (lo.x + lo.y + hi.x + hi.y);
}

__global__ void __launch_bounds__(kSmallBounds) finish_small_kernel(const __grid_constant__ FinishItem it, unsigned *status, int beside)
{
    extern __shared__ __align__(16) int32_t dyn[];   // the tap kernel's sets, then this CTA's sums, four to a quad
    __shared__ long long part[kSmallThreads][4];
    __shared__ __align__(16) unsigned long long max_s[kSmallCtas][2];
    ptx::cluster_arrive();   // (met before the first write to another CTA's shared memory)
    if (!beside) ptx::grid_dep_wait();
    const int rank = (int)blockIdx.x;
    if (it.use_b1) {
        const int slabs = tap_slabs(it), copies_log = slabs <= kSmallCtas / 4 ? 2 : (slabs <= kSmallCtas / 2 ? 1 : 0), copies = 1 << copies_log;
        const int rows_here = (it.d.n * it.ho + copies - 1) >> copies_log;
        for (int i = rank; i < slabs * copies; i += kSmallCtas)
            finish_taps_slab<kSmallThreads, false, false>(it, i >> copies_log, i & (copies - 1), copies, rows_here, dyn);
    }
    ptx::cluster_wait();
    if (it.use_b1) {
        __threadfence();
        ptx::cluster_sync();   // every CTA's tap sums are in the cells
    }
    long long *sums = reinterpret_cast<long long *>(dyn);
    const int groups = it.groups, bw = kSmallThreads / groups, tx = threadIdx.x % bw, ty = threadIdx.x / bw;
    const uint32_t quads = (uint32_t)(it.n / 4), mine = (quads + kSmallCtas - 1) / kSmallCtas;   // quads of a CTA: at most bw
    const uint32_t first = rank * mine, end = min(quads, first + mine), q = first + tx;
    const bool in = q < end;
    // the b1 term of the thread's quad is at hand when the GEMM ends
    const long long term = it.use_b1 && ty == 0 && in ? finish_b1_term_fresh(it, finish_b1(it), q) : 0;
    __syncthreads();   // (the sums go where the tap sums' sets were)
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    unsigned long long mx = 0;
    long long v[4] = {0, 0, 0, 0};
    if (in) {
        const int4 *p = reinterpret_cast<const int4 *>(it.parts) + q;
        int s = ty;
        for (; s + 7 * groups < it.num_parts; s += 8 * groups) {
            int4 a[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) a[u] = __ldg(p + (size_t)(s + u * groups) * quads);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                v[0] += a[u].x;
                v[1] += a[u].y;
                v[2] += a[u].z;
                v[3] += a[u].w;
            }
        }
        for (; s < it.num_parts; s += groups) {
            const int4 a = __ldg(p + (size_t)s * quads);
            v[0] += a.x;
            v[1] += a.y;
            v[2] += a.z;
            v[3] += a.w;
        }
    }
    if (groups > 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) part[threadIdx.x][c] = v[c];
        __syncthreads();
        if (ty == 0)
            for (int u = 1; u < groups; ++u)
#pragma unroll
                for (int c = 0; c < 4; ++c) v[c] += part[u * bw + tx][c];
        __syncthreads();
    }
    if (ty == 0 && in) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            v[c] += term;
            sums[4 * (size_t)(q - first) + c] = v[c];
            if (it.copy_out) it.copy_out[4 * (size_t)q + c] = v[c];
            const unsigned long long a = (unsigned long long)(v[c] < 0 ? -v[c] : v[c]);
            mx = a > mx ? a : mx;
        }
    }
    mx = block_max_u64(mx);   // (its barriers also publish the sums to the block)
    if (threadIdx.x == 0) part[0][0] = (long long)mx;
    __syncthreads();
    if (threadIdx.x < kSmallCtas) {
        const unsigned long long m = (unsigned long long)part[0][0];
        ptx::st_cluster_128(ptx::cluster_addr(ptx::smem_u32(&max_s[rank][0]), threadIdx.x), (uint32_t)m, (uint32_t)(m >> 32), 0u, 0u);
    }
    ptx::cluster_sync();
    if (it.use_b1 && it.tap_clear)   // (every CTA has read the cells)
        for (uint32_t i = rank * kSmallThreads + threadIdx.x; i < (uint32_t)(it.d.c_out * it.d.kh * it.d.kw); i += kSmallCtas * kSmallThreads)
            clear_tap_cell(it, i);
    unsigned long long M = 0;
#pragma unroll
    for (int r = 0; r < kSmallCtas; ++r) M = max_s[r][0] > M ? max_s[r][0] : M;
    const int t = M ? round_log2_u64(M) : 7;
    if (rank == 0 && threadIdx.x == 0) {
        const int p_in = __ldg(it.e3_exp) - 7;
        *it.g_exp = M ? p_in + t - 7 : p_in;
        if (!M) atomicOr(status, EOQ_DEV_SQ_ZERO);
    }
    const bool fast = t >= 8 && M < 0x7e000000ull;
    const int sh = t - 7, half_m1 = fast ? (1 << (sh - 1)) - 1 : 0;
    for (uint32_t q = first + threadIdx.x; q < end; q += kSmallThreads) {
        int cd[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const long long v = sums[4 * (size_t)(q - first) + c];
            cd[c] = fast ? sq_code32_shr((int32_t)v, sh, half_m1) : sq_code64(v, t);
        }
        reinterpret_cast<uint32_t *>(it.g)[q] = pack4_sat(cd[0], cd[1], cd[2], cd[3]);
    }
}

}  // namespace

// Ranges of rows of a slab's tap sums, a block each.  A block reads at least 16 KB of e3 (a fraction of a round of its loads; the small
// ones of a batch of 1 leave SMs to the error chain) and beyond kTapReplicas blocks 128 KB, two rounds: fewer of them leave the chain beside them
// more of the device (ResNet-20 step at batch 128 with 32 KB 532 us, with 128 KB 516).  A layer that has the device to itself (`alone`) is split
// down to 32 KB, into a block for every SM in all (512 -> 2048 channels by 1 x 1, 7 x 7, batch 32, 256 blocks: 19.2 us for the weight gradient, 128: 16.7).
static int split_taps(const FinishItem &it, int sm_count, bool alone)
{
    const unsigned long long bytes = it.pixels * (it.d.c_out < kTapSlab ? it.d.c_out : kTapSlab), share = (alone ? 32ull : 128ull) << 10;
    const int most = !alone ? 32 : (sm_count / tap_slabs(it) > 0 ? sm_count / tap_slabs(it) : 1);
    int ranges = 1;
    while (ranges < kTapReplicas && 2 * ranges <= most && bytes > (16ull << 10) * ranges) ranges *= 2;
    const unsigned long long want = (bytes + share - 1) / share;
    return want <= (unsigned long long)ranges ? ranges : (want < (unsigned long long)most ? (int)want : (most > ranges ? most : ranges));
}

// The launch geometry of an item, from its sizes.
static void plan_finish_item(FinishItem &it, int sm_count, bool alone)
{
    it.groups = it.num_parts >= 64 ? 16 : (it.num_parts >= 32 ? 8 : (it.num_parts >= 8 ? 4 : 1));
    const size_t quads = (size_t)it.n / 4, bw = kThreads / it.groups;
    size_t fb = (quads + bw - 1) / bw;
    const size_t fin_cap = (size_t)sm_count * (alone ? kSumBlocks : 4), cap = (size_t)sm_count * (alone ? 8 : 4);
    it.fin_blocks = (int)(fb < 1 ? 1 : (fb > fin_cap ? fin_cap : fb));
    size_t qb = (quads + kThreads - 1) / kThreads;
    it.sq_blocks = (int)(qb < 1 ? 1 : (qb > cap ? cap : qb));
}

void plan_finish(FinishBatch &b, const FinishItem *items, int num, int sm_count, bool whole_device, const ReduceHook &hook)
{
    b.num = num;
    b.tap_first[0] = b.fin_first[0] = b.sq_first[0] = 0;
    for (int k = 0; k < num; ++k) {
        FinishItem &it = b.item[k];
        it = items[k];
        it.keep_sums = hook.fn != nullptr;
        it.tap_ranges = split_taps(it, sm_count, num == 1 && whole_device);
        it.tap_rows = (it.d.n * it.ho - 1) / it.tap_ranges + 1;
        it.tap_add = it.tap_ranges > kTapReplicas;
        it.tap_clear = it.tap_clear && it.use_b1 && (split_taps(it, sm_count, true) > kTapReplicas || split_taps(it, sm_count, false) > kTapReplicas);
        plan_finish_item(it, sm_count, num == 1);
        b.tap_first[k + 1] = b.tap_first[k] + (it.use_b1 ? tap_slabs(it) * it.tap_ranges : 0);
        b.fin_first[k + 1] = b.fin_first[k] + it.fin_blocks;
        b.sq_first[k + 1] = b.sq_first[k] + it.sq_blocks;
    }
}

// shared memory of an item's tap blocks: at least (1 + border rows)(1 + border columns) sets
static size_t tap_set_bytes(const FinishItem &it)
{
    return it.use_b1 ? sizeof(int32_t) * kTapSlab * (1 + it.bc.nrc) * (1 + it.bc.ncc) : 0;
}

// slice groups of the small kernel: as many as leave its CTAs one pass over their quads
static int small_groups(const FinishItem &it)
{
    const size_t mine = (it.n / 4 + kSmallCtas - 1) / kSmallCtas;
    int groups = 16;
    while (groups > 1 && (kSmallThreads / groups < (int)mine || groups > it.num_parts)) groups /= 2;
    return groups;
}

bool finish_is_small(const FinishItem &it, const ReduceHook &hook)
{
    if (hook.fn || it.n > 4ull * kSmallCtas * kSmallThreads || (it.use_b1 && it.pixels * it.d.c_out > kSmallErrorBytes)) return false;
    return it.num_parts <= 32 * small_groups(it);   // (four rounds of loads)
}

cudaError_t launch_finish_small(FinishItem it, unsigned *status, int sm_count, bool beside, cudaStream_t s)
{
    it.keep_sums = it.tap_add = 0;
    plan_finish_item(it, sm_count, true);
    it.groups = small_groups(it);
    const size_t sums = (it.n / 4 + kSmallCtas - 1) / kSmallCtas * 4 * sizeof(long long), sets = tap_set_bytes(it);
    return launch_chained_clusters(kSmallCtas, finish_small_kernel, kSmallCtas, kSmallThreads, sums > sets ? sums : sets, s, it, status,
                                   (int)beside);   // (16 KB of sums, or 17 KB of sets)
}

bool finish_taps_first(const FinishItem &it)
{
    constexpr size_t kTapsFirstBytes = 256 * 1024;
    return !it.tap_add && it.pixels * it.d.c_out <= kTapsFirstBytes;
}

cudaError_t launch_finish_taps(const FinishBatch &b, TapsOrder order, cudaStream_t s)
{
    size_t smem = 0;   // at most 64 border classes, 130 sets: 17 KB
    for (int k = 0; k < b.num; ++k) smem = tap_set_bytes(b.item[k]) > smem ? tap_set_bytes(b.item[k]) : smem;
    if (order == kTapsFirst) {
        static std::atomic<unsigned long long> allowed;
        const cudaError_t e = allow_smem((const void *)finish_taps_kernel<kTapsFirst>, 48 * 1024, allowed, true);
        if (e != cudaSuccess) return e;
    }
    const auto kernel = order == kTapsFirst    ? finish_taps_kernel<kTapsFirst>
                        : order == kTapsBeside ? finish_taps_kernel<kTapsBeside>
                                               : finish_taps_kernel<kTapsBehind>;
    launch_chained(kernel, b.tap_first[b.num], kTapThreads, smem, s, b);
    return cudaGetLastError();
}

cudaError_t launch_finish_sums(const FinishBatch &b, unsigned *status, cudaStream_t s, const ReduceHook &hook)
{
    launch_chained(finish_sums_kernel, b.fin_first[b.num], kThreads, 0, s, b);
    if (hook.fn)
        // replicas (one layer per call): local sums, b1 term included (it is linear in the error) -> all-reduce ->
        // maximum of the global sums; the copy for the caller is taken from the global sums as well
        for (int k = 0; k < b.num; ++k) {
            const FinishItem &it = b.item[k];
            hook(it.acc, (size_t)it.n, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, s);
            launch_chained(finish_max_kernel, it.fin_blocks, kThreads, 0, s, it.acc, (size_t)it.n, it.max_cell);
            if (it.copy_out) cudaMemcpyAsync(it.copy_out, it.acc, (size_t)it.n * sizeof(long long), cudaMemcpyDeviceToDevice, s);
        }
    launch_chained(finish_code_kernel, b.sq_first[b.num], kThreads, 0, s, b, status);
    return cudaGetLastError();
}

}  // namespace eoq
