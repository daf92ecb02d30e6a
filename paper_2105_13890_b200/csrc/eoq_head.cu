// The end of the network (arXiv 2105.13890): global average pooling as exact integer sums, the floating-point last layer
// (Sec. 5.1 leaves it unquantized) written operation by operation so that it is reproducible bit for bit, and the
// quantized error it hands back.  Every float accumulation is a chain of fused multiply-adds in ascending index order, so
// what bounds these kernels is the length of one chain (4 cycles per link) plus the latency of bringing the operands to
// shared memory ahead of it.
#include "eoq_cells.cuh"
#include "eoq_device.cuh"
#include "eoq_internal.h"

namespace eoq {

namespace {

constexpr int kThreads = 256;

// sums[b][ch] = sum over the hw positions of x[b][.][ch]; one warp per (sample, 16-channel group)
__global__ void __launch_bounds__(kThreads) avgpool_sum_kernel(const int8_t *__restrict__ x, int hw, int c, int items, int32_t *__restrict__ sums)
{
    ptx::grid_dep_wait_launch_small();
    const int groups = c / 16, item = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (item >= items) return;
    const int b = item / groups, g = item - b * groups;
    int acc[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[q] = 0;
#pragma unroll 4
    for (int i = lane; i < hw; i += 32) {
        const int4 v = __ldg(reinterpret_cast<const int4 *>(x + ((size_t)b * hw + i) * c + g * 16));
        const int8_t *e = reinterpret_cast<const int8_t *>(&v);
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[q] += e[q];
    }
    int mine = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int s = __reduce_add_sync(0xffffffffu, acc[q]);
        mine = lane == q ? s : mine;
    }
    if (lane < 16) sums[(size_t)b * c + g * 16 + lane] = mine;
}

// exp(x) from fused multiply-adds and a power-of-two scaling only (x <= 88): x = k ln2 + r with ln 2 in two parts (the
// reduction of Cody and Waite, with the split the Cephes library publishes), then the degree-7 Taylor polynomial
__device__ __forceinline__ float exp_fma(float x)
{
    if (x < -87.0f) return 0.0f;
    if (x > 88.0f) x = 88.0f;
    const float kf = rintf(__fmul_rn(x, 1.44269504088896341f));
    float r = __fmaf_rn(-kf, 0.693145751953125f, x);
    r = __fmaf_rn(-kf, 1.42860682030941723212e-6f, r);
    float p = 1.0f / 5040.0f;
    p = __fmaf_rn(p, r, 1.0f / 720.0f);
    p = __fmaf_rn(p, r, 1.0f / 120.0f);
    p = __fmaf_rn(p, r, 1.0f / 24.0f);
    p = __fmaf_rn(p, r, 1.0f / 6.0f);
    p = __fmaf_rn(p, r, 0.5f);
    p = __fmaf_rn(p, r, 1.0f);
    p = __fmaf_rn(p, r, 1.0f);
    // 2^k with k in [-126, 127] is a normal number and the product is exact short of underflow, which x >= -87 excludes;
    // p < 2 and k = 127 only for x close to 88, where p * 2^127 stays finite
    return __fmul_rn(p, __int_as_float(((int)kf + 127) << 23));
}

// Asynchronous copies of one element or of four from global to shared memory; in = false fills with zeros.
__device__ __forceinline__ void cp_async_4(void *dst, const void *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_16(void *dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

__device__ __forceinline__ float pooled_of(int32_t sum, float fhw) { return __fdiv_rn(__fmul_rn(__int2float_rn(sum), 0.0078125f), fhw); }

// pooled[b][k] = (float)sum * 2^-7 / hw
__global__ void __launch_bounds__(kThreads) head_pooled_kernel(const int32_t *__restrict__ sums, int count, int hw, float *pooled)
{
    ptx::grid_dep_wait_launch_small();
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i < count) pooled[i] = pooled_of(__ldg(sums + i), (float)hw);
}

// logits[b][j] = bias[j] + sum_k fma(W[j][k], pooled[b][k], .), k ascending into one accumulator per (b, j).  A warp
// owns one class and a lane one sample; weights and activations of up to kHeadK channels arrive in shared memory by
// asynchronous copies, all in flight at once, and are read four at a time (rows padded by four floats: the lanes of a
// quarter warp hit different banks).  kFromSums (few samples): the activations are formed here, without a launch of
// their own.  Bound by the chain (512 links, 1.3 us) and the latency of the copies; with a division per filled element,
// loads in turn and a shuffle per link 512 x 1000 took 18.5 us at batch 1, 30.7 us at batch 64 (with the kernel for the
// activations); now 5.2 and 13.0 us.
constexpr int kHeadWarps = 8, kHeadK = 512, kFoldSamples = 8;
template <bool kFromSums>
__global__ void __launch_bounds__(32 * kHeadWarps)
head_logits_kernel(const int32_t *__restrict__ sums, int n, int c, int hw, int classes, const float *__restrict__ W,
                   const float *__restrict__ bias, float *pooled, float *__restrict__ logits)
{
    ptx::grid_dep_wait_launch_small();
    extern __shared__ float4 head_smem[];
    const int kc = min(c, kHeadK), ld = ((kc + 3) & ~3) + 4;
    float *ps = reinterpret_cast<float *>(head_smem), *ws = ps + 32 * ld;
    const int b0 = blockIdx.y * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nb = min(32, n - b0), j = blockIdx.x * kHeadWarps + warp;
    const float *act = kFromSums ? reinterpret_cast<const float *>(sums) : pooled;
    const bool vec = c % 4 == 0 && ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(act)) & 15) == 0;
    float acc = j < classes ? __ldg(bias + j) : 0.0f;
    for (int k0 = 0; k0 < c; k0 += kc) {
        const int kn = min(kc, c - k0);
        if (k0) __syncthreads();
        // one row at a time per warp: this warp's row of W, then its share of the samples
        for (int r = j < classes ? -1 : 0; r * kHeadWarps + warp < nb; ++r) {
            const int sb = r * kHeadWarps + warp;
            const float *src = r < 0 ? W + (size_t)j * c + k0 : act + (size_t)(b0 + sb) * c + k0;
            float *dst = r < 0 ? ws + warp * ld : ps + sb * ld;
            if (vec)
                for (int k = lane * 4; k < kn; k += 128) cp_async_16(dst + k, src + k, true);
            else
                for (int k = lane; k < kn; k += 32) cp_async_4(dst + k, src + k, true);
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        if (kFromSums) {
            const float fhw = (float)hw;
            for (int i = threadIdx.x; i < nb * kn; i += 32 * kHeadWarps) {
                const int sb = i / kn, k = i - sb * kn;
                const float v = pooled_of(__float_as_int(ps[sb * ld + k]), fhw);
                ps[sb * ld + k] = v;
                if (blockIdx.x == 0) pooled[(size_t)(b0 + sb) * c + k0 + k] = v;
            }
            __syncthreads();
        }
        if (lane < nb) {
            const float *p = ps + lane * ld, *w = ws + warp * ld;
            int k = 0;
            // eight links while the operands of the next eight come out of shared memory (the last round
            // reads up to 16 floats past the row: the next row, or the buffer's spare end)
            float4 pa = *reinterpret_cast<const float4 *>(p), pb = *reinterpret_cast<const float4 *>(p + 4);
            float4 wa = *reinterpret_cast<const float4 *>(w), wb = *reinterpret_cast<const float4 *>(w + 4);
#pragma unroll 4
            for (; k + 8 <= kn; k += 8) {
                const float4 p0 = pa, p1 = pb, w0 = wa, w1 = wb;
                pa = *reinterpret_cast<const float4 *>(p + k + 8);
                pb = *reinterpret_cast<const float4 *>(p + k + 12);
                wa = *reinterpret_cast<const float4 *>(w + k + 8);
                wb = *reinterpret_cast<const float4 *>(w + k + 12);
                acc = __fmaf_rn(w0.x, p0.x, acc);
                acc = __fmaf_rn(w0.y, p0.y, acc);
                acc = __fmaf_rn(w0.z, p0.z, acc);
                acc = __fmaf_rn(w0.w, p0.w, acc);
                acc = __fmaf_rn(w1.x, p1.x, acc);
                acc = __fmaf_rn(w1.y, p1.y, acc);
                acc = __fmaf_rn(w1.z, p1.z, acc);
                acc = __fmaf_rn(w1.w, p1.w, acc);
            }
            for (; k < kn; ++k) acc = __fmaf_rn(w[k], p[k], acc);
        }
    }
    if (lane < nb && j < classes) logits[(size_t)(b0 + lane) * classes + j] = acc;
}

// One block per sample: softmax with the maximum subtracted, the gradient of the mean cross-entropy with respect to
// the logits, the sample's loss.  The exponentials are formed in parallel; the denominator is then summed by one
// thread over j ascending into one accumulator, which is the order that makes the result reproducible.  That chain
// bounds the kernel: with the exponentials in shared memory (kShared) a link costs the latency of the addition alone,
// 5.9 us instead of 8.5 us for 1000 classes.
template <bool kShared>
__global__ void __launch_bounds__(kThreads)
head_softmax_kernel(const float *__restrict__ logits, int n, int classes, const int32_t *__restrict__ labels, float *dl, double *loss_n)
{
    ptx::grid_dep_wait_launch_small();
    extern __shared__ float4 head_smem[];
    __shared__ float red[32];
    __shared__ float den_s;
    const int b = blockIdx.x;
    const float *l = logits + (size_t)b * classes;
    float *d = dl + (size_t)b * classes;
    float *ex = kShared ? reinterpret_cast<float *>(head_smem) : d;
    float m = -3.4e38f;
#pragma unroll 4
    for (int j = threadIdx.x; j < classes; j += kThreads) {
        const float v = __ldg(l + j);
        if (kShared) ex[j] = v;
        m = v > m ? v : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float other = __shfl_xor_sync(0xffffffffu, m, o);
        m = other > m ? other : m;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = red[0];
#pragma unroll
    for (int i = 1; i < kThreads / 32; ++i) m = red[i] > m ? red[i] : m;
#pragma unroll 4
    for (int j = threadIdx.x; j < classes; j += kThreads) ex[j] = exp_fma(__fsub_rn(kShared ? ex[j] : __ldg(l + j), m));
    const int y = __ldg(labels + b);
    __syncthreads();
    if (threadIdx.x == 0) {
        float den = 0.0f;
        int j = 0;
        if (kShared) {
#pragma unroll 8
            for (; j + 4 <= classes; j += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(ex + j);
                den = __fadd_rn(den, v.x);
                den = __fadd_rn(den, v.y);
                den = __fadd_rn(den, v.z);
                den = __fadd_rn(den, v.w);
            }
        }
        for (; j < classes; ++j) den = __fadd_rn(den, ex[j]);
        den_s = den;
    }
    const float inv_n = __fdiv_rn(1.0f, (float)n), ly = __ldg(l + y);
    __syncthreads();
    const float den = den_s;
    if (threadIdx.x == kThreads - 1) loss_n[b] = (double)logf(den) - (double)__fsub_rn(ly, m);
#pragma unroll 4
    for (int j = threadIdx.x; j < classes; j += kThreads) {
        const float pr = __fdiv_rn(ex[j], den);
        d[j] = __fmul_rn(__fsub_rn(pr, j == y ? 1.0f : 0.0f), inv_n);
    }
}

// dpooled[b][k] = sum_j fma(dl[b][j], W[j][k], .), j ascending (W before its update); one thread also forms the mean loss.
// Every output is one chain of `classes` dependent multiply-adds (2.4 us for 1000), so the only thing to hide is the
// traffic: a block owns kDpCh channels x kDpN samples and keeps kDpStages - 1 tiles of kDpK rows of W in flight with
// asynchronous copies; tiles are long because what a tile costs besides its links delays the chain.  One tile of 32
// rows ahead left a memory latency on every 32 links: 19 us for 1000 classes, now 9 us at batch 1 and 11 us at batch 64.
constexpr int kDpCh = 32, kDpN = 8, kDpK = 64, kDpStages = 6;
struct DpStage {
    float w[kDpK][kDpCh];
    float d[kDpN][kDpK + 4];   // read as float4, one row per warp
};
__global__ void __launch_bounds__(kDpCh *kDpN)
head_dpooled_kernel(const float *__restrict__ dl, const float *__restrict__ W, int n, int c, int classes, float *dpooled,
                    const double *loss_n, float *loss_out)
{
    ptx::grid_dep_wait_launch_small();
    extern __shared__ float4 head_smem[];
    DpStage *st = reinterpret_cast<DpStage *>(head_smem);
    if (blockIdx.y == gridDim.y - 1) {   // an extra row of blocks: the mean loss, in sample order, beside the chains
        if (blockIdx.x == 0 && threadIdx.x == 0 && loss_out) {
            double s = 0.0;
#pragma unroll 8
            for (int i = 0; i < n; ++i) s += __ldg(loss_n + i);
            *loss_out = (float)(s / n);
        }
        return;
    }
    const int cl = threadIdx.x % kDpCh, nl = threadIdx.x / kDpCh;
    const int k = blockIdx.x * kDpCh + cl, b = blockIdx.y * kDpN + nl;
    const bool vec = (c % 4 == 0) && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
    const int tiles = (classes + kDpK - 1) / kDpK;
    // a warp copies rows wr, wr + 32 of a tile (four channels per lane, four rows per warp and step) and two values of
    // its own sample's dl per lane
    const int wr = threadIdx.x / (kDpCh / 4), wc = (threadIdx.x % (kDpCh / 4)) * 4, wk = blockIdx.x * kDpCh + wc;
    const float *w_src = W + (size_t)wr * c + min(wk, c - 1);
    const float *d_src = dl + (size_t)min(b, n - 1) * classes + cl;
    const size_t w_half = (size_t)32 * c;
    int f_row = 0, f_slot = 0;
    auto fetch = [&]() {
        if (f_row < classes) {
            DpStage &s = st[f_slot];
            const bool in0 = f_row + wr < classes, in1 = f_row + wr + 32 < classes;
            if (vec) {
                cp_async_16(&s.w[wr][wc], in0 ? w_src : W, in0 && wk < c);
                cp_async_16(&s.w[wr + 32][wc], in1 ? w_src + w_half : W, in1 && wk < c);
            } else {
                for (int q = 0; q < 4; ++q) {
                    const bool ch = wk + q < c;
                    cp_async_4(&s.w[wr][wc + q], in0 && ch ? w_src + q : W, in0 && ch);
                    cp_async_4(&s.w[wr + 32][wc + q], in1 && ch ? w_src + w_half + q : W, in1 && ch);
                }
            }
            const bool d0 = f_row + cl < classes, d1 = f_row + cl + 32 < classes;
            cp_async_4(&s.d[nl][cl], d0 ? d_src : dl, d0);
            cp_async_4(&s.d[nl][cl + 32], d1 ? d_src + 32 : dl, d1);
            w_src += 2 * w_half;
            d_src += kDpK;
            f_row += kDpK;
            f_slot = f_slot + 1 == kDpStages ? 0 : f_slot + 1;
        }
        cp_async_commit();   // (an empty group keeps the count of groups in step)
    };
#pragma unroll 1
    for (int t = 0; t < kDpStages - 1; ++t) fetch();
    float acc = 0.0f;
    int slot = 0;
    for (int t = 0; t < tiles; ++t) {
        cp_async_wait<kDpStages - 2>();
        __syncthreads();   // tile t has arrived for everyone, and everyone is done with tile t - 1
        fetch();
        const DpStage &s = st[slot];
        slot = slot + 1 == kDpStages ? 0 : slot + 1;
        const int len = min(kDpK, classes - t * kDpK);
        if (b >= n) continue;
        const float *w = &s.w[0][cl], *d = s.d[nl];
        if (len == kDpK) {
            // eight links while the operands of the next eight come out of shared memory
            float4 da = *reinterpret_cast<const float4 *>(d), db = *reinterpret_cast<const float4 *>(d + 4);
            float wa[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) wa[q] = w[q * kDpCh];
#pragma unroll
            for (int jj = 8; jj <= kDpK; jj += 8) {
                const float4 d0 = da, d1 = db;
                float w0[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) w0[q] = wa[q];
                if (jj < kDpK) {
                    da = *reinterpret_cast<const float4 *>(d + jj);
                    db = *reinterpret_cast<const float4 *>(d + jj + 4);
#pragma unroll
                    for (int q = 0; q < 8; ++q) wa[q] = w[(jj + q) * kDpCh];
                }
                acc = __fmaf_rn(d0.x, w0[0], acc);
                acc = __fmaf_rn(d0.y, w0[1], acc);
                acc = __fmaf_rn(d0.z, w0[2], acc);
                acc = __fmaf_rn(d0.w, w0[3], acc);
                acc = __fmaf_rn(d1.x, w0[4], acc);
                acc = __fmaf_rn(d1.y, w0[5], acc);
                acc = __fmaf_rn(d1.z, w0[6], acc);
                acc = __fmaf_rn(d1.w, w0[7], acc);
            }
        } else {
            for (int jj = 0; jj < len; ++jj) acc = __fmaf_rn(d[jj], w[jj * kDpCh], acc);
        }
    }
    if (k < c && b < n) dpooled[(size_t)b * c + k] = acc;
}

// The same with the block's columns of W whole in shared memory (up to kDpMost classes; W in 16-byte pieces): they are fetched
// beside the softmax kernel.  That one starts its successor only after its own wait, behind which the logits kernel and all in
// front of it are complete, so W is; past the L1 it is read as they left it.  What remains behind the wait is the latency of
// dl and the chain itself, without a barrier in it.  Head without its update, 512 channels and 1000 classes, against the kernel
// above: 15.1 us for 19.0 at batch 1, 27.2 for 35.4 at 64, 44.9 for 51.9 at 128 (two waves of blocks, of which an SM holds one);
// in more waves the other one, three blocks to an SM, covers its loads better (81.5 for 77.6 at 256, 61.7 for 60.2 with 1536
// channels at 64).
constexpr int kDpMost = 1344;
static size_t dp_resident_bytes(int classes) { return ((size_t)(classes + 8) * kDpCh + (size_t)kDpN * (((classes + 3) & ~3) + 12)) * sizeof(float); }
__global__ void __launch_bounds__(kDpCh *kDpN)
head_dpooled_resident_kernel(const float *__restrict__ dl, const float *__restrict__ W, int n, int c, int classes, float *dpooled,
                             const double *loss_n, float *loss_out)
{
    extern __shared__ float4 head_smem[];
    float *ws = reinterpret_cast<float *>(head_smem), *ds = ws + (size_t)(classes + 8) * kDpCh;
    const int cl = threadIdx.x % kDpCh, nl = threadIdx.x / kDpCh;
    const int k0 = blockIdx.x * kDpCh, b = blockIdx.y * kDpN + nl;
    const bool chains = blockIdx.y < gridDim.y - 1;
    if (chains)
        for (int i = threadIdx.x; i < classes * (kDpCh / 4); i += kDpCh * kDpN) {
            const int j = i / (kDpCh / 4), q = (i % (kDpCh / 4)) * 4;
            const bool in = k0 + q < c;   // (c is a multiple of 4)
            cp_async_16(ws + j * kDpCh + q, in ? W + (size_t)j * c + k0 + q : W, in);
        }
    ptx::grid_dep_wait_launch_small();
    if (!chains) {   // an extra row of blocks: the mean loss, in sample order, beside the chains
        if (blockIdx.x == 0 && threadIdx.x == 0 && loss_out) {
            double s = 0.0;
#pragma unroll 8
            for (int i = 0; i < n; ++i) s += __ldg(loss_n + i);
            *loss_out = (float)(s / n);
        }
        return;
    }
    float *d = ds + (size_t)nl * (((classes + 3) & ~3) + 12);
    if (b < n) {   // a warp fetches its own sample's row
        const float *src = dl + (size_t)b * classes;
        if (classes % 4 == 0 && (reinterpret_cast<uintptr_t>(dl) & 15) == 0)
            for (int j = cl * 4; j < classes; j += kDpCh * 4) cp_async_16(d + j, src + j, true);
        else
            for (int j = cl; j < classes; j += kDpCh) cp_async_4(d + j, src + j, true);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    if (b >= n) return;
    const float *w = ws + cl;
    float acc = 0.0f;
    int j = 0;
    // eight links while the operands of the next eight come out of shared memory (the last round reads up to eight rows and
    // values past the end: the buffers have them to spare)
    float4 da = *reinterpret_cast<const float4 *>(d), db = *reinterpret_cast<const float4 *>(d + 4);
    float wa[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) wa[q] = w[q * kDpCh];
#pragma unroll 4
    for (; j + 8 <= classes; j += 8) {
        const float4 d0 = da, d1 = db;
        float w0[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) w0[q] = wa[q];
        da = *reinterpret_cast<const float4 *>(d + j + 8);
        db = *reinterpret_cast<const float4 *>(d + j + 12);
#pragma unroll
        for (int q = 0; q < 8; ++q) wa[q] = w[(j + 8 + q) * kDpCh];
        acc = __fmaf_rn(d0.x, w0[0], acc);
        acc = __fmaf_rn(d0.y, w0[1], acc);
        acc = __fmaf_rn(d0.z, w0[2], acc);
        acc = __fmaf_rn(d0.w, w0[3], acc);
        acc = __fmaf_rn(d1.x, w0[4], acc);
        acc = __fmaf_rn(d1.y, w0[5], acc);
        acc = __fmaf_rn(d1.z, w0[6], acc);
        acc = __fmaf_rn(d1.w, w0[7], acc);
    }
    for (; j < classes; ++j) acc = __fmaf_rn(d[j], w[j * kDpCh], acc);
    if (k0 + cl < c) dpooled[(size_t)b * c + k0 + cl] = acc;
}

// W[j][k] <- fma(-lr, sum_b fma(dl[b][j], pooled[b][k], .), W[j][k]), b ascending; bias[j] alike (thread k == 0).
// kV = 4: a thread owns four adjacent channels, so that a link of its four chains costs one and a quarter loads
// instead of eight (64 samples, 1000 x 512 weights: 18 -> 14.5 us beside the backward pass).
template <int kV>
__global__ void __launch_bounds__(128)
head_update_kernel(const float *__restrict__ dl, const float *__restrict__ pooled, int n, int c, int classes, float lr, float *W, float *bias)
{
    ptx::grid_dep_wait_launch_small();
    const int i = blockIdx.x * blockDim.x + threadIdx.x, cv = c / kV;
    if (i >= classes * cv) return;
    const int j = i / cv, k = (i - j * cv) * kV;
    float acc[kV];
#pragma unroll
    for (int q = 0; q < kV; ++q) acc[q] = 0.0f;
    auto load = [&](int b, float (&p)[kV]) {
        if (kV == 4) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(pooled + (size_t)b * c + k));
            p[0] = v.x;
            p[1 % kV] = v.y;
            p[2 % kV] = v.z;
            p[3 % kV] = v.w;
        } else {
            p[0] = __ldg(pooled + (size_t)b * c + k);
        }
    };
    int b = 0;
    for (; b + 8 <= n; b += 8) {
        float d8[8], p8[8][kV];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            d8[u] = __ldg(dl + (size_t)(b + u) * classes + j);
            load(b + u, p8[u]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int q = 0; q < kV; ++q) acc[q] = __fmaf_rn(d8[u], p8[u][q], acc[q]);
    }
    for (; b < n; ++b) {
        float p1[kV];
        const float d1 = __ldg(dl + (size_t)b * classes + j);
        load(b, p1);
#pragma unroll
        for (int q = 0; q < kV; ++q) acc[q] = __fmaf_rn(d1, p1[q], acc[q]);
    }
    float *w = W + (size_t)j * c + k;
    if (kV == 4) {
        float4 v = *reinterpret_cast<float4 *>(w);
        v.x = __fmaf_rn(-lr, acc[0], v.x);
        v.y = __fmaf_rn(-lr, acc[1 % kV], v.y);
        v.z = __fmaf_rn(-lr, acc[2 % kV], v.z);
        v.w = __fmaf_rn(-lr, acc[3 % kV], v.w);
        *reinterpret_cast<float4 *>(w) = v;
    } else {
        w[0] = __fmaf_rn(-lr, acc[0], w[0]);
    }
    if (k == 0) {
        float db = 0.0f;
#pragma unroll 8
        for (int i2 = 0; i2 < n; ++i2) db = __fadd_rn(db, __ldg(dl + (size_t)i2 * classes + j));
        bias[j] = __fmaf_rn(-lr, db, bias[j]);
    }
}

// ------------------------------------------------------------------ error handed back by the head

// max |dpooled| / hw (as float bit patterns; the division is monotonic) into the handle's cell
__global__ void __launch_bounds__(kThreads) head_error_max_kernel(const float *__restrict__ dpooled, int count, int hw, DeviceState *dev)
{
    uint32_t mx = 0;
#pragma unroll 4
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < count; i += gridDim.x * kThreads)
        mx = max(mx, __float_as_uint(__ldg(dpooled + i)) & 0x7fffffffu);
    mx = block_max_u32(mx);
    if (threadIdx.x == 0) {
        if (mx) atomicMax(&dev->absmax_u32, __float_as_uint(__fdiv_rn(__uint_as_float(mx), (float)hw)));
        if (mx >= 0x7f800000u) atomicOr(&dev->status, EOQ_DEV_NONFINITE);
    }
}

// e[b][pos][ch] = SQ code of dpooled[b][ch] / hw for every position.  A block serves one sample: a thread forms the 16
// codes of its channel group once and writes them to its share of the positions.  kScan: every block finds the maximum
// over all of dpooled itself (up to kScanMost values, which sit in the L2), so no launch in front of it has to; else it
// is in the handle's cell (a reduce hook may have completed it).
constexpr int kScanMost = 65536;
constexpr int kSpreadThreads = 512;
template <bool kScan>
__global__ void __launch_bounds__(kSpreadThreads)
head_error_spread_kernel(const float *__restrict__ dpooled, int n, int hw, int c, int8_t *e, int32_t *e_exp, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    __shared__ uint32_t max_s;
    const float fhw = (float)hw;
    uint32_t mbits;
    bool last = false;
    if (kScan) {
        uint32_t mx = 0;
        const int count = n * c;
        if ((reinterpret_cast<uintptr_t>(dpooled) & 15) == 0) {   // c is a multiple of 16
#pragma unroll 16
            for (int i = threadIdx.x; i < count / 4; i += kSpreadThreads) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(dpooled) + i);
                mx = max(max(mx, max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu)),
                         max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu));
            }
        } else {
            for (int i = threadIdx.x; i < count; i += kSpreadThreads) mx = max(mx, __float_as_uint(__ldg(dpooled + i)) & 0x7fffffffu);
        }
        mx = block_max_u32(mx);
        if (threadIdx.x == 0) {
            max_s = __float_as_uint(__fdiv_rn(__uint_as_float(mx), fhw));
            if (blockIdx.x == 0 && mx >= 0x7f800000u) atomicOr(&dev->status, EOQ_DEV_NONFINITE);
        }
        __syncthreads();
        mbits = max_s;
    } else {
        if (threadIdx.x == 0) max_s = *reinterpret_cast<volatile uint32_t *>(&dev->absmax_u32);
        __syncthreads();
        mbits = max_s;
        if (threadIdx.x == 0) last = last_reader(dev);
    }
    const bool usable = mbits != 0 && mbits < 0x7f800000u;
    const int up = usable ? 7 - round_log2_f32bits(mbits) : 7;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *e_exp = -up;
        if (mbits == 0) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
    }
    const int groups = c / 16, b = blockIdx.x;
    for (int g0 = 0; g0 < groups; g0 += kSpreadThreads) {
        const int gn = min(groups - g0, kSpreadThreads), lanes = kSpreadThreads / gn;   // position lanes per group
        const int g = g0 + (int)threadIdx.x % gn, pl = (int)threadIdx.x / gn;
        if (pl >= lanes) continue;
        const float *src = dpooled + (size_t)b * c + g * 16;
        int q[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) q[k] = clampi(__float2int_rn(scalbnf(__fdiv_rn(__ldg(src + k), fhw), up)), -127, 127);
        const uint4 v = make_uint4(pack4_sat(q[0], q[1], q[2], q[3]), pack4_sat(q[4], q[5], q[6], q[7]), pack4_sat(q[8], q[9], q[10], q[11]),
                                   pack4_sat(q[12], q[13], q[14], q[15]));
        for (int pos = pl; pos < hw; pos += lanes) *reinterpret_cast<uint4 *>(e + (((size_t)b * hw + pos) * groups + g) * 16) = v;
    }
    if (last) dev->absmax_u32 = 0;
}

}  // namespace

cudaError_t launch_avgpool_sum(const int8_t *x, int n, int hw, int c, int32_t *sums, cudaStream_t st)
{
    const int items = n * (c / 16);
    launch_chained(avgpool_sum_kernel, (items + kThreads / 32 - 1) / (kThreads / 32), kThreads, 0, st, x, hw, c, items, sums);
    return cudaGetLastError();
}

cudaError_t launch_head_update(const float *dl, const float *pooled, int n, int c, int classes, float lr, float *W, float *bias,
                               cudaStream_t st)
{
    const bool vec = c % 4 == 0 && ((reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(pooled)) & 15) == 0;
    const int items = classes * (vec ? c / 4 : c);
    if (vec) launch_chained(head_update_kernel<4>, (items + 127) / 128, 128, 0, st, dl, pooled, n, c, classes, lr, W, bias);
    else launch_chained(head_update_kernel<1>, (items + 127) / 128, 128, 0, st, dl, pooled, n, c, classes, lr, W, bias);
    return cudaGetLastError();
}

bool head_folds_pooling(int n) { return n <= kFoldSamples; }

cudaError_t launch_head(const int32_t *sums, int n, int c, int hw, int classes, float *W, float *bias, const int32_t *labels,
                        float lr, float *loss_out, float *dpooled, float *logits, float *pooled, float *dl, double *loss_n,
                        cudaStream_t st)
{
    const int kc = c < kHeadK ? c : kHeadK, ld = ((kc + 3) & ~3) + 4;
    const size_t logits_smem = ((size_t)(32 + kHeadWarps) * ld + 16) * sizeof(float), dp_smem = kDpStages * sizeof(DpStage);
    const bool fold = head_folds_pooling(n);
    cudaError_t e = cudaFuncSetAttribute(fold ? head_logits_kernel<true> : head_logits_kernel<false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(((32 + kHeadWarps) * (kHeadK + 4) + 16) * sizeof(float)));
    const dim3 dp_grid((c + kDpCh - 1) / kDpCh, (n + kDpN - 1) / kDpN + 1);
    const bool resident = c % 4 == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0 && classes <= kDpMost &&
                          dp_grid.x * dp_grid.y <= 2u * kPartSms;
    if (e == cudaSuccess)
        e = resident ? cudaFuncSetAttribute(head_dpooled_resident_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dp_resident_bytes(kDpMost))
                     : cudaFuncSetAttribute(head_dpooled_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dp_smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((classes + kHeadWarps - 1) / kHeadWarps, (n + 31) / 32);
    if (fold) {
        launch_chained(head_logits_kernel<true>, grid, 32 * kHeadWarps, logits_smem, st, sums, n, c, hw, classes, W, bias, pooled, logits);
    } else {
        launch_chained(head_pooled_kernel, (n * c + kThreads - 1) / kThreads, kThreads, 0, st, sums, n * c, hw, pooled);
        launch_chained(head_logits_kernel<false>, grid, 32 * kHeadWarps, logits_smem, st, sums, n, c, hw, classes, W, bias, pooled, logits);
    }
    const size_t soft_smem = ((size_t)classes * sizeof(float) + 15) & ~(size_t)15;
    if (soft_smem <= 48 * 1024 - 256) launch_chained(head_softmax_kernel<true>, n, kThreads, soft_smem, st, logits, n, classes, labels, dl, loss_n);
    else launch_chained(head_softmax_kernel<false>, n, kThreads, 0, st, logits, n, classes, labels, dl, loss_n);
    if (resident)
        launch_chained(head_dpooled_resident_kernel, dp_grid, kDpCh * kDpN, dp_resident_bytes(classes), st, dl, W, n, c, classes, dpooled, loss_n, loss_out);
    else launch_chained(head_dpooled_kernel, dp_grid, kDpCh * kDpN, dp_smem, st, dl, W, n, c, classes, dpooled, loss_n, loss_out);
    if (lr != 0.0f) return launch_head_update(dl, pooled, n, c, classes, lr, W, bias, st);
    return cudaGetLastError();
}

bool head_error_is_single(int n, int c, const ReduceHook &hook) { return !hook.fn && (long long)n * c <= kScanMost; }

cudaError_t launch_head_error(const float *dpooled, int n, int c, int hw, int8_t *e, int32_t *e_exp, DeviceState *dev, int sm_count,
                              cudaStream_t st, const ReduceHook &hook)
{
    if (head_error_is_single(n, c, hook)) {
        launch_chained(head_error_spread_kernel<true>, n, kSpreadThreads, 0, st, dpooled, n, hw, c, e, e_exp, dev);
        return cudaGetLastError();
    }
    const int blocks = (n * c + kThreads - 1) / kThreads;
    head_error_max_kernel<<<blocks < sm_count ? blocks : sm_count, kThreads, 0, st>>>(dpooled, n * c, hw, dev);
    hook(&dev->absmax_u32, 1, EOQ_REDUCE_I32, EOQ_REDUCE_MAX, st);
    launch_chained(head_error_spread_kernel<false>, n, kSpreadThreads, 0, st, dpooled, n, hw, c, e, e_exp, dev);
    return cudaGetLastError();
}

}  // namespace eoq
