// Glue between the quantized convolution units of a Fixup residual network (arXiv 2105.13890, Sec. 3.2.1 chains the
// units: x0 of a layer is x5 of the one before, e0 the error its successor hands back): the exact join of two error streams
// followed by Q_e, and the update of the scalar parameters (Sec. 3.2.3) on their 16-bit
// range.  All of it is bandwidth- or latency-bound support work; none of it touches the tensor cores.
#include "eoq_cells.cuh"
#include "eoq_device.cuh"
#include "eoq_internal.h"
#include "eoq_next_head.cuh"

namespace eoq {

namespace {

constexpr int kThreads = 256;

inline int blocks_for(size_t items, int sm_count, int per_sm = 8)
{
    size_t b = (items + kThreads - 1) / kThreads, cap = (size_t)sm_count * per_sm;
    if (b > cap) b = cap;
    return b < 1 ? 1 : (int)b;
}

// ------------------------------------------------------------------ join of two error streams + Q_e

// pass = 0: max |S| into the handle's 64-bit cell; pass = 1: codes of SQ(S), their sum, exponent; cells back to zero.
// kNext: the error head of the layer that consumes the joined error rides along (see NextHead): pass 0 also reduces
// the maximum over the positions that layer's ReLU lets through, pass 1 also writes that layer's e3 and its two sums.
// Bound by memory and by the latency of its loads: a thread's next group travels while it works on one, operands are scaled, added and
// biased by one dot product per element whatever lies between their exponents (see join_mul) and rounded by one multiply-add.  Every
// distance in 32 bits, in the Q_e passes (sq_i32_kernel) too: ResNet-18 step at batch 64 1338 -> 1240 us, at batch 13 604 -> 583.
template <int kPass, bool kNext>
__global__ void join_kernel(const int8_t *__restrict__ a, const int32_t *a_exp, const int8_t *__restrict__ b, const int32_t *b_exp,
                            const uint8_t *__restrict__ mask_b, size_t n16, int8_t *out, int32_t *out_exp, long long *sum_out,
                            const uint8_t *__restrict__ next_mask, const int16_t *__restrict__ next_x2, const int32_t *next_gamma,
                            int8_t *__restrict__ e3, int32_t *e3_exp, long long *sum_e1, long long *sum_e1x2, DeviceState *dev)
{
    ptx::grid_dep_wait_launch_small();
    const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (kPass == 1 && first < n16) {   // on their way while the maxima are read
        ptx::prefetch_l1(a + first * 16);
        ptx::prefetch_l1(b + first * 16);
        if (mask_b) ptx::prefetch_l1(mask_b + first * 2);
        if (kNext) {
            ptx::prefetch_l1(next_mask + first * 2);
            if (next_x2) ptx::prefetch_l1(next_x2 + first * 16);
        }
    }
    const JoinShift j = join_shift(__ldg(a_exp), __ldg(b_exp));
    long long sum = 0, s1 = 0, s2 = 0;
    int t = 7;
    NextHead nh = {};
    unsigned long long M = 0;
    bool last = false;
    if (kPass == 0 && blockIdx.x == 0 && threadIdx.x == 0) {   // the second pass adds to the sums where the caller wants them
        if (sum_out) *sum_out = 0;
        if (kNext && sum_e1) *sum_e1 = 0;
        if (kNext && sum_e1x2) *sum_e1x2 = 0;
    }
    if (kPass == 1) {
        __shared__ unsigned long long cell_s[2];   // (the protocol of sq_i32_kernel)
        if (threadIdx.x == 0) {
            cell_s[0] = *(volatile unsigned long long *)&dev->absmax_u64;
            cell_s[1] = *(volatile unsigned long long *)&dev->absmax2_u64;
        }
        __syncthreads();
        if (threadIdx.x == 0) last = last_reader(dev);
        M = cell_s[0];
        t = M ? round_log2_u64(M) : 7;
        const int p0 = M ? j.p + t - 7 : j.p;
        if (kNext) {
            const unsigned long long Mm = cell_s[1];
            nh = next_head_setup(next_gamma, (uint32_t)abs(sq_code64((long long)Mm, t)), dev);
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *out_exp = p0;
            if (!M) atomicOr(&dev->status, EOQ_DEV_SQ_ZERO);
            if (kNext) next_head_exponent(nh, p0, e3_exp, dev);
        }
    }
    const JoinMul jm = join_mul(j);
    const JoinCode jc = join_code(jm, M, t);
    uint32_t mx32 = 0, mxm32 = 0;
    struct Group {
        int4 a, b;
        uint32_t m, nm;
    };
    auto load = [&](size_t i) {
        Group g;
        g.a = __ldg(reinterpret_cast<const int4 *>(a) + i);
        g.b = __ldg(reinterpret_cast<const int4 *>(b) + i);
        g.m = mask_b ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(mask_b) + i) : 0xffffu;
        g.nm = kNext ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(next_mask) + i) : 0u;
        return g;
    };
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    Group cur = {};
    if (first < n16) cur = load(first);
    for (size_t i = first; i < n16; i += stride) {
        Group ahead = {};   // the thread's next group travels while this one is worked on
        if (i + stride < n16) {
            ahead = load(i + stride);
            if (kPass == 1 && kNext && next_x2) ptx::prefetch_l1(next_x2 + (i + stride) * 16);
        }
        const uint32_t nm = cur.nm;
        const uint32_t aw[4] = {(uint32_t)cur.a.x, (uint32_t)cur.a.y, (uint32_t)cur.a.z, (uint32_t)cur.a.w};
        const uint32_t bw[4] = {(uint32_t)cur.b.x, (uint32_t)cur.b.y, (uint32_t)cur.b.z, (uint32_t)cur.b.w};
        uint32_t cw[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t g = bw[q] & bits_to_bytes(cur.m >> (4 * q));
            uint32_t u[4];
            if (kPass == 0) {
                join_sums(jm.pair, aw[q], g, 0u, u);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t v = (uint32_t)abs((int32_t)u[k]);
                    mx32 = max(mx32, v);
                    if (kNext && ((nm >> (4 * q + k)) & 1u)) mxm32 = max(mxm32, v);
                }
            } else {
                int32_t v[4];
                join_sums(jc.pair, aw[q], g, kHeadMagic, u);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    v[k] = __viaddmax_s32((int32_t)__float_as_uint(__fmaf_rn(__uint_as_float(u[k]), jc.scale, jc.rest)), -(int32_t)kHeadMagic, -127);
                cw[q] = pack4_sat(v[0], v[1], v[2], v[3]);
            }
        }
        if (kPass == 1) {
            int sum16 = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) sum16 = __dp4a((int)cw[q], 0x01010101, sum16);
            sum += sum16;
            reinterpret_cast<int4 *>(out)[i] = make_int4((int)cw[0], (int)cw[1], (int)cw[2], (int)cw[3]);
            if (kNext) {
                uint32_t e1[4], c3[4];
                int a1 = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    e1[q] = cw[q] & bits_to_bytes(nm >> (4 * q));
                    a1 = __dp4a((int)e1[q], 0x01010101, a1);
                    c3[q] = next_head_codes(nh, e1[q]);
                }
                s1 += a1;
                if (next_x2) s2 += dot16_s8_s16(e1, reinterpret_cast<const int4 *>(next_x2) + 2 * i);
                reinterpret_cast<int4 *>(e3)[i] = make_int4((int)c3[0], (int)c3[1], (int)c3[2], (int)c3[3]);
            }
        }
        cur = ahead;
    }
    ptx::grid_dep_launch();
    if (kPass == 0) {
        mx32 = block_max_u32(mx32);
        __syncthreads();
        if (kNext) mxm32 = block_max_u32(mxm32);
        if (threadIdx.x == 0) {
            if (mx32) atomicMax(&dev->absmax_u64, join_magnitude(jm, mx32));
            if (kNext && mxm32) atomicMax(&dev->absmax2_u64, join_magnitude(jm, mxm32));
        }
    } else {
        long long v[3] = {sum, s1, s2};
        block_sums_i64(v);
        if (threadIdx.x == 0) {
            auto add = [](long long *dst, long long x) {
                if (dst && x) atomicAdd(reinterpret_cast<unsigned long long *>(dst), (unsigned long long)x);
            };
            add(sum_out, v[0]);
            if (kNext) {
                add(sum_e1, v[1]);
                add(sum_e1x2, v[2]);
            }
        }
        if (last) dev->absmax_u64 = dev->absmax2_u64 = 0;
    }
}

// ------------------------------------------------------------------ scalar parameters (Sec. 3.2.3 on a single value)

// One thread per scalar: g = Q_g({total}) (SQ of a single value), u = Q_u(lr g), theta <- Q(theta - u) saturated to 16 bits.
__global__ void scalar_update_kernel(const __grid_constant__ ScalarBatch b, int32_t lr_mant, int32_t lr_exp, int stochastic,
                                     unsigned long long seed, const unsigned long long *step_dev, unsigned long long step)
{
    ptx::grid_dep_wait_launch_small();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= b.num) return;
    const ScalarItem &it = b.item[i];
    if (step_dev) step = *step_dev;
    const long long total = *it.total;
    const int p_total = *it.exp + it.exp_bias;
    int g = 0, pg = p_total;
    if (total != 0) {
        const unsigned long long M = (unsigned long long)(total < 0 ? -total : total);
        const int t = round_log2_u64(M);
        g = sq_code64(total, t);
        pg = p_total + t - 7;
    }
    if (it.grad_out) { it.grad_out[0] = g; it.grad_out[1] = pg; }
    int theta = *it.theta;
    if (g != 0) {
        const int a = lr_mant * g;  // |a| < 2^15
        const int tu = round_log2_u32((uint32_t)abs(a));
        const int u = sq_code32(a, tu);
        const int d = (pg + lr_exp + tu - 7) + 7;  // exponent of u relative to the grid 2^-7
        long long next;
        if (d >= 0) {
            next = (long long)theta - (long long)u * (1ll << min(d, 40));
        } else if (-d > 40) {
            next = theta;
        } else {
            const int s = -d;
            const long long v = (long long)theta * (1ll << s) - u;
            if (!stochastic) {
                next = rne_shr64(v, s);
            } else {
                const unsigned long long r = rounding_bits(rounding_key(seed, step, (unsigned long long)it.tensor_id), 0) & ((1ull << s) - 1ull);
                next = (v + (long long)r) >> s;
            }
        }
        theta = (int)(next < -32768 ? -32768 : (next > 32767 ? 32767 : next));
    }
    *it.theta = theta;
    if (it.mirror) *it.mirror = theta;
}

}  // namespace

// ------------------------------------------------------------------ launchers

cudaError_t launch_join(const int8_t *a, const int32_t *a_exp, const int8_t *b, const int32_t *b_exp, const uint8_t *mask_b,
                        size_t n_el, int8_t *out, int32_t *out_exp, long long *sum_out, const uint8_t *next_mask,
                        const int16_t *next_x2, const int32_t *next_gamma, int8_t *e3, int32_t *e3_exp, long long *sum_e1,
                        long long *sum_e1x2, DeviceState *dev, int sm_count, cudaStream_t st, const ReduceHook &hook)
{
    const size_t n16 = n_el / 16;
    const int blocks = blocks_for(n16, sm_count, 8);
    if (e3) {
        launch_chained(join_kernel<0, true>, blocks, kThreads, 0, st, a, a_exp, b, b_exp, mask_b, n16, out, out_exp, sum_out, next_mask, next_x2,
                                                          next_gamma, e3, e3_exp, sum_e1, sum_e1x2, dev);
        hook(&dev->absmax_u64, 1, EOQ_REDUCE_I64, EOQ_REDUCE_MAX, st);
        hook(&dev->absmax2_u64, 1, EOQ_REDUCE_I64, EOQ_REDUCE_MAX, st);
        launch_chained(join_kernel<1, true>, blocks, kThreads, 0, st, a, a_exp, b, b_exp, mask_b, n16, out, out_exp, sum_out, next_mask, next_x2,
                                                          next_gamma, e3, e3_exp, sum_e1, sum_e1x2, dev);
        if (sum_out) hook(sum_out, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, st);
        if (sum_e1) hook(sum_e1, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, st);
        if (sum_e1x2) hook(sum_e1x2, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, st);
    } else {
        launch_chained(join_kernel<0, false>, blocks, kThreads, 0, st, a, a_exp, b, b_exp, mask_b, n16, out, out_exp, sum_out, nullptr, nullptr,
                                                           nullptr, nullptr, nullptr, nullptr, nullptr, dev);
        hook(&dev->absmax_u64, 1, EOQ_REDUCE_I64, EOQ_REDUCE_MAX, st);
        launch_chained(join_kernel<1, false>, blocks, kThreads, 0, st, a, a_exp, b, b_exp, mask_b, n16, out, out_exp, sum_out, nullptr, nullptr,
                                                           nullptr, nullptr, nullptr, nullptr, nullptr, dev);
        if (sum_out) hook(sum_out, 1, EOQ_REDUCE_I64, EOQ_REDUCE_SUM, st);
    }
    return cudaGetLastError();
}

cudaError_t launch_join_second(const int8_t *a, const int32_t *a_exp, const int8_t *b, const int32_t *b_exp, const uint8_t *mask_b,
                               size_t n_el, int8_t *out, int32_t *out_exp, long long *sum_out, const NextHeadArgs *next,
                               DeviceState *dev, int sm_count, cudaStream_t st)
{
    const size_t n16 = n_el / 16;
    const int blocks = blocks_for(n16, sm_count, 8);
    if (next)
        launch_chained(join_kernel<1, true>, blocks, kThreads, 0, st, a, a_exp, b, b_exp, mask_b, n16, out, out_exp, sum_out, next->mask, next->x2,
                                                          next->gamma, next->e3, next->e3_exp, next->sum_e1, next->sum_e1x2, dev);
    else
        launch_chained(join_kernel<1, false>, blocks, kThreads, 0, st, a, a_exp, b, b_exp, mask_b, n16, out, out_exp, sum_out, nullptr, nullptr,
                                                           nullptr, nullptr, nullptr, nullptr, nullptr, dev);
    return cudaGetLastError();
}

cudaError_t launch_scalar_update(const ScalarBatch &b, int32_t lr_mant, int32_t lr_exp, int stochastic, uint64_t seed,
                                 const unsigned long long *step_dev, uint64_t step, cudaStream_t st)
{
    launch_chained(scalar_update_kernel, (b.num + 63) / 64, 64, 0, st, b, lr_mant, lr_exp, stochastic, seed, step_dev, step);
    return cudaGetLastError();
}

}  // namespace eoq
