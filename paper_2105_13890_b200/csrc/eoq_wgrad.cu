// Weight-gradient kernel for sm_100a (arXiv 2105.13890, Sec. 3.2.1: g_w = Q_g(e3 * x1)).
//   D[(tap, ic), oc] = sum over error pixels q of  x[q shifted by tap, ic] * e3[q, oc]
// The reduction runs over pixels, which is the slow axis of both NHWC operands, so both are fed to
// tcgen05.mma as MN-major tiles: a TMA im2col load brings [pixels][channels] of the activation for one
// filter tap, a tiled TMA load brings [pixels][channels] of the error.  The pixel range is split across
// CTAs (split-K); each leaves its int32 partial sums in the slice of its split, and a finishing kernel adds the slices in
// 64 bits.
// Roles: warps 0, 2, 3 TMA producers, warp 1 MMA issuer and TMEM owner, warps 4-7 epilogue.  All waits are bounded.
// A thread gets a TMA instruction out only every few hundred cycles, most of them address arithmetic, and a stage has several: the
// stages rotate over the three producers and a stage's loads go out by the lanes of one.  With a thread each for a third of every
// stage's loads the 64 -> 128 channel 3x3/2 layer at batch 64 took 23.0 us (now 11.0), 512 -> 256 1x1 28 x 28 at batch 32 17.4 (9.6).
#include "eoq_device.cuh"
#include "eoq_epilogue.cuh"
#include "eoq_internal.h"

namespace eoq {

namespace {

constexpr int kMaxStages = 8;
constexpr int kProducers = 3;

// Descriptor of an MN-major operand made of sub-tiles [pixels][row_bytes], `sub_bytes` apart along M/N.
// Swizzled rows: atoms along M/N are `sub_bytes` apart (leading offset), 8-pixel groups 8*row_bytes apart
// (stride offset).  16-byte rows carry no swizzle and the two offsets swap roles.
__device__ __forceinline__ uint64_t mn_major_desc(uint32_t addr, int row_bytes, uint32_t sub_bytes)
{
    if (row_bytes == 16) return make_smem_desc(addr, 128, sub_bytes, 0);
    return make_smem_desc(addr, sub_bytes, 8u * row_bytes, layout_type_for(row_bytes));
}

__global__ void __launch_bounds__(kWgradThreads, 1)
wgrad_kernel(const __grid_constant__ WgradParams p, const __grid_constant__ CUtensorMap map_x,
             const __grid_constant__ CUtensorMap map_e)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kMaxStages + 2];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile uint32_t abort_s;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    const int px = p.pixels_per_stage;
    const uint32_t a_sub = (uint32_t)px * p.kc, b_sub = (uint32_t)px * p.nc;
    const int b_subs = p.tile_n / p.nc;
    const uint32_t a_mtile = (uint32_t)p.subs_per_mtile * a_sub;  // bytes of one M tile's activation sub-tiles
    const uint32_t stage_bytes = (uint32_t)p.mtiles_per_cta * a_mtile + (uint32_t)b_subs * b_sub;
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
    const uint32_t done_bar = bar0 + 8u * (2 * kMaxStages);

    uint32_t tmem_cols = 32;
    while (tmem_cols < (uint32_t)(p.mtiles_per_cta * p.tile_n)) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.num_stages; ++s) {
            ptx::mbar_init(full_bar(s), 1);
            ptx::mbar_init(empty_bar(s), 1);
        }
        ptx::mbar_init(done_bar, 1);
        abort_s = 0;
        ptx::fence_barrier_init();
        ptx::prefetch_tensormap(&map_x);
        ptx::prefetch_tensormap(&map_e);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&tmem_base_s), tmem_cols);
        ptx::tmem_relinquish();
    }
    // work unit of this CTA
    const int tiles = p.num_m_groups * p.num_n_tiles;
    const int ks = blockIdx.x / tiles, tile = blockIdx.x % tiles;
    const int mt0 = (tile / p.num_n_tiles) * p.mtiles_per_cta, nt = tile % p.num_n_tiles;
    const int my_mtiles = min(p.mtiles_per_cta, p.num_m_tiles - mt0);  // M tiles this CTA accumulates
    const int total_subs = p.ntaps * p.chunks_per_tap;
    int subs_total = 0;  // activation sub-tiles this CTA loads per stage
    for (int jm = 0; jm < my_mtiles; ++jm) subs_total += min(p.subs_per_mtile, total_subs - (mt0 + jm) * p.subs_per_mtile);
    const int q_begin = ks * p.stages_per_split * px;
    int my_stages = p.stages_per_split;
    {
        const int remaining = (p.P - q_begin + px - 1) / px;
        my_stages = remaining < my_stages ? remaining : my_stages;
        if (my_stages < 0) my_stages = 0;
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    // Everything up to here touched no global memory.  Behind the layer's tap sums the kernels that wrote the operands are complete
    // already (they were when the tap sums let this launch in), and the tap sums write nothing that it reads.
    if (!p.wait_late) ptx::grid_dep_wait();
    if (p.launch_early) ptx::grid_dep_launch();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < p.zero_n16; i += gridDim.x * blockDim.x) p.zero[i] = make_int4(0, 0, 0, 0);
    const uint32_t tmem_base = tmem_base_s;
    const RoleCtx ctx{&abort_s, p.dev};

    if (warp == 0 || warp == 2 || warp == 3) {
        // Producer q fills the stages q, q + 3, q + 6, ... of the CTA's range; the loads of a stage (activation sub-tiles first, then
        // the error sub-tiles) are spread over its lanes, whose sub-tiles are the same in every stage.
        const int q = warp == 0 ? 0 : warp - 1;
        const int n_ops = subs_total + b_subs;
        auto place = [&](int o, int &tap, int &chunk) -> uint32_t {   // an activation sub-tile's tap and channels, its place in a stage
            const int jm = o / p.subs_per_mtile, s = mt0 * p.subs_per_mtile + o;
            tap = s / p.chunks_per_tap;
            chunk = s - tap * p.chunks_per_tap;
            return jm * a_mtile + (o - jm * p.subs_per_mtile) * a_sub;
        };
        int tap0 = 0, chunk0 = 0;
        uint32_t place0 = 0;
        if (lane < subs_total) place0 = place(lane, tap0, chunk0);
        const uint32_t bytes = subs_total * a_sub + b_subs * b_sub;
        int stage = q % p.num_stages;
        uint32_t phase = (uint32_t)(q / p.num_stages) & 1u, inflight = 0, inflight_parity = 0;
        bool ok = true;
        const int pix_per_img = p.ho * p.wo;
        for (int it = q; it < my_stages; it += kProducers) {
            const int q0 = q_begin + it * px;
            const int img = q0 / pix_per_img, rem = q0 - img * pix_per_img, y = rem / p.wo;
            const int cw = (rem - y * p.wo) * p.src_stride_w + p.base_w, ch = y * p.src_stride + p.base_h;
            if (!(ok = __all_sync(0xffffffffu, wait_bar(empty_bar(stage), phase ^ 1u, ctx)))) break;
            const uint32_t a_dst = smem_base + stage * stage_bytes;
            const uint32_t b_dst = a_dst + p.mtiles_per_cta * a_mtile;
            if (lane == 0) ptx::mbar_expect_tx(full_bar(stage), bytes);
            __syncwarp();
            for (int o = lane; o < n_ops; o += 32) {
                if (o < subs_total) {
                    int tap = tap0, chunk = chunk0;
                    const uint32_t at = o < 32 ? place0 : place(o, tap, chunk);
                    ptx::tma_load_im2col_4d(a_dst + at, &map_x, full_bar(stage), chunk * p.kc, cw, ch, img, (uint16_t)p.tap_dw[tap],
                                            (uint16_t)p.tap_dh[tap]);
                } else {
                    const int j = o - subs_total;
                    ptx::tma_load_2d(b_dst + j * b_sub, &map_e, full_bar(stage), nt * p.tile_n + j * p.nc, q0);
                }
            }
            inflight |= 1u << stage;
            inflight_parity = (inflight_parity & ~(1u << stage)) | (phase << stage);
            stage += kProducers;
            while (stage >= p.num_stages) { stage -= p.num_stages; phase ^= 1u; }
        }
        if (!ok && lane == 0)
            for (int s = 0; s < p.num_stages; ++s)
                if (inflight & (1u << s))
                    for (uint32_t i = 0; i < kSpinLimit; ++i)
                        if (ptx::mbar_try_wait(full_bar(s), (inflight_parity >> s) & 1u)) break;
    } else if (warp == 1) {
        // the whole warp runs the issue loop; one elected lane issues the MMAs and commits (see elect_one)
        const uint32_t leader = elect_one();
        const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
        const uint32_t idesc = make_idesc_i8(kTileM, p.tile_n, true, true);
        // descriptor halves that do not change; the loop adds row offsets to the low halves
        const uint64_t a_proto = mn_major_desc(0, p.kc, a_sub), b_proto = mn_major_desc(0, p.nc, b_sub);
        const uint32_t a_hi = (uint32_t)(a_proto >> 32), b_hi = (uint32_t)(b_proto >> 32);
        const uint32_t a_lead = (uint32_t)a_proto, b_lead = (uint32_t)b_proto;  // leading-offset field, address 0
        const uint32_t a_step16 = (32u * p.kc) >> 4, b_step16 = (32u * p.nc) >> 4;  // 32 pixels further down
        const uint32_t a_mtile16 = a_mtile >> 4;
        int stage = 0;
        uint32_t phase = 0, accumulate = 0;
        bool ok = true;
        for (int it = 0; it < my_stages; ++it) {
            if (!(ok = __all_sync(0xffffffffu, wait_bar(full_bar(stage), phase, ctx)))) break;
            ptx::tc_fence_after();
            uint32_t a_lo = ((smem_base + stage * stage_bytes) >> 4) | a_lead;
            uint32_t b_lo = (((smem_base + stage * stage_bytes) >> 4) + ((p.mtiles_per_cta * a_mtile) >> 4)) | b_lead;
            for (int k = 0; k < px; k += 32) {
                // the M tiles of the group meet the same error tile; each has its own accumulator columns
                uint32_t a_j = a_lo, d_j = tmem_base;
                for (int jm = 0; jm < my_mtiles; ++jm, a_j += a_mtile16, d_j += p.tile_n)
                    ptx::mma_i8(d_j, smem_desc_join(a_j, a_hi), smem_desc_join(b_lo, b_hi), idesc, accumulate, leader);
                accumulate = 1;
                a_lo += a_step16;
                b_lo += b_step16;
            }
            ptx::mma_commit(empty_bar(stage), leader);
            if (++stage == p.num_stages) { stage = 0; phase ^= 1u; }
        }
        ptx::mma_commit(done_bar, leader);
        if (!ok)
            for (uint32_t i = 0; i < kSpinLimit; ++i)
                if (ptx::mbar_try_wait(done_bar, 0)) break;
    } else {
        // Every lane has a row of the accumulator, neighbouring lanes neighbouring weights of one output channel: a store per
        // column and warp, 128 bytes wide.
        const int quad = warp & 3;
        int32_t *slice = p.partials + (size_t)ks * p.c_out * p.rows_total;
        const bool ok = __all_sync(0xffffffffu, wait_bar(done_bar, 0, ctx));
        if (ok) ptx::tc_fence_after();
        for (int jm = 0; jm < my_mtiles && ok; ++jm) {
            const int mt = mt0 + jm;
            int row = mt * kTileM + quad * 32 + lane;  // (tap, ic) flattened: tap * c_in + ic
            bool valid = row < p.rows_total;
            if (p.row_window_kw) {
                // filter-row path: the rows are (filter row, tap 0..7, channel): drop the padding taps
                const int per_frow = 8 * p.c_in, fr = row / per_frow, within = row % per_frow;
                const int t = within / p.c_in;
                valid = fr < p.ntaps && t < p.row_window_kw;
                row = (fr * p.row_window_kw + t) * p.c_in + within % p.c_in;
            }
            const uint32_t t_row = tmem_base + jm * p.tile_n + ((uint32_t)(quad * 32) << 16);
            for (int c0 = 0; c0 < p.tile_n; c0 += 32) {
                uint32_t r[32];
                const int oc0 = nt * p.tile_n + c0;
                const int ncol = min(min(32, p.tile_n - c0), p.c_out - oc0);   // (multiples of 16)
                if (ncol <= 0) break;
                if (ncol == 32) ptx::tmem_ld_32x32(t_row + c0, r);
                else ptx::tmem_ld_32x16(t_row + c0, r);
                ptx::tmem_ld_wait();
                if (valid) {
                    int32_t *dst = slice + (size_t)oc0 * p.rows_total + row;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < 16 || ncol == 32) dst[(size_t)j * p.rows_total] = (int32_t)r[j];
                }
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, tmem_cols);
    }
    if (p.wait_late) ptx::grid_dep_wait();   // (what comes behind this launch waits for it alone)
}

}  // namespace

size_t wgrad_smem_bytes(const WgradParams &p)
{
    const size_t stage = (size_t)p.mtiles_per_cta * p.subs_per_mtile * p.pixels_per_stage * p.kc +
                         (size_t)p.tile_n * p.pixels_per_stage;
    return stage * p.num_stages + 1024;
}

cudaError_t launch_wgrad(const WgradParams &p, const CUtensorMap &map_x, const CUtensorMap &map_e, cudaStream_t stream)
{
    static std::atomic<unsigned long long> allowed;
    const cudaError_t e = allow_smem((const void *)wgrad_kernel, 208 * 1024, allowed, true);
    if (e != cudaSuccess) return e;
    const int grid = p.num_m_groups * p.num_n_tiles * p.num_k_splits;
    const size_t need = wgrad_smem_bytes(p), least = p.wait_late ? 116 * 1024 : 0;   // (as launch_wgrad_patch)
    return launch_chained(wgrad_kernel, grid, kWgradThreads, need > least ? need : least, stream, p, map_x, map_e);
}

}  // namespace eoq
