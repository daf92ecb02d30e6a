// Forward convolution of a first layer with wide filters on few channels (stride * c_in = 16 bytes: the 7x7/2 layer on 8 channels;
// arXiv 2105.13890, Sec. 3.2.1).
//
// The im2col kernel fetches every filter row of every output pixel as a TMA row of its own (64 bytes, 7 of them per pixel), and the
// TMA's rows bound it: 7x7/2 on 224 x 224 images at batch 64 took 79 us.  Here neighbouring output pixels' windows start 16 bytes
// apart in an input row, which is just the distance between the rows of a core matrix without swizzle: eight pixels' 16-byte chunks
// are 128 contiguous bytes, the next chunk of the same pixels starts 16 bytes further.  So a descriptor with a leading offset of 16
// and a stride offset of 128 bytes reads the windows out of the input row as it lies in memory, overlaps and all, and a patch of
// (r - 1) * stride + kh input rows, one TMA box, serves r output rows.  An M tile is one output row; rows of
// more than 125 pixels (8 channels; 121 with 16) are cut into several tiles (plan_rows; at most 128 output channels).  What
// bounds it now is the MMAs (two per filter row and tile, about 60 cycles each) and the epilogue: 224 x 224 images at batch 64
// 77.8 -> 35.0 us, 178 x 178 at batch 13 14.5 -> 9.7, one 224 x 224 image 5.6 -> 4.2 (back to back).
//
// Roles: warp 0 patch loads, warp 1 TMEM owner + tcgen05.mma issuer, warp 2 weights (resident), warps 4-19 epilogue (as in the patch
// kernel).  All waits are bounded.
#include "eoq_device.cuh"
#include "eoq_epilogue.cuh"
#include "eoq_internal.h"

namespace eoq {

namespace {

constexpr int kMaxPatches = 4;

// A CTA's sequence of patches, blockIdx, blockIdx + grid, ...: image, block of output rows, column tile, carried from patch to patch
// (the divisions stay out of the MMA issuer's loop).
struct PatchWalk {
    int patch, img, yb, xt;
    int step_img, step_yb, step_xt;
    __device__ __forceinline__ explicit PatchWalk(const RowsPlan &pl) : patch((int)blockIdx.x)
    {
        auto split = [&](int v, int &i, int &y, int &x) {
            const int rows = pl.x_tiles == 1 ? v : v / pl.x_tiles;
            x = v - rows * pl.x_tiles;
            i = rows / pl.row_blocks;
            y = rows - i * pl.row_blocks;
        };
        split(patch, img, yb, xt);
        split((int)gridDim.x, step_img, step_yb, step_xt);
    }
    __device__ __forceinline__ void next(const RowsPlan &pl)
    {
        patch += gridDim.x;
        xt += step_xt;
        yb += step_yb;
        img += step_img;
        if (xt >= pl.x_tiles) { xt -= pl.x_tiles; ++yb; }
        if (yb >= pl.row_blocks) { yb -= pl.row_blocks; ++img; }
    }
};

__global__ void __launch_bounds__(kPatchThreads, 1)
igemm_rows_kernel(const __grid_constant__ IgemmParams p, const __grid_constant__ RowsPlan pl, const __grid_constant__ CUtensorMap map_a,
                  const __grid_constant__ CUtensorMap map_b)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kMaxPatches + 1 + 9];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile uint32_t abort_s;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t b_sub = (uint32_t)p.tile_n * p.kc;
    const uint32_t a_region = smem_base + (uint32_t)p.ntaps * b_sub;   // the weights first: their swizzle wants the alignment
    const uint32_t table_off = (uint32_t)p.ntaps * b_sub + (uint32_t)pl.num_a * pl.a_bytes + pl.slack;
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto a_full = [&](int s) { return bar0 + 8u * s; };
    auto a_empty = [&](int s) { return bar0 + 8u * (kMaxPatches + s); };
    const uint32_t b_full = bar0 + 8u * (2 * kMaxPatches);
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * kMaxPatches + 1 + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * kMaxPatches + 5 + a); };
    const uint32_t drain_bar = bar0 + 8u * (2 * kMaxPatches + 9);

    uint32_t acc_stride = 32;
    while (acc_stride < (uint32_t)p.tile_n) acc_stride <<= 1;
    const uint32_t buf_stride = 2 * acc_stride;   // two partial accumulators that successive MMAs alternate between
    const uint32_t tmem_cols = p.ep_groups * buf_stride;

    if (threadIdx.x == 0) {
        for (int s = 0; s < pl.num_a; ++s) {
            ptx::mbar_init(a_full(s), 1);
            ptx::mbar_init(a_empty(s), 1);
        }
        ptx::mbar_init(b_full, 1);
        for (int a = 0; a < p.ep_groups; ++a) {
            ptx::mbar_init(tfull_bar(a), 1);
            ptx::mbar_init(tempty_bar(a), kEpilogueWarps / p.ep_groups);
        }
        ptx::mbar_init(drain_bar, 1);
        abort_s = 0;
        ptx::fence_barrier_init();
        ptx::prefetch_tensormap(&map_a);
        ptx::prefetch_tensormap(&map_b);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&tmem_base_s), tmem_cols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    ptx::grid_dep_wait();   // everything up to here touched no global memory
    const uint32_t tmem_base = tmem_base_s;
    const RoleCtx ctx{&abort_s, p.dev};
    const int patches = pl.n_img * pl.row_blocks * pl.x_tiles;

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------------------------------------------ patch loads
            int ia = 0;
            uint32_t pha = 0, inflight = 0, inflight_parity = 0;
            bool ok = true;
            for (PatchWalk at(pl); at.patch < patches; at.next(pl)) {
                if (!(ok = wait_bar<64>(a_empty(ia), pha ^ 1u, ctx))) break;
                ptx::mbar_expect_tx(a_full(ia), (uint32_t)pl.a_box_bytes);
                // columns in 8-byte units from the first window's start; rows outside the image arrive as zeros
                ptx::tma_load_3d(a_region + ia * pl.a_bytes, &map_a, a_full(ia), pl.first_col8 + at.xt * pl.tile_px * 2,
                                 at.yb * pl.r_rows * pl.stride - pl.pad, at.img);
                inflight |= 1u << ia;
                inflight_parity = (inflight_parity & ~(1u << ia)) | (pha << ia);
                if (++ia == pl.num_a) { ia = 0; pha ^= 1u; }
            }
            if (!ok)
                for (int s = 0; s < pl.num_a; ++s)
                    if (inflight & (1u << s))
                        for (uint32_t i = 0; i < kSpinLimit; ++i)
                            if (ptx::mbar_try_wait(a_full(s), (inflight_parity >> s) & 1u)) break;
        }
    } else if (warp == 2) {
        // ---------------------------------------------------------------------- weights: a filter row of all columns per load
        if (lane == 0) ptx::mbar_expect_tx(b_full, (uint32_t)p.ntaps * b_sub);
        __syncwarp();
        if (lane < p.ntaps) ptx::tma_load_3d(smem_base + lane * b_sub, &map_b, b_full, 0, lane, 0);
        // completion is observed by the MMA thread, which every path out of this kernel waits for
    } else if (warp == 1) {
        // ---------------------------------------------------------------------- MMA issuer (whole warp, see elect_one)
        const uint32_t leader = elect_one();
        const uint32_t tmem_d = __shfl_sync(0xffffffffu, tmem_base_s, 0);
        const uint32_t idesc = make_idesc_i8(kTileM, p.tile_n, false, false);
        const uint32_t a_hi = smem_desc_hi(128, 0), b_hi = smem_desc_hi(8u * p.kc, layout_type_for(p.kc));
        const uint32_t a_lead = (16u >> 4) << 16;
        const uint32_t row16 = (uint32_t)pl.row_pitch >> 4, b_sub16 = b_sub >> 4, b_lo0 = smem_base >> 4;
        int ia = 0, acc = 0;
        uint32_t pha = 0, acc_phase = 0;
        bool ok = __all_sync(0xffffffffu, wait_bar(b_full, 0, ctx));
        for (PatchWalk at(pl); at.patch < patches && ok; at.next(pl)) {
            const int rows = min(pl.r_rows, p.hq - at.yb * pl.r_rows);
            if (!(ok = __all_sync(0xffffffffu, wait_bar(a_full(ia), pha, ctx)))) break;
            uint32_t a_row = (((a_region + ia * pl.a_bytes) >> 4) | a_lead);
            for (int yl = 0; yl < rows; ++yl, a_row += pl.stride * row16) {
                if (!(ok = __all_sync(0xffffffffu, wait_bar(tempty_bar(acc), acc_phase ^ 1u, ctx)))) break;
                ptx::tc_fence_after();
                const uint32_t d0 = tmem_d + acc * buf_stride, d1 = d0 + acc_stride;
                uint32_t a_lo = a_row, b_lo = b_lo0, fresh = 1u;
                if (p.kc == 64 && p.ntaps == 7) {
#pragma unroll
                    for (int t = 0; t < 7; ++t)
                        mma_k_steps<2>(d0, d1, a_lo + t * row16, b_lo + t * b_sub16, a_hi, idesc, 0, t == 0, t == 0, leader, b_hi, 2u);
                } else if (p.kc == 64) {
                    for (int t = 0; t < p.ntaps; ++t, a_lo += row16, b_lo += b_sub16) {
                        mma_k_steps<2>(d0, d1, a_lo, b_lo, a_hi, idesc, 0, fresh, fresh, leader, b_hi, 2u);
                        fresh = 0;
                    }
                } else {
                    for (int t = 0; t < p.ntaps; ++t, a_lo += row16, b_lo += b_sub16) {
                        mma_k_steps<4>(d0, d1, a_lo, b_lo, a_hi, idesc, 0, fresh, fresh, leader, b_hi, 2u);
                        fresh = 0;
                    }
                }
                ptx::mma_commit(tfull_bar(acc), leader);
                if (++acc == p.ep_groups) { acc = 0; acc_phase ^= 1u; }
            }
            if (ok) ptx::mma_commit(a_empty(ia), leader);
            if (++ia == pl.num_a) { ia = 0; pha ^= 1u; }
        }
        ptx::grid_dep_launch();   // what remains is the epilogue of the last tiles
        if (!ok) {
            ptx::mma_commit(drain_bar, leader);
            for (uint32_t i = 0; i < kSpinLimit; ++i)
                if (ptx::mbar_try_wait(drain_bar, 0)) break;
            for (uint32_t i = 0; i < kSpinLimit; ++i)
                if (ptx::mbar_try_wait(b_full, 0)) break;
        }
    } else if (warp >= 4) {
        // ---------------------------------------------------------------------- epilogue (see the patch kernel)
        const int quad = warp & 3;
        const int ew = (warp - 4) >> 2;
        const int parts = 4 / p.ep_groups, grp = ew / parts, part = ew - grp * parts;
        const int row = quad * 32 + lane;
        const int groups = p.tile_n / 16;
        const int g_begin = (groups * part) / parts, g_end = (groups * (part + 1)) / parts;
        const FwdScalars fs = load_fwd_scalars(p);
        const int32_t *ts = stage_b1_table(p, fs.b1, smem_raw + (smem_base - ptx::smem_u32(smem_raw)) + table_off, (int)threadIdx.x - 128,
                                           32 * kEpilogueWarps);
        const int shift = input_shift(p);
        const FwdShift sh = forward_shift(p, fs, shift);
        uint32_t acc_phase = 0;
        int turn = grp;   // tiles until this group's next one
        bool ok = true;
        for (PatchWalk at(pl); at.patch < patches && ok; at.next(pl)) {
            const int y0 = at.yb * pl.r_rows, rows = min(pl.r_rows, p.hq - y0), x = at.xt * pl.tile_px + row;
            const bool in_row = row < pl.tile_px && x < p.wq;
            for (int yl = 0; yl < rows; ++yl) {
                if (turn-- != 0) continue;
                turn = p.ep_groups - 1;
                const int y = y0 + yl;
                size_t pix = 0;
                int cls = 0;
                if (in_row) {
                    pix = ((size_t)at.img * p.hq + y) * p.wq + x;
                    if (p.b1_table)
                        cls = border_class(y, p.hq, p.b1_nlo_h, p.b1_nhi_h, p.b1_nrc) * p.b1_ncc +
                              border_class(x, p.wq, p.b1_nlo_w, p.b1_nhi_w, p.b1_ncc);
                }
                int col = g_begin * 16;
                size_t off = pix * p.N + col;
                const int4 zero4 = make_int4(0, 0, 0, 0);
                const int32_t *tb = ts ? ts + cls * p.N + col : nullptr;
                const int32_t *tg = (!ts && p.b1_table) ? p.b1_table + (size_t)cls * p.N + col : nullptr;
                if (!(ok = __all_sync(0xffffffffu, wait_bar<64>(tfull_bar(grp), acc_phase, ctx)))) break;
                ptx::tc_fence_after();
                const uint32_t t_row = tmem_base + grp * buf_stride + ((uint32_t)(quad * 32) << 16);
                for (int g = g_begin; g < g_end; ++g, col += 16, off += 16) {
                    uint32_t r[32], r2[32];
                    ptx::tmem_ld_32x16(t_row + g * 16, r);
                    ptx::tmem_ld_32x16(t_row + acc_stride + g * 16, r2);
                    const int4 sc = in_row && p.shortcut ? __ldg(reinterpret_cast<const int4 *>(p.shortcut + off)) : zero4;
                    ptx::tmem_ld_wait();
                    if (in_row) forward_group(p, fs, sh, r, r2, 2u, off, tb, tg, sc, shift);
                    if (tb) tb += 16;
                    if (tg) tg += 16;
                }
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(tempty_bar(grp));
                acc_phase ^= 1u;
            }
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, tmem_cols);
    }
}

}  // namespace

size_t igemm_rows_smem_bytes(const IgemmParams &p, const RowsPlan &pl)
{
    return (size_t)p.ntaps * p.tile_n * p.kc + (size_t)pl.num_a * pl.a_bytes + pl.slack + 1024 + kTableSmemBytes;
}

cudaError_t launch_igemm_rows(const IgemmParams &p, const RowsPlan &pl, const CUtensorMap &map_a, const CUtensorMap &map_b, int grid,
                              cudaStream_t stream)
{
    static std::atomic<unsigned long long> allowed;
    const cudaError_t e = allow_smem((const void *)igemm_rows_kernel, 226 * 1024, allowed);
    if (e != cudaSuccess) return e;
    return launch_chained(igemm_rows_kernel, grid, kPatchThreads, igemm_rows_smem_bytes(p, pl), stream, p, pl, map_a, map_b);
}

}  // namespace eoq
