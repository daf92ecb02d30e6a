// Weight gradient of a first layer on the filter-row path (arXiv 2105.13890, Sec. 3.2.1: g_w = Q_g(e3 * x1)): 8 input channels,
// filters 5 to 8 taps wide.  The activation operand of filter row fr is the row of 8-pixel windows stride * y - pad + fr, and
// consecutive output rows share all but `stride` of their window rows: these stay in a ring in shared memory, so an output row
// loads `stride` window rows and its error row instead of kh window rows.  TMA delivers a row of a tile every 3 to 5 cycles
// whatever its width, which bounded the per-tap kernel: 7 x 7 stride 2 on 224 x 224 images at batch 64, 126 us with 8 rows
// per pixel, 42 us here with 3.
// One CTA owns a range of output rows (of all images), accumulates all filter rows side by side in tensor memory and leaves
// its int32 sums in a slice of its own.  An M tile is two filter rows of 64 bytes (two ring slots, adjacent because windows start
// at even slots and the ring is even).
// Roles: warps 0, 2, 3 TMA producers, warp 1 MMA issuer and TMEM owner, warps 4-7 epilogue.  All waits are bounded.
#include "eoq_device.cuh"
#include "eoq_epilogue.cuh"
#include "eoq_internal.h"

namespace eoq {

namespace {

constexpr int kMaxStages = 4;
constexpr int kProducers = 3;

// Position in the CTA's range of output rows: (image, row) and the ring slot its first window row sits in.
struct RowWalk {
    int img, y, slot, first_new;   // first_new: filter row of the first window row that is not in the ring yet
    __device__ __forceinline__ RowWalk(const WgradRowsPlan &pl, int row) : img(row / pl.ho), y(row % pl.ho), slot(0), first_new(0) {}
    __device__ __forceinline__ void next(const WgradRowsPlan &pl)
    {
        if (++y == pl.ho) {
            y = 0;
            ++img;
            slot += pl.span;
            first_new = 0;
        } else {
            slot += pl.stride;
            first_new = max(0, pl.kh - pl.stride);
        }
        while (slot >= pl.slots) slot -= pl.slots;
    }
};

__global__ void __launch_bounds__(kWgradThreads, 1)
wgrad_rows_kernel(const __grid_constant__ WgradRowsPlan pl, const __grid_constant__ CUtensorMap map_x,
                  const __grid_constant__ CUtensorMap map_e)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kMaxStages + 1];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile uint32_t abort_s;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t slot_bytes = (uint32_t)(pl.kp * pl.kc), e_sub = (uint32_t)(pl.kp * pl.nc), e_bytes = (uint32_t)(pl.kp * pl.c_out);
    const uint32_t e_base = smem_base + (uint32_t)pl.slots * slot_bytes;
    const int e_subs = pl.c_out / pl.nc;
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
    const uint32_t done_bar = bar0 + 8u * (2 * kMaxStages);
    uint32_t tmem_cols = 32;
    while (tmem_cols < (uint32_t)(pl.mtiles * pl.c_out)) tmem_cols <<= 1;

    const int row_begin = blockIdx.x * pl.rows_per_split, row_end = min(pl.n_img * pl.ho, row_begin + pl.rows_per_split);

    // The error buffers' pixels between wo and kp are never written by a load: clear them once, so that the rounded-up tail of
    // the reduction adds nothing (whatever the window rows hold there).
    {
        const int tail = (pl.kp - pl.wo) * pl.nc;
        for (int s = 0; s < pl.num_stages * e_subs; ++s) {
            uint8_t *p = smem_raw + (e_base - ptx::smem_u32(smem_raw)) + s * e_sub + pl.wo * pl.nc;
            for (int i = threadIdx.x * 16; i < tail; i += blockDim.x * 16) *reinterpret_cast<int4 *>(p + i) = make_int4(0, 0, 0, 0);
        }
        ptx::fence_proxy_async();
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < pl.num_stages; ++s) {
            ptx::mbar_init(full_bar(s), kProducers);   // every producer announces its share of the row's bytes
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
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    ptx::grid_dep_wait();   // everything up to here touched no global memory
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < pl.zero_n16; i += gridDim.x * blockDim.x) pl.zero[i] = make_int4(0, 0, 0, 0);
    const uint32_t tmem_base = tmem_base_s;
    const RoleCtx ctx{&abort_s, pl.dev};

    if (warp == 0 || warp == 2 || warp == 3) {
        if (lane == 0) {
            // producer q issues the loads number q, q + 3, q + 6, ... of every output row (new window rows, then the error)
            const int q = warp == 0 ? 0 : warp - 1;
            int stage = 0;
            uint32_t phase = 0, inflight = 0, inflight_parity = 0;
            bool ok = true;
            RowWalk w(pl, row_begin);
            for (int row = row_begin; row < row_end; ++row, w.next(pl)) {
                // A stage comes free when the row num_stages earlier is through: the ring then holds the window rows of all
                // rows since (plan_wgrad_rows).
                if (!(ok = wait_bar<32>(empty_bar(stage), phase ^ 1u, ctx))) break;
                const int fresh = pl.kh - w.first_new, n_ops = fresh + e_subs;
                uint32_t bytes = 0;
                for (int o = q; o < n_ops; o += kProducers) bytes += (uint32_t)(pl.wo * (o < fresh ? pl.kc : pl.nc));
                ptx::mbar_expect_tx(full_bar(stage), bytes);
                for (int o = q; o < n_ops; o += kProducers) {
                    if (o < fresh) {
                        const int fr = w.first_new + o;
                        int slot = w.slot + fr;
                        if (slot >= pl.slots) slot -= pl.slots;
                        ptx::tma_load_im2col_4d(smem_base + slot * slot_bytes, &map_x, full_bar(stage), 0, 0, w.y * pl.stride - pl.pad, w.img,
                                                0, (uint16_t)fr);
                    } else {
                        const int j = o - fresh;
                        ptx::tma_load_2d(e_base + stage * e_bytes + j * e_sub, &map_e, full_bar(stage), j * pl.nc, row * pl.wo);
                    }
                }
                inflight |= 1u << stage;
                inflight_parity = (inflight_parity & ~(1u << stage)) | (phase << stage);
                if (++stage == pl.num_stages) { stage = 0; phase ^= 1u; }
            }
            if (!ok)
                for (int s = 0; s < pl.num_stages; ++s)
                    if (inflight & (1u << s))
                        for (uint32_t i = 0; i < kSpinLimit; ++i)
                            if (ptx::mbar_try_wait(full_bar(s), (inflight_parity >> s) & 1u)) break;
        }
    } else if (warp == 1) {
        // the whole warp runs the issue loop; one elected lane issues the MMAs and commits (see elect_one)
        const uint32_t leader = elect_one();
        const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
        const uint32_t idesc = make_idesc_i8(kTileM, pl.c_out, true, true);
        // MN-major descriptors: the two filter rows of an M tile are one slot apart, 8-pixel groups 8 rows apart
        const uint32_t a_hi = smem_desc_hi(8u * pl.kc, layout_type_for(pl.kc)), b_hi = smem_desc_hi(8u * pl.nc, layout_type_for(pl.nc));
        const uint32_t a_lead = ((slot_bytes >> 4) & 0x3FFFu) << 16, b_lead = ((e_sub >> 4) & 0x3FFFu) << 16;
        const uint32_t a_step16 = (32u * pl.kc) >> 4, b_step16 = (32u * pl.nc) >> 4, slot16 = slot_bytes >> 4;
        const int k_steps = pl.kp / 32, per_tile = kTileM / pl.kc;
        int stage = 0;
        uint32_t phase = 0, accumulate = 0;
        bool ok = true;
        RowWalk w(pl, row_begin);
        for (int row = row_begin; row < row_end; ++row, w.next(pl)) {
            if (!(ok = __all_sync(0xffffffffu, wait_bar(full_bar(stage), phase, ctx)))) break;
            ptx::tc_fence_after();
            uint32_t b_lo = ((e_base + stage * e_bytes) >> 4) | b_lead;
            for (int k = 0; k < k_steps; ++k, b_lo += b_step16) {
                int slot = w.slot;
                uint32_t d = tmem_base;
                for (int j = 0; j < pl.mtiles; ++j, d += pl.c_out) {
                    const uint32_t a_lo = ((smem_base >> 4) + slot * slot16 + k * a_step16) | a_lead;
                    ptx::mma_i8(d, smem_desc_join(a_lo, a_hi), smem_desc_join(b_lo, b_hi), idesc, accumulate, leader);
                    slot += per_tile;
                    if (slot >= pl.slots) slot -= pl.slots;
                }
                accumulate = 1;
            }
            ptx::mma_commit(empty_bar(stage), leader);
            if (++stage == pl.num_stages) { stage = 0; phase ^= 1u; }
        }
        ptx::mma_commit(done_bar, leader);
        ptx::grid_dep_launch();   // what remains is the epilogue
        if (!ok)
            for (uint32_t i = 0; i < kSpinLimit; ++i)
                if (ptx::mbar_try_wait(done_bar, 0)) break;
    } else {
        const int quad = warp & 3;
        int32_t *slice = pl.partials + (size_t)blockIdx.x * pl.c_out * pl.rows_total;
        const bool ok = __all_sync(0xffffffffu, wait_bar<64>(done_bar, 0, ctx));
        if (ok) ptx::tc_fence_after();
        for (int j = 0; j < pl.mtiles && ok; ++j) {
            // rows of the accumulator: (filter row, tap 0..7, channel); the padding taps and rows are dropped
            const int r = j * kTileM + quad * 32 + lane, fr = r / pl.kc, within = r % pl.kc, tap = within / pl.c_in;
            const bool valid = fr < pl.kh && tap < pl.kw;
            int32_t *dst = slice + (size_t)(fr * pl.kw + tap) * pl.c_in + within % pl.c_in;
            const uint32_t t_row = tmem_base + j * pl.c_out + ((uint32_t)(quad * 32) << 16);
            for (int c0 = 0; c0 < pl.c_out; c0 += 16) {
                uint32_t v[32];
                ptx::tmem_ld_32x16(t_row + c0, v);
                ptx::tmem_ld_wait();
                if (valid) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) dst[(size_t)(c0 + i) * pl.rows_total] = (int32_t)v[i];
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
}

}  // namespace

size_t wgrad_rows_smem_bytes(const WgradRowsPlan &pl)
{
    return (size_t)pl.slots * pl.kp * pl.kc + (size_t)pl.num_stages * pl.kp * pl.c_out + 1024;
}

cudaError_t launch_wgrad_rows(const WgradRowsPlan &pl, const CUtensorMap &map_x, const CUtensorMap &map_e, cudaStream_t stream)
{
    static std::atomic<unsigned long long> allowed;
    const cudaError_t e = allow_smem((const void *)wgrad_rows_kernel, 208 * 1024, allowed);
    if (e != cudaSuccess) return e;
    return launch_chained(wgrad_rows_kernel, pl.num_splits, kWgradThreads, wgrad_rows_smem_bytes(pl), stream, pl, map_x, map_e);
}

}  // namespace eoq
