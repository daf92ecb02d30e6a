// Implicit-GEMM convolution kernel for sm_100a: forward pass and error back-propagation of the EOQ layer
// (arXiv 2105.13890, Sec. 3.2.1).  One persistent CTA per SM walks 128-row output tiles:
//   warps 0, 2, 3: TMA producers (im2col loads of the activation/error operand, tiled loads of the weights); a
//              thread gets a TMA instruction out only every few hundred cycles, most of them address arithmetic, but
//              threads issue side by side: the pipeline stages rotate over three warps, a stage's loads over their lanes
//   warp 1       : owns tensor memory, issues tcgen05.mma kind::i8 (int8 x int8 -> int32 in TMEM)
//   warps 4-19   : epilogue; read the accumulators with tcgen05.ld and apply the layer's quantizers in registers
// Up to four accumulator buffers in TMEM let the epilogue of a tile overlap the main loops of the next ones.
// Every wait is bounded: when one runs out the CTA raises EOQ_DEV_TIMEOUT, drains and returns.
#include "eoq_device.cuh"
#include "eoq_epilogue.cuh"
#include "eoq_internal.h"

namespace eoq {

namespace {

constexpr int kMaxStages = 8;
constexpr int kProducers = 3;

// kEpi: EpilogueKind; forward and dgrad are kernels of their own (registers, code size).
// kSplit: a cluster of p.split CTAs shares one tile.  Each runs its part of the reduction, hands every other CTA the partial
// sums of that CTA's share of the (column group, pixel) pairs through distributed shared memory, and takes the epilogue of its own
// share.  Small batches leave a handful of tiles with long reductions: the 512-channel 7 x 7 layer at batch 1 took 13.3 us on
// 4 CTAs.  The exchange is the price, bound by distributed shared memory: with whole tiles of 128 rows exchanged by columns it was
// 3.5 us of that layer's 7.4 on 32 CTAs; of the 49 pixels that exist it takes about 1 us.
// `block` of `grid`: the calling CTA among those that walk this GEMM's tiles.
template <int kEpi, bool kSplit>
__device__ __forceinline__ void igemm_body(const IgemmParams &p, const CUtensorMap &map_a, const CUtensorMap &map_b, const int block, const int grid)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kMaxStages + 9];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile uint32_t abort_s;

    const int warp = warp_index_uniform(), lane = threadIdx.x & 31;
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_sub = (uint32_t)kTileM * p.kc, b_sub = (uint32_t)p.tile_n * p.kc;
    const uint32_t stage_bytes = (uint32_t)p.subs_per_stage * (a_sub + b_sub);
    // Weights read MN-major: a sub-tile is atoms of kc rows of b_row bytes, `b_atom` bytes apart along the columns, and the next
    // sub-tile lies `b_next` bytes further.  With 16 rows an MMA spans two sub-tiles, so those of a stage share their atoms (rows of
    // one sub-tile behind those of the other) and the K groups of an MMA keep one distance.
    const bool b_shared = p.b_mn && p.kc == 16;
    const uint32_t b_atom = (uint32_t)(b_shared ? p.subs_per_stage * 16 : p.kc) * p.b_row, b_next = b_shared ? 16u * p.b_row : b_sub;
    const uint32_t bar0 = ptx::smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * kMaxStages + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * kMaxStages + 4 + a); };
    const uint32_t drain_bar = bar0 + 8u * (2 * kMaxStages + 8);

    uint32_t acc_stride = 32;
    while (acc_stride < (uint32_t)p.tile_n) acc_stride <<= 1;
    // Tiles up to 128 columns keep two partial accumulators that successive MMAs alternate between (summed
    // exactly in the epilogue), which removes the wait of an MMA on its predecessor's write-back.
    const uint32_t nacc = (p.tile_n <= 128 && p.kc >= 32 && p.num_sub * (p.kc / 32) >= 2) ? 2u : 1u;
    const uint32_t buf_stride = nacc * acc_stride;
    const uint32_t tmem_cols = p.ep_groups * buf_stride;

    if (kSplit) ptx::cluster_arrive();   // met below: the other blocks must have started before their shared memory is written
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.num_stages; ++s) {
            ptx::mbar_init(full_bar(s), 1);
            ptx::mbar_init(empty_bar(s), 1);
        }
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
    const int num_tiles = p.num_m_tiles * p.num_n_tiles;
    const int k_iters = (p.num_sub + p.subs_per_stage - 1) / p.subs_per_stage;
    const int pix_per_img = p.hq * p.wq;
    // Every CTA walks the reduction from another starting point (the integer sums do not depend on the order): in step, all
    // CTAs of a column tile would ask the same L2 slices for the same weights at the same time.
    // A cluster divides the iterations instead.
    const int rank = kSplit ? (int)((unsigned)block % (unsigned)p.split) : 0;
    const int k_first = kSplit ? k_iters * rank / p.split : (int)((unsigned)block % (unsigned)k_iters);
    const int k_count = kSplit ? k_iters * (rank + 1) / p.split - k_first : k_iters;
    const int tile_first = kSplit ? block / p.split : block;   // (a cluster has one tile)

    // where a tile's loads start; of the first tile while the kernels in front still run
    struct Source {
        int nt, img, cw, ch;
    };
    auto source_of = [&](int tile) {
        const int mt = tile / p.num_n_tiles, m0 = mt * kTileM, img = m0 / pix_per_img, rem = m0 - img * pix_per_img, y = rem / p.wq;
        return Source{tile - mt * p.num_n_tiles, img, (rem - y * p.wq) * p.src_stride_w + p.base_w, y * p.src_stride + p.base_h};
    };
    const bool producer = warp == 0 || warp == 2 || warp == 3;
    Source at = {};
    if (producer) at = source_of(tile_first);

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (kSplit) ptx::cluster_wait();
    ptx::grid_dep_wait();   // everything up to here touched no global memory
    if (kEpi == kEpiDgrad && blockIdx.x == 0 && threadIdx.x < 4 && p.zero_sums[threadIdx.x]) *p.zero_sums[threadIdx.x] = 0;
    const uint32_t tmem_base = tmem_base_s;
    const RoleCtx ctx{&abort_s, p.dev};

    if (producer) {
        // ------------------------------------------------------------------ TMA producers
        // producer q fills the pipeline slots q, q + 3, q + 6, ... of the CTA's sequence of (tile, k iteration); the loads of a slot
        // are spread over its lanes (what a thread computes between two loads is most of a load's time)
        const int q = warp == 0 ? 0 : warp - 1;
        const int atoms = p.b_mn ? p.tile_n / p.b_row : 1;
        int stage = q % p.num_stages;
        uint32_t phase = (uint32_t)(q / p.num_stages) & 1u;
        int turn = q;  // slots until this producer's next one
        uint32_t inflight = 0, inflight_parity = 0;
        bool ok = true;
        for (int tile = tile_first; tile < num_tiles && ok;) {
            for (int step = 0, kit = k_first; step < k_count; ++step, kit = kit + 1 == k_iters ? 0 : kit + 1) {
                if (turn-- != 0) continue;
                turn = kProducers - 1;
                if (!(ok = __all_sync(0xffffffffu, wait_bar<32>(empty_bar(stage), phase ^ 1u, ctx)))) break;
                const int s0 = kit * p.subs_per_stage;
                const int subs = min(p.subs_per_stage, p.num_sub - s0);
                const uint32_t a_dst = smem_base + stage * stage_bytes;
                const uint32_t b_dst = a_dst + p.subs_per_stage * a_sub;
                if (lane == 0) ptx::mbar_expect_tx(full_bar(stage), subs * ((uint32_t)p.a_rows * p.kc + b_sub));
                __syncwarp();
                for (int i = lane; i < subs * (1 + atoms); i += 32) {
                    const int j = i < subs ? i : (i - subs) / atoms;
                    const int s = s0 + j;
                    const int sd = min(s, p.real_sub - 1);  // a padding sub-tile re-reads real data; its weights are zero
                    const int tap = sd / p.chunks_per_tap, chunk = sd - tap * p.chunks_per_tap;
                    if (i < subs) {
                        ptx::tma_load_im2col_4d(a_dst + j * a_sub, &map_a, full_bar(stage), chunk * p.kc, at.cw, at.ch, at.img,
                                                (uint16_t)p.tap_dw[tap], (uint16_t)p.tap_dh[tap]);
                    } else if (p.b_mn) {
                        // weights in place, [reduction rows][tap][columns]: tile_n / b_row atoms of [kc rows][b_row bytes]; zeros
                        // for a padding sub-tile, as below
                        const int a = i - subs - j * atoms;
                        ptx::tma_load_3d(b_dst + j * b_next + a * b_atom, &map_b, full_bar(stage), at.nt * p.tile_n + a * p.b_row,
                                         s < p.real_sub ? (int)p.tap_b[tap] : 0x7fff, chunk * p.kc);
                    } else {
                        // tap coordinate p.ntaps lies outside the weight tensor: the padding sub-tile is zero-filled
                        ptx::tma_load_3d(b_dst + j * b_sub, &map_b, full_bar(stage), chunk * p.kc,
                                         s < p.real_sub ? (int)p.tap_b[tap] : 0x7fff, at.nt * p.tile_n);
                    }
                }
                inflight |= 1u << stage;
                inflight_parity = (inflight_parity & ~(1u << stage)) | (phase << stage);
                stage += kProducers;
                while (stage >= p.num_stages) { stage -= p.num_stages; phase ^= 1u; }
            }
            tile += grid;
            if (tile < num_tiles) at = source_of(tile);
        }
        if (!ok && lane == 0) {
            // wait, bounded, for the copies this warp still has in flight
            for (int s = 0; s < p.num_stages; ++s)
                if (inflight & (1u << s))
                    for (uint32_t i = 0; i < kSpinLimit; ++i)
                        if (ptx::mbar_try_wait(full_bar(s), (inflight_parity >> s) & 1u)) break;
        }
        if (kSplit) ptx::cluster_sync();
    } else if (warp == 1) {
        // the whole warp runs the issue loop; one elected lane issues the MMAs and commits (see elect_one)
        const uint32_t leader = elect_one();
        const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_s, 0);
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t idesc = make_idesc_i8(kTileM, p.tile_n, false, p.b_mn != 0);
        // Descriptors are assembled from precomputed halves; the loop only adds offsets in 16-byte units.
        // kc >= 32: swizzled K-major sub-tiles, rows kc bytes wide, 8-row groups 8*kc apart; a 32-byte K step
        // moves the start address inside the swizzle span.  kc == 16: no swizzle, one MMA spans two sub-tiles
        // (two taps): the second half of K sits one sub-tile further (leading offset), 8-row groups 128 B apart.
        const bool wide = p.kc >= 32;
        const uint32_t hi = wide ? smem_desc_hi(8u * p.kc, layout_type_for(p.kc)) : smem_desc_hi(128, 0);
        const uint32_t a_sub16 = a_sub >> 4, b_sub16 = b_next >> 4;
        const uint32_t a_lead = wide ? 0u : (a_sub16 << 16);
        uint32_t b_lead = wide ? 0u : (b_sub16 << 16);
        // B read MN-major: atoms b_atom apart along the columns (leading offset), 8-row groups 8 * b_row apart (stride
        // offset); 16-byte rows carry no swizzle and the two offsets swap roles; a 32-deep K step is 32 rows of an atom
        uint32_t b_hi = hi, b_k16 = 2u;
        if (p.b_mn) {
            if (p.b_row == 16) {
                b_hi = smem_desc_hi(b_atom, 0);
                b_lead = (128u >> 4) << 16;
            } else {
                b_hi = smem_desc_hi(8u * p.b_row, layout_type_for(p.b_row));
                b_lead = ((b_atom >> 4) & 0x3FFFu) << 16;
            }
            b_k16 = (32u * p.b_row) >> 4;
        }
        const int sub_step = wide ? 1 : 2, k_steps = wide ? p.kc / 32 : 1;
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        bool ok = true;
        for (int tile = tile_first; tile < num_tiles && ok; tile += grid) {
            if (!(ok = __all_sync(0xffffffffu, wait_bar(tempty_bar(acc), acc_phase ^ 1u, ctx)))) break;
            ptx::tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * buf_stride, d_other = nacc == 2 ? d_tmem + acc_stride : d_tmem;
            uint32_t accumulate = 0;
            uint32_t fresh0 = 1u, fresh1 = nacc == 2 ? 1u : 0u;
            for (int step = 0, kit = k_first; step < k_count; ++step, kit = kit + 1 == k_iters ? 0 : kit + 1) {
                if (!(ok = __all_sync(0xffffffffu, wait_bar(full_bar(stage), phase, ctx)))) break;
                ptx::tc_fence_after();
                const int subs = min(p.subs_per_stage, p.num_sub - kit * p.subs_per_stage);
                // (a descriptor's address has 14 bits; in a cluster, shared-memory addresses carry the CTA's rank above them)
                const uint32_t stage16 = ((smem_base + stage * stage_bytes) >> 4) & 0x3FFFu;
                uint32_t a_lo = stage16 | a_lead;
                uint32_t b_lo = (stage16 + p.subs_per_stage * a_sub16) | b_lead;
                if (wide && k_steps >= 2) {
                    // 2 or 4 MMAs per sub-tile, alternating between the two partial accumulators
                    for (int j = 0; j < subs; ++j) {
                        if (k_steps == 4) mma_k_steps<4>(d_tmem, d_other, a_lo, b_lo, hi, idesc, 0, fresh0, fresh1, leader, b_hi, b_k16);
                        else mma_k_steps<2>(d_tmem, d_other, a_lo, b_lo, hi, idesc, 0, fresh0, fresh1, leader, b_hi, b_k16);
                        fresh0 = 0;
                        fresh1 = 0;
                        a_lo += a_sub16;
                        b_lo += b_sub16;
                    }
                } else {
                    for (int j = 0; j < subs; j += sub_step) {
                        // one MMA per step; with two accumulators successive steps alternate
                        const bool odd = nacc == 2 && (accumulate & 2u);
                        ptx::mma_i8(odd ? d_other : d_tmem, smem_desc_join(a_lo, hi), smem_desc_join(b_lo, b_hi), idesc,
                                    odd ? (fresh1 ? 0u : 1u) : (fresh0 ? 0u : 1u), leader);
                        if (odd) fresh1 = 0; else fresh0 = 0;
                        if (nacc == 2) accumulate ^= 2u;
                        a_lo += sub_step * a_sub16;
                        b_lo += sub_step * b_sub16;
                    }
                }
                ptx::mma_commit(empty_bar(stage), leader);
                if (++stage == p.num_stages) { stage = 0; phase ^= 1u; }
            }
            if (ok) ptx::mma_commit(tfull_bar(acc), leader);
            if (++acc == p.ep_groups) { acc = 0; acc_phase ^= 1u; }
        }
        ptx::grid_dep_launch();   // what remains is the epilogue of the last tiles
        if (!ok) {
            ptx::mma_commit(drain_bar, leader);
            for (uint32_t i = 0; i < kSpinLimit; ++i)
                if (ptx::mbar_try_wait(drain_bar, 0)) break;
        }
        if (kSplit) ptx::cluster_sync();
    } else {
        // ---------------------------------------------------------------------- epilogue
        // A warp may read the TMEM lanes of quadrant (warp % 4).  The four warps of a quadrant form ep_groups groups; group
        // `grp` serves every ep_groups-th tile of this CTA (accumulator buffer `grp`) and its warps split the tile's columns.
        // Everything that does not depend on the sums is formed before the wait for the tile's MMAs.
        const int quad = warp & 3;
        const int ew = (warp - 4) >> 2;
        // (In a cluster all of them are one group, whatever the number of columns: each must reach the cluster's barrier.)
        const int parts = kSplit ? 4 : 4 / p.ep_groups, grp = kSplit ? 0 : ew / parts, part = ew - grp * parts;
        const int groups = p.tile_n / 16;                 // 16-column groups of the tile
        int row = quad * 32 + lane;
        int g_begin = (groups * part) / parts, g_end = (groups * (part + 1)) / parts;
        // A cluster deals out its tile's (column group, pixel) pairs, pixels that exist only, in equal shares: one pair per epilogue
        // thread.  Cells of the exchange: [source CTA][4][pair of the share] x 16 bytes.
        const int rows_in = kSplit ? min(kTileM, p.M - tile_first / p.num_n_tiles * kTileM) : kTileM;
        const int share = kSplit ? (groups * rows_in + p.split - 1) / p.split : 0;
        const uint32_t red_base = smem_base + p.num_stages * stage_bytes + kTableSmemBytes;
        bool mine = true;
        if (kSplit) {
            const int tid = (int)threadIdx.x - 128, pair = rank * share + tid;
            mine = tid < share && pair < groups * rows_in;
            g_begin = mine ? pair / rows_in : 0;
            g_end = g_begin + 1;
            row = mine ? pair - g_begin * rows_in : 0;
        }
        constexpr bool fwd = kEpi == kEpiForward;
        const FwdScalars fs = fwd ? load_fwd_scalars(p) : FwdScalars{0, 0, 0};
        // the b1 table of the whole layer goes to shared memory (behind the pipeline stages), once, times b1
        const int32_t *ts = fwd ? stage_b1_table(p, fs.b1, smem_raw + (smem_base - ptx::smem_u32(smem_raw)) + p.num_stages * stage_bytes,
                                                 (int)threadIdx.x - 128, 32 * kEpilogueWarps)
                                : nullptr;
        const int shift = input_shift(p);
        const FwdShift sh = forward_shift(p, fs, shift);
        uint32_t acc_phase = 0, mx = 0, mx_masked = 0;
        bool ok = true;
        for (int tile = tile_first + grp * grid; tile < num_tiles && ok; tile += p.ep_groups * grid) {
            const int mt = tile / p.num_n_tiles, nt = tile % p.num_n_tiles;
            const int m = mt * kTileM + row;
            const bool valid = m < p.M && mine;
            size_t pix = 0;
            int cls = 0;
            if (valid) {
                const int img = m / pix_per_img, rem = m % pix_per_img;
                const int y = rem / p.wq, x = rem % p.wq;
                pix = ((size_t)img * p.out_h + (y * p.out_step + p.out_off_h)) * p.out_w + (x * p.out_step + p.out_off_w);
                if (p.b1_table)
                    cls = border_class(y, p.hq, p.b1_nlo_h, p.b1_nhi_h, p.b1_nrc) * p.b1_ncc +
                          border_class(x, p.wq, p.b1_nlo_w, p.b1_nhi_w, p.b1_ncc);
            }
            int col = nt * p.tile_n + g_begin * 16;
            size_t off = pix * p.N + col;
            const int4 zero4 = make_int4(0, 0, 0, 0);
            // the shortcut codes do not depend on the sums: the first group's are requested before the wait for the MMAs
            int4 sc = (fwd && valid && col < p.N && p.shortcut) ? __ldg(reinterpret_cast<const int4 *>(p.shortcut + off)) : zero4;
            const int32_t *tb = ts ? ts + cls * p.N + col : nullptr;
            const int32_t *tg = (!ts && p.b1_table) ? p.b1_table + (size_t)cls * p.N + col : nullptr;
            ok = __all_sync(0xffffffffu, wait_bar(tfull_bar(grp), acc_phase, ctx));  // warp-uniform
            ptx::tc_fence_after();
            const uint32_t t_row = tmem_base + grp * buf_stride + ((uint32_t)(quad * 32) << 16);
            if (kSplit) {
                const int r_own = quad * 32 + lane;   // the tensor-memory lane of this thread
#pragma unroll 1
                for (int g = part; g < groups && ok && quad * 32 < rows_in; g += 4) {
                    uint32_t r[32], r2[32];
                    ptx::tmem_ld_32x16(t_row + g * 16, r);
                    if (nacc == 2) ptx::tmem_ld_32x16(t_row + acc_stride + g * 16, r2);
                    ptx::tmem_ld_wait();
                    if (nacc == 2) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) r[i] += r2[i];
                    }
                    if (r_own < rows_in) {
                        const int pair = g * rows_in + r_own, owner = pair / share, slot = pair - owner * share;
                        const uint32_t dst = ptx::cluster_addr(red_base + (rank * 4 * share + slot) * 16, owner);
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            ptx::st_cluster_128(dst + c * share * 16, r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
                    }
                }
                ptx::cluster_sync();
            }
            if (!ok) break;
            for (int g = g_begin; g < g_end; ++g, col += 16, off += 16) {
                uint32_t r[32];
                uint32_t r2[32];
                if (kSplit) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) r[i] = 0;
                    if (mine)
#pragma unroll 2
                        for (int src = 0; src < p.split; ++src) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const int4 v = ptx::ld_shared_128(red_base + ((src * 4 + c) * share + (int)threadIdx.x - 128) * 16);
                                r[4 * c] += v.x;
                                r[4 * c + 1] += v.y;
                                r[4 * c + 2] += v.z;
                                r[4 * c + 3] += v.w;
                            }
                        }
                } else {
                    ptx::tmem_ld_32x16(t_row + g * 16, r);
                    if (nacc == 2) ptx::tmem_ld_32x16(t_row + acc_stride + g * 16, r2);
                }
                // the next group's shortcut codes travel while this group is computed
                int4 sc_next = zero4;
                if (g + 1 < g_end && fwd && valid && col + 16 < p.N && p.shortcut)
                    sc_next = __ldg(reinterpret_cast<const int4 *>(p.shortcut + off + 16));
                if (!kSplit) ptx::tmem_ld_wait();
                if (nacc == 2 && !fwd && !kSplit) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) r[i] += r2[i];  // the two partial accumulators of the tile
                }
                if (valid && col < p.N) {
                    if (fwd) {
                        forward_group(p, fs, sh, r, r2, kSplit ? 1u : nacc, off, tb, tg, sc, shift);
                    } else {
                        mx = max(mx, dgrad_16(p, r, off, mx_masked));
                    }
                }
                sc = sc_next;
                if (tb) tb += 16;
                if (tg) tg += 16;
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(tempty_bar(grp));
            acc_phase ^= 1u;
        }
        if (!fwd) {
            mx = warp_max_u32(mx);
            if (lane == 0 && mx) atomicMax(&p.dev->absmax_u32, mx);
            if (p.next_mask) {
                mx_masked = warp_max_u32(mx_masked);
                if (lane == 0 && mx_masked) atomicMax(&p.dev->absmax_u64, (unsigned long long)mx_masked);
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

template <int kEpi, bool kSplit>
__global__ void __launch_bounds__(kGemmThreads, 1)
igemm_kernel(const __grid_constant__ IgemmParams p, const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b)
{
    igemm_body<kEpi, kSplit>(p, map_a, map_b, (int)blockIdx.x, (int)gridDim.x);
}

// The GEMMs of a strided error back-propagation's residue classes, which write disjoint pixels, in one launch: a class has a range of
// CTAs.  Bound as igemm_kernel.  On branch streams of their own, with fork and join, the 48 -> 80 channel layer 37 x 29 at batch 5 called
// by itself took 36.8 us (28.6 so), and at batch 1 the four GEMMs of 256 -> 512 channels 14 x 14 ended 12.6 us behind the kernel in
// front (8.5 so); ResNet-20 step at batch 128 576 -> 567 us.
template <bool kSplit>
__global__ void __launch_bounds__(kGemmThreads, 1) igemm_classes_kernel(const __grid_constant__ IgemmClasses c)
{
    int k = 0;
    while (k + 1 < c.num && (int)blockIdx.x >= c.first[k + 1]) ++k;
    igemm_body<kEpiDgrad, kSplit>(c.p[k], c.map_a[k], c.map_b[k], (int)blockIdx.x - c.first[k], c.first[k + 1] - c.first[k]);
}

}  // namespace

size_t igemm_smem_bytes(const IgemmParams &p)
{
    return (size_t)p.num_stages * p.subs_per_stage * ((size_t)kTileM + p.tile_n) * p.kc + 1024 + kTableSmemBytes +
           (p.split > 1 ? (size_t)kTileM * p.tile_n * sizeof(int32_t) + 64 * p.split : 0);   // (shares are rounded up)
}

cudaError_t launch_igemm(const IgemmParams &p, const CUtensorMap &map_a, const CUtensorMap &map_b, int grid,
                         cudaStream_t stream)
{
    const size_t smem = igemm_smem_bytes(p);
    const auto kernel = p.split > 1 ? (p.epilogue == kEpiForward ? igemm_kernel<kEpiForward, true> : igemm_kernel<kEpiDgrad, true>)
                                    : (p.epilogue == kEpiForward ? igemm_kernel<kEpiForward, false> : igemm_kernel<kEpiDgrad, false>);
    static std::atomic<unsigned long long> allowed[2][2];
    const cudaError_t e = allow_smem((const void *)kernel, 226 * 1024, allowed[p.split > 1][p.epilogue == kEpiForward]);
    if (e != cudaSuccess) return e;
    return launch_chained_clusters(p.split, kernel, grid, kGemmThreads, smem, stream, p, map_a, map_b);
}

cudaError_t launch_igemm_classes(const IgemmClasses &c, cudaStream_t stream)
{
    size_t smem = 0;
    for (int k = 0; k < c.num; ++k) smem = igemm_smem_bytes(c.p[k]) > smem ? igemm_smem_bytes(c.p[k]) : smem;
    const int split = c.p[0].split;   // (of all classes: a launch has one cluster size)
    const auto kernel = split > 1 ? igemm_classes_kernel<true> : igemm_classes_kernel<false>;
    static std::atomic<unsigned long long> allowed[2];
    const cudaError_t e = allow_smem((const void *)kernel, 226 * 1024, allowed[split > 1]);
    if (e != cudaSuccess) return e;
    return launch_chained_clusters(split, kernel, c.first[c.num], kGemmThreads, smem, stream, c);
}

}  // namespace eoq
