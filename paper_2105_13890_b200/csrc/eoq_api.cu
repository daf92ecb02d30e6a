// C ABI of libeoq: argument checks, TMA descriptors, launch plans.  Declarations and their contract: eoq.h.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdio.h>
#include <string.h>

#include <new>

#include "eoq_internal.h"

using namespace eoq;

namespace {

// --------------------------------------------------------------------------------- driver entry points

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const int *, const int *, cuuint32_t, cuuint32_t,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn g_encode_tiled = nullptr;
EncodeIm2colFn g_encode_im2col = nullptr;

bool load_driver_entry_points()
{
    if (g_encode_tiled && g_encode_im2col) return true;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess || !fn) return false;
    g_encode_tiled = reinterpret_cast<EncodeTiledFn>(fn);
    fn = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &fn, cudaEnableDefault, &q) != cudaSuccess || !fn) return false;
    g_encode_im2col = reinterpret_cast<EncodeIm2colFn>(fn);
    return true;
}

CUtensorMapSwizzle swizzle_for(int row_bytes)
{
    switch (row_bytes) {
        case 128: return CU_TENSOR_MAP_SWIZZLE_128B;
        case 64: return CU_TENSOR_MAP_SWIZZLE_64B;
        case 32: return CU_TENSOR_MAP_SWIZZLE_32B;
        default: return CU_TENSOR_MAP_SWIZZLE_NONE;
    }
}

// Widest of 128/64/32/16 channel bytes that divides c (c is a multiple of 16).
int chunk_bytes(int c)
{
    for (int k = 128; k > 16; k >>= 1)
        if (c % k == 0) return k;
    return 16;
}

// Channel bytes of one K sub-tile of the patch kernels.  Their loads are tiled, so a chunk may reach past the last channel
// (the rest arrives as zeros): an odd multiple of 16 channels takes the chunk with the least of patch loads (about 600 cycles
// each, whatever the width) and MMAs (about 70 per tap and 32 channels), whichever bounds; 16 channels are one chunk of 32.
int patch_chunk(int c, int taps)
{
    if (c % 32 == 0) return chunk_bytes(c);
    int best = 32;
    double best_cost = 0;
    for (int kc = 32; kc <= 128; kc <<= 1) {
        const int chunks = (c + kc - 1) / kc;
        const double load = 600.0 * chunks, mma = 70.0 * taps * chunks * (kc / 32), cost = load > mma ? load : mma;
        if (kc == 32 || cost < best_cost) {
            best = kc;
            best_cost = cost;
        }
    }
    return best;
}

// View for the filter-row path: the pixel of the walk is a 128-byte window of 8 adjacent 16-channel pixels that
// starts at memory column (first_col + k * stride) of a row w_mem pixels long, so consecutive windows overlap
// (the W stride of the view is smaller than its inner extent).  Rows are walked with zero fill above and below.
bool make_row_window_map(CUtensorMap *map, const void *ptr, int n, int h, int w_mem, int c, int first_col, int count_w,
                         int count_h, int stride, int pad_h, int pixels)
{
    const cuuint64_t window = 8u * c;  // bytes of 8 adjacent pixels
    cuuint64_t dims[4] = {window, (cuuint64_t)count_w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[3] = {(cuuint64_t)stride * c, (cuuint64_t)w_mem * c, (cuuint64_t)w_mem * c * h};
    int lower[2] = {0, -pad_h};
    int upper[2] = {0, (count_h - 1) * stride + 1 - pad_h - h};
    if (upper[1] < -128 || upper[1] > 127 || pad_h > 128) return false;
    cuuint32_t estr[4] = {1, 1, (cuuint32_t)stride, 1};
    const char *base = static_cast<const char *>(ptr) + (long long)first_col * c;
    return g_encode_im2col(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<char *>(base), dims, strides, lower, upper,
                           (cuuint32_t)window, (cuuint32_t)pixels, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           swizzle_for((int)window), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// im2col view of an NHWC int8 tensor [n][h][w][c]: `pixels` consecutive positions of the walk that starts at
// (lower_w, lower_h) and advances by `stride`, `box_c` channels each.  count_w/h = positions per row/column.
bool make_im2col_map(CUtensorMap *map, const void *ptr, int n, int h, int w, int c, int lower_w, int lower_h,
                     int count_w, int count_h, int stride, int box_c, int pixels)
{
    cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[3] = {(cuuint64_t)c, (cuuint64_t)c * w, (cuuint64_t)c * w * h};
    int lower[2] = {lower_w, lower_h};
    // the walk covers count positions: (extent + upper - lower - 1) / stride + 1 = count
    int upper[2] = {(count_w - 1) * stride + 1 + lower_w - w, (count_h - 1) * stride + 1 + lower_h - h};
    for (int i = 0; i < 2; ++i)
        if (lower[i] < -128 || lower[i] > 127 || upper[i] < -128 || upper[i] > 127) return false;
    cuuint32_t estr[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
    return g_encode_im2col(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(ptr), dims, strides, lower, upper,
                           (cuuint32_t)box_c, (cuuint32_t)pixels, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           swizzle_for(box_c), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tiled view of an NHWC int8 tensor with a (box_c, box_w, box_h, 1) box: one patch of pixels, halo included.
bool make_patch_map(CUtensorMap *map, const void *ptr, int n, int h, int w, int c, int box_c, int box_w, int box_h)
{
    if (box_w > 256 || box_h > 256) return false;
    cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[3] = {(cuuint64_t)c, (cuuint64_t)c * w, (cuuint64_t)c * w * h};
    cuuint32_t box[4] = {(cuuint32_t)box_c, (cuuint32_t)box_w, (cuuint32_t)box_h, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(box_c), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tiled view of the rows of an NHWC int8 tensor, `row_bytes` each (a multiple of 16), in 8-byte units: a box of `box8` units of
// `box_rows` rows.
bool make_input_rows_map(CUtensorMap *map, const void *ptr, int n, int h, size_t row_bytes, int box8, int box_rows)
{
    cuuint64_t dims[3] = {(cuuint64_t)row_bytes / 8, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[2] = {(cuuint64_t)row_bytes, (cuuint64_t)row_bytes * h};
    cuuint32_t box[3] = {(cuuint32_t)box8, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tiled view of a [rows][taps][c] int8 tensor with a (box_c, 1, box_rows) box.
bool make_weight_map(CUtensorMap *map, const void *ptr, int rows, int taps, int c, int box_c, int box_rows)
{
    cuuint64_t dims[3] = {(cuuint64_t)c, (cuuint64_t)taps, (cuuint64_t)rows};
    cuuint64_t strides[2] = {(cuuint64_t)c, (cuuint64_t)c * taps};
    cuuint32_t box[3] = {(cuuint32_t)box_c, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    return g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(box_c), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tiled view of a [rows][c] int8 matrix with a (box_c, box_rows) box.
bool make_matrix_map(CUtensorMap *map, const void *ptr, size_t rows, int c, int box_c, int box_rows)
{
    cuuint64_t dims[2] = {(cuuint64_t)c, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)c};
    cuuint32_t box[2] = {(cuuint32_t)box_c, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(box_c), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// --------------------------------------------------------------------------------- checks and geometry

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
inline size_t round256(size_t v) { return (v + 255) & ~(size_t)255; }

struct Geometry {
    int ho, wo, taps;
    size_t in_elems, out_elems, w_elems;
};

int check_desc(const eoq_conv_desc_t *d, Geometry *g)
{
    if (!d) return EOQ_ERR_BAD_ARG;
    if (d->n <= 0 || d->h <= 0 || d->w <= 0 || d->c_in <= 0 || d->c_out <= 0 || d->kh <= 0 || d->kw <= 0 ||
        d->stride <= 0 || d->pad < 0)
        return EOQ_ERR_BAD_ARG;
    if (d->h + 2 * d->pad < d->kh || d->w + 2 * d->pad < d->kw) return EOQ_ERR_BAD_ARG;
    if ((d->c_in % 16 && d->c_in != 8) || d->c_out % 16) return EOQ_ERR_ALIGNMENT;  // 8: the filter-row path only
    if (d->x_wmargin < 0 || d->x_wmargin > 64) return EOQ_ERR_BAD_ARG;
    if (d->kh * d->kw > kMaxTaps || d->kh > 16 || d->kw > 16 || d->stride > 8 || d->pad > 64) return EOQ_ERR_UNSUPPORTED;
    g->ho = (d->h + 2 * d->pad - d->kh) / d->stride + 1;
    g->wo = (d->w + 2 * d->pad - d->kw) / d->stride + 1;
    g->taps = d->kh * d->kw;
    g->in_elems = (size_t)d->n * d->h * d->w * d->c_in;
    g->out_elems = (size_t)d->n * g->ho * g->wo * d->c_out;
    g->w_elems = (size_t)d->c_out * g->taps * d->c_in;
    if ((size_t)d->n * d->h * d->w >= (1u << 31) || (size_t)d->n * g->ho * g->wo >= (1u << 31)) return EOQ_ERR_UNSUPPORTED;
    return EOQ_OK;
}

// Rows (or columns) whose filter window leaves the image at the low / high end.
void border_counts(int extent_in, int extent_out, int k, int stride, int pad, int *nlo, int *nhi, int *ncls)
{
    int lo = 0, hi = 0;
    for (int y = 0; y < extent_out; ++y) {
        if (y * stride - pad < 0) ++lo;
        if (y * stride - pad + k - 1 > extent_in - 1) ++hi;
    }
    *nlo = lo;
    *nhi = hi;
    *ncls = (lo + hi + 1 >= extent_out) ? extent_out : lo + hi + 1;
}

BorderClasses border_classes(const eoq_conv_desc_t &d, const Geometry &g)
{
    BorderClasses bc;
    border_counts(d.h, g.ho, d.kh, d.stride, d.pad, &bc.nlo_h, &bc.nhi_h, &bc.nrc);
    border_counts(d.w, g.wo, d.kw, d.stride, d.pad, &bc.nlo_w, &bc.nhi_w, &bc.ncc);
    return bc;
}

int record(Handle *h, cudaError_t e)
{
    if (e == cudaSuccess) return EOQ_OK;
    h->last_cuda_error = (int)e;
    return EOQ_ERR_CUDA;
}

// 16- or 8-channel inputs under filters 5 to 8 taps wide (the 7x7 first layer) stored with wide enough zero margins
// take the filter-row path: a filter row is 8 adjacent pixels, one 128- or 64-byte K sub-tile, instead of one TMA
// row per tap.  The window of an output pixel starts (stride * c_in) bytes after its neighbour's and the first one
// (x_wmargin - pad) pixels into the row: both must be multiples of 16 bytes, which 8 channels meet for even strides
// and an even distance between margin and padding.
inline bool use_row_window(const eoq_conv_desc_t &d, int wo)
{
    if ((d.c_in != 16 && d.c_in != 8) || d.kw < 5 || d.kw > 8) return false;
    if (d.c_in == 8 && ((d.stride & 1) || ((d.x_wmargin - d.pad) & 1) || (d.w & 1))) return false;
    const int need_right = (wo - 1) * d.stride - d.pad + 8 - d.w;
    return d.x_wmargin >= d.pad && d.x_wmargin >= need_right;
}

// CTAs of a persistent GEMM over `tiles` tiles.  The kernel lasts as long as its busiest CTA, ceil(tiles / SMs)
// tiles; spreading the tiles evenly over the fewest CTAs that keep that maximum costs nothing and leaves the other
// SMs to kernels of other streams (448 tiles on 148 SMs: 112 CTAs of 4 tiles instead of 148 of 3 or 4).
inline int persistent_grid(int tiles, int sm_count)
{
    if (tiles <= sm_count) return tiles < 1 ? 1 : tiles;
    const int per_cta = (tiles + sm_count - 1) / sm_count;
    return (tiles + per_cta - 1) / per_cta;
}

// Tiles a CTA keeps in the epilogue at once.  One group of warps on one tile leaves every wait of that tile exposed (a
// 128 x 64 tile took 2,250 cycles alone, 2,650 per tile with two of them, against about 1,100 of issue), so as many tiles as
// the CTA gets and tensor memory holds are worked on side by side; a CTA with a single tile puts all its warps on it.
void plan_epilogue(IgemmParams &p, int grid)
{
    if (p.split > 1) {   // every epilogue warp takes part in the exchange
        p.ep_groups = 1;
        return;
    }
    const int tiles = p.num_m_tiles * p.num_n_tiles, per_cta = (tiles + grid - 1) / grid;
    int cols = 32;
    while (cols < p.tile_n) cols <<= 1;
    const int buffer = p.tile_n <= 128 ? 2 * cols : cols;   // two partial accumulators up to 128 columns
    p.ep_groups = per_cta >= 3 && 4 * buffer <= 512 ? 4 : (per_cta >= 2 && 2 * buffer <= 512 ? 2 : 1);
    if (p.tile_n / 16 < 4 / p.ep_groups) p.ep_groups = p.tile_n >= 32 ? 2 : 4;   // at least one 16-column group per warp
}

// Columns of a tile and CTAs that share one, with what follows from them.
void set_columns(IgemmParams &p, int tile_n, int split)
{
    p.tile_n = tile_n;
    p.num_n_tiles = (p.N + tile_n - 1) / tile_n;
    p.split = split;
    p.b_row = p.b_mn ? chunk_bytes(tile_n) : 0;
    const size_t stage = (size_t)p.subs_per_stage * (kTileM + tile_n) * p.kc;
    // (a split's exchange takes a tile's worth of shared memory from the stages)
    const int stages = (int)((200 * 1024 - (split > 1 ? (size_t)kTileM * tile_n * sizeof(int32_t) : 0)) / stage);
    p.num_stages = stages > 8 ? 8 : (stages < 2 ? 2 : stages);
}

// Shared tiling choices of the implicit GEMM: K sub-tiles, pipeline depth, column tile.  (p.b_mn is set before.)
void plan_igemm(IgemmParams &p, int src_channels, int ntaps, int sm_count)
{
    p.kc = chunk_bytes(src_channels);
    p.chunks_per_tap = src_channels / p.kc;
    p.ntaps = ntaps;
    p.real_sub = ntaps * p.chunks_per_tap;
    p.num_sub = (p.kc == 16 && (p.real_sub & 1)) ? p.real_sub + 1 : p.real_sub;
    p.subs_per_stage = 128 / p.kc;
    if (p.subs_per_stage > p.num_sub) p.subs_per_stage = p.num_sub;
    p.num_m_tiles = (p.M + kTileM - 1) / kTileM;
    // An MMA costs at least ~57 cycles whatever its width and reaches the tensor peak only from 128 columns
    // up, so tiles stay 128 wide even when that leaves some SMs without one; 256 when there are tiles to spare.
    int tn = p.N < 256 ? p.N : 256;
    const bool spare = (long long)p.num_m_tiles * ((p.N + 255) / 256) >= 2LL * sm_count;
    if (tn == 256 && !spare) tn = 128;
    if (p.N > 128 && !p.b_mn) {
        // Forward: cuts of equal width (28 x 28 at batch 64, 1024 -> 304 channels: two of 160 instead of 256 and 48, 28.3 -> 25.9 us).
        // Up to 512 terms the epilogue bounds the layer, and its time goes by the columns of the busiest CTA: narrow tiles then where
        // that has at least four wide ones and they leave it fewer columns (64 -> 512 channels with shortcut 54.3 -> 45.0 us,
        // 512 -> 512 59.6 -> 53.7; without shortcut 1024 -> 256 at 14 x 14, batch 512: 35.6 us wide, 36.6 narrow).
        auto cut = [&](int most) { const int parts = (p.N + most - 1) / most; return ((p.N + parts - 1) / parts + 15) / 16 * 16; };
        auto columns = [&](int cols) { return ((long long)p.num_m_tiles * ((p.N + cols - 1) / cols) + sm_count - 1) / sm_count * cols; };
        tn = tn < 256 && p.N < 256 ? tn : cut(tn);
        if (p.N >= 256 && spare && ntaps * src_channels <= 512 && columns(tn) >= 4 * tn && columns(cut(128)) < columns(tn)) tn = cut(128);
    }
    set_columns(p, tn, 1);
    p.a_rows = kTileM;   // a problem of fewer pixels loads no more of them (TMA time goes by rows; the rest of the tile is never stored)
    while (p.a_rows > 16 && p.M <= p.a_rows / 2) p.a_rows /= 2;
}

// ---- problems of few tiles (small batches)
// Where the tiles leave at least half of the CTAs idle, everything runs at once and the time of one tile counts: narrower tiles then
// (shorter epilogues, fewer weights per CTA), several CTAs per tile (a cluster, see igemm_kernel), and whichever of the two kernels
// is faster.  The estimates are in microseconds of a kernel in a chain of its like, fitted to layers of 1 to 13 images; what they
// choose against the wide tiles before: 128 channels 28 x 28, one image: 6.1 -> 4.3 (32 columns, patch kernel); 256 channels
// 14 x 14: 7.1 -> 5.3; 512 channels 7 x 7: 7.6 -> 5.8 (128 columns, 8 CTAs a tile), 3.6 of which any kernel takes.
constexpr double kFewPerCta = 0.0025;   // a CTA more to bring up
// bytes of a TMA row: its time
double few_row(int bytes) { return 0.0004 + 3.4e-6 * bytes; }

double few_igemm_time(const IgemmParams &p)
{
    const int k_iters = (p.num_sub + p.subs_per_stage - 1) / p.subs_per_stage;
    const int iters = (k_iters + p.split - 1) / p.split, rows = p.M < kTileM ? p.M : kTileM;
    const double load = 0.0009 * p.subs_per_stage * (p.a_rows + (p.b_mn ? p.kc * (p.tile_n / p.b_row) : p.tile_n));
    const double mma = 0.0485 * p.subs_per_stage * (p.kc < 32 ? 0.5 : p.kc / 32);   // (92 cycles each, with their waits and commits)
    double t = 3.6 + iters * (load > mma ? load : mma) + 6e-5 * rows * p.tile_n / p.split +
               kFewPerCta * p.num_m_tiles * p.num_n_tiles * p.split;
    if (p.split > 1) t += 0.3 + 0.025 * rows * p.tile_n * 4 / 1024.0;   // the exchange
    return t;
}

// The fastest column tile at `split` CTAs per tile within `ctas` (false: none).
bool narrow_tiles(const IgemmParams &p, int split, int ctas, IgemmParams &best, double &best_time)
{
    const int k_iters = (p.num_sub + p.subs_per_stage - 1) / p.subs_per_stage;
    bool found = false;
    for (int cuts = 1; cuts <= 32; cuts *= 2) {
        const int tn = ((p.N + cuts - 1) / cuts + 15) / 16 * 16;
        if (tn > 128) continue;
        if (!(split > 1 && (p.kc < 64 || k_iters < split || tn / 16 > 4 * split))) {
            IgemmParams q = p;
            set_columns(q, tn, split);
            if (q.num_m_tiles * q.num_n_tiles * split <= (split > 1 ? ctas / 2 : ctas)) {
                const double time = few_igemm_time(q);
                if (!found || time < 0.97 * best_time) {
                    best = q;
                    best_time = time;
                    found = true;
                }
            }
        }
        if (tn == 16) break;
    }
    return found;
}

// Columns per tile and CTAs per tile of the im2col kernel.  Clusters take at most half of the CTAs (beyond that many, some wait for
// room: 512 channels 7 x 7, one image: 64 CTAs 5.9 us, 128 CTAs 6.7) and want every CTA to have a K iteration of at least two MMAs.
void plan_few_tiles(IgemmParams &p, int ctas)
{
    if (2 * p.num_m_tiles * p.num_n_tiles > ctas) return;
    const int k_iters = (p.num_sub + p.subs_per_stage - 1) / p.subs_per_stage;
    IgemmParams best = p;
    double best_time = few_igemm_time(p);
    for (int cuts = 1; cuts <= 32; cuts *= 2) {
        const int tn = ((p.N + cuts - 1) / cuts + 15) / 16 * 16;
        if (tn > 128) continue;
        for (int split = 1; split <= 8; split *= 2) {
            if (split > 1 && (p.kc < 64 || k_iters < split || tn / 16 > 4 * split)) continue;
            IgemmParams q = p;
            set_columns(q, tn, split);
            if (q.num_m_tiles * q.num_n_tiles * split > (split > 1 ? ctas / 2 : ctas)) continue;
            const double time = few_igemm_time(q);
            if (time < 0.97 * best_time) {
                best = q;
                best_time = time;
            }
        }
        if (tn == 16) break;
    }
    p = best;
}

// Tiles and CTAs of the residue classes that share a launch (cl.num of them, planned by plan_igemm).
// CTAs: the fewest per class with which the class that takes longest is done first.  A tile costs its taps and, about half of one, its
// sums: by taps alone the class of one tap ended last.
// Few tiles: as plan_few_tiles, each class within its share of the CTAs, with one split for all of them.
void plan_classes(IgemmClasses &cl, int ctas)
{
    if (cl.num == 1) {
        plan_few_tiles(cl.p[0], ctas);
    } else {
        int share[kMaxClasses], total = 0;
        for (int k = 0; k < cl.num; ++k) total += 2 * cl.p[k].ntaps + 1;
        bool few = true;
        for (int k = 0; k < cl.num; ++k) {
            share[k] = ctas * (2 * cl.p[k].ntaps + 1) / total;
            if (share[k] < 1) share[k] = 1;
            few = few && 2 * cl.p[k].num_m_tiles * cl.p[k].num_n_tiles <= share[k];
        }
        double best_time = 0;
        IgemmParams best[kMaxClasses];
        for (int split = 1; few && split <= 8; split *= 2) {
            IgemmParams q[kMaxClasses];
            double slowest = 0;
            bool ok = true;
            for (int k = 0; k < cl.num && ok; ++k) {
                double time = 0;
                ok = narrow_tiles(cl.p[k], split, share[k], q[k], time);
                if (time > slowest) slowest = time;
            }
            if (ok && (split == 1 || slowest < 0.97 * best_time)) {
                best_time = slowest;
                memcpy(best, q, sizeof(IgemmParams) * cl.num);
            }
        }
        if (best_time > 0) memcpy(cl.p, best, sizeof(IgemmParams) * cl.num);
    }
    int cost[kMaxClasses], tiles[kMaxClasses];
    long long work = 0;
    for (int k = 0; k < cl.num; ++k) {
        tiles[k] = cl.p[k].num_m_tiles * cl.p[k].num_n_tiles;
        cost[k] = 2 * cl.p[k].ntaps + 1;
        work += (long long)tiles[k] * cost[k];
    }
    // The least time from work / ctas on in which the classes get by with `ctas` CTAs, or with one each: they need fewer the longer it is,
    // and one each once it covers all tiles of every class.  It is mostly near: steps that double, then bisection.  (Counted up one by one,
    // 12,544 tiles a class under a cap of three CTAs took 20,908 steps.)
    auto divide = [&](long long time) -> bool {
        int used = 0;
        cl.first[0] = 0;
        for (int k = 0; k < cl.num; ++k) {
            const long long per_cta = cl.p[0].split > 1 ? 1 : time / cost[k];   // (a cluster has one tile)
            if (per_cta < 1) return false;
            used += (int)((tiles[k] + per_cta - 1) / per_cta);
            cl.first[k + 1] = used * cl.p[0].split;
        }
        return used <= ctas || used <= cl.num;
    };
    long long low = work / ctas, high = low, most = low;   // `most` is enough, times below `low` are not
    for (int k = 0; k < cl.num; ++k) most = std::max(most, (long long)tiles[k] * cost[k]);
    for (long long step = 1; high < most && !divide(high); step *= 2) {
        low = high + 1;
        high = std::min(most, high + step);
    }
    while (low < high) {
        const long long mid = (low + high) / 2;
        if (divide(mid)) high = mid;
        else low = mid + 1;
    }
    divide(high);
    for (int k = 0; k < cl.num; ++k) plan_epilogue(cl.p[k], (cl.first[k + 1] - cl.first[k]) / cl.p[0].split);
}

// Plan of the patch variant for a stride-1 k x k correlation over a source [n][hs][ws][c_src] producing a
// [n][hq][wq] grid with n_cols columns.  Returns false when the geometry does not suit it (then the per-tap
// path is used): strided or 1x1 filters, rows too wide for a tile, or tiles that would be mostly padding.
// `ctas`: that the launch may use; `columns`: of a tile, 0 for the plan's own choice.
bool plan_patch(IgemmParams &p, PatchPlan &pl, int n_img, int c_src, int hq, int wq, int k, int pad_src, int n_cols,
                int sm_count, int ctas, int columns = 0)
{
    if (k < 2 || c_src % 16 || pad_src < 0 || pad_src > k - 1) return false;
    const int pw = wq + k - 1;
    if (pw > kTileM) return false;
    int r = kTileM / pw;
    if (r > hq) r = hq;
    const int tiles_per_img = (hq + r - 1) / r;
    if ((double)hq * wq < 0.6 * (double)tiles_per_img * kTileM) return false;
    pl.n_img = n_img;
    pl.kdim = k;
    pl.pad = pad_src;
    pl.pw = pw;
    pl.r_rows = r;
    pl.tiles_per_img = tiles_per_img;
    p.kc = patch_chunk(c_src, k * k);
    pl.chunks = (c_src + p.kc - 1) / p.kc;
    p.chunks_per_tap = pl.chunks;
    p.ntaps = k * k;
    const int patch_rows = r + k - 1;
    pl.a_box_bytes = p.kc * pw * patch_rows;
    const int rows_read = (k - 1) * (pw + 1) + kTileM;  // the last tap's tile ends here
    const int rows = pw * patch_rows > rows_read ? pw * patch_rows : rows_read;
    pl.a_bytes = (int)((((size_t)rows * p.kc) + 1023) & ~(size_t)1023);
    p.M = n_img * hq * wq;
    p.N = n_cols;
    p.hq = hq;
    p.wq = wq;
    p.num_m_tiles = n_img * tiles_per_img;
    // 256 columns where that saves a wave of tiles: a 256-column MMA reads 12 KB of shared memory for twice the work of a
    // 128-column one that reads 8 KB, and its tile costs about 1.4 times as much (256 channels, 14 x 14, batch 64: one wave of
    // 128 wide tiles instead of two of narrow ones, 16.9 -> 13.6 us).
    int tn = n_cols < 256 ? n_cols : 256;
    if (tn == 256) {
        auto waves = [&](int cols) { return ((long long)p.num_m_tiles * ((n_cols + cols - 1) / cols) + sm_count - 1) / sm_count; };
        if (7 * waves(256) >= 5 * waves(128)) tn = 128;
    }
    if (columns) tn = columns;
    p.tile_n = tn;
    p.num_n_tiles = (n_cols + tn - 1) / tn;
    p.b_row = p.b_mn ? chunk_bytes(tn) : 0;
    const size_t budget = 200 * 1024;
    const size_t b_sub = (size_t)tn * p.kc;
    const size_t b_all = b_sub * pl.chunks * p.ntaps;
    // resident where the tiles of a CTA share their weights: one column tile, or one tile per CTA (which needs one patch buffer, two
    // if it has several chunks)
    const bool one_tile = (long long)p.num_m_tiles * p.num_n_tiles <= ctas;
    pl.b_resident = ((p.num_n_tiles == 1 || one_tile) && b_all + (one_tile && pl.chunks == 1 ? 1 : 2) * (size_t)pl.a_bytes <= budget &&
                     b_all < (1u << 20)) ? 1 : 0;
    if (pl.b_resident) {
        size_t na = (budget - b_all) / pl.a_bytes;
        // 64 channels 56 x 56, batch 512: 152 us with at most 4 patches in flight, 140 with 6, 145 with 8
        pl.num_a = na > 6 ? 6 : (int)na;
        pl.num_b = 1;
    } else {
        pl.num_a = pl.chunks > 1 ? 3 : 2;
        if ((size_t)pl.num_a * pl.a_bytes + 2 * b_sub > budget) return false;
        size_t nb = (budget - (size_t)pl.num_a * pl.a_bytes) / b_sub;
        pl.num_b = nb > 8 ? 8 : (int)nb;
    }
    return pl.num_a >= 2 || (pl.b_resident && pl.num_a >= 1);
}

double few_patch_time(const IgemmParams &p, const PatchPlan &pl)
{
    const int subs = pl.chunks * p.ntaps, mmas = subs * (p.kc / 32);
    const double weights = p.b_mn ? p.kc * (p.tile_n / p.b_row) * few_row(p.b_row) : p.tile_n * few_row(p.kc);
    // weights through the ring: about 0.3 us a sub-tile, with its wait and commit; resident ones arrive in front of the MMAs
    const double body = pl.b_resident ? subs * weights + mmas * (p.tile_n > 114 ? 0.034 : 0.028) : subs * 0.3;
    return 3.0 + body + 4e-5 * kTileM * p.tile_n + kFewPerCta * p.num_m_tiles * p.num_n_tiles;
}

// Plan of a stride-1 k x k correlation (p.b_mn says how the weights are read); false: the im2col kernel takes it.
bool plan_stride1(IgemmParams &p, PatchPlan &pl, int n_img, int c_src, int hq, int wq, int k, int pad_src, int n_cols, int sm_count,
                  int ctas)
{
    if (!plan_patch(p, pl, n_img, c_src, hq, wq, k, pad_src, n_cols, sm_count, ctas)) return false;
    if (2 * p.num_m_tiles * p.num_n_tiles > ctas) return true;
    double time = few_patch_time(p, pl);
    for (int cuts = 2; cuts <= 32; cuts *= 2) {
        const int tn = ((n_cols + cuts - 1) / cuts + 15) / 16 * 16;
        IgemmParams q = p;
        PatchPlan ql = pl;
        if (!plan_patch(q, ql, n_img, c_src, hq, wq, k, pad_src, n_cols, sm_count, ctas, tn)) continue;
        if (q.num_m_tiles * q.num_n_tiles > ctas) break;
        const double t = few_patch_time(q, ql);
        if (t < 0.97 * time) {
            time = t;
            p = q;
            pl = ql;
        }
        if (tn == 16) break;
    }
    IgemmParams g;
    memset(&g, 0, sizeof(g));
    g.M = p.M;
    g.N = p.N;
    g.b_mn = p.b_mn;
    plan_igemm(g, c_src, p.ntaps, sm_count);
    plan_few_tiles(g, ctas);
    return few_igemm_time(g) > 0.97 * time;
}

// Plan of the input-row forward kernel for a filter-row layer (see use_row_window); false: the im2col kernel takes it.
bool plan_rows(IgemmParams &p, RowsPlan &pl, const eoq_conv_desc_t &d, const Geometry &g, int ctas)
{
    if (d.stride * d.c_in != 16 || d.c_out > 128 || (d.w + 2 * d.x_wmargin) * d.c_in % 16 || (d.x_wmargin - d.pad) * d.c_in % 16) return false;
    memset(&pl, 0, sizeof(pl));
    pl.n_img = d.n;
    pl.stride = d.stride;
    pl.pad = d.pad;
    // a box row has at most 256 units of 8 bytes: 125 windows of 8 channels, 121 of 16
    const int most_px = (2048 - 8 * d.c_in) / 16 + 1;
    pl.x_tiles = (g.wo + most_px - 1) / most_px;
    pl.tile_px = (g.wo + pl.x_tiles - 1) / pl.x_tiles;
    pl.first_col8 = (d.x_wmargin - d.pad) * d.c_in / 8;
    pl.row_pitch = 16 * (pl.tile_px - 1) + 8 * d.c_in;
    pl.slack = (16 * (kTileM - 1) + 8 * d.c_in - pl.row_pitch + 127) / 128 * 128;
    p.kc = 8 * d.c_in;
    p.ntaps = d.kh;
    p.tile_n = d.c_out;
    p.num_n_tiles = 1;
    p.split = 1;
    const long long budget = 200 * 1024 - (long long)p.ntaps * p.tile_n * p.kc - pl.slack;
    // Output rows per patch: a CTA's rows at about 1,100 cycles each and 150 per patch, and the load of its first patch (35 bytes a
    // cycle) in front of them.
    double best = 0;
    for (int r = 1; r <= 16 && r <= g.ho; ++r) {
        const int rows_in = (r - 1) * d.stride + d.kh;
        const long long bytes = ((long long)rows_in * pl.row_pitch + 127) / 128 * 128;
        if (rows_in > 256 || 2 * bytes > budget) break;
        const int blocks = (g.ho + r - 1) / r;
        const long long patches = (long long)d.n * blocks * pl.x_tiles;
        const int per_cta = (int)((patches + ctas - 1) / ctas);
        const double load = rows_in * pl.row_pitch / 35.0, rows = r * 1100.0 + 150.0;
        const double cost = load + per_cta * (rows > load ? rows : load);
        if (pl.r_rows == 0 || cost < best) {
            best = cost;
            pl.r_rows = r;
            pl.row_blocks = blocks;
            pl.a_box_bytes = rows_in * pl.row_pitch;
            pl.a_bytes = (int)bytes;
            const long long na = budget / bytes;
            pl.num_a = na > 4 ? 4 : (int)na;
        }
    }
    if (!pl.r_rows) return false;
    const long long patches = (long long)d.n * pl.row_blocks * pl.x_tiles;
    if (patches > 0x7fffffff) return false;
    p.num_m_tiles = (int)patches;   // (for the grid; the epilogue's groups go by output rows)
    return true;
}

// Plan of the patch variant of the weight gradient; false when the geometry does not suit it.
bool plan_wgrad_patch(WgradPatchPlan &pl, const eoq_conv_desc_t &d, int ho, int wo, int target_ctas = kWgradTargetCtas)
{
    if (d.stride != 1 || d.kh != d.kw || d.kh < 2 || d.x_wmargin != 0 || d.c_in % 16 || d.c_out % 16) return false;
    if (d.pad > d.kh - 1) return false;
    memset(&pl, 0, sizeof(pl));
    pl.n_img = d.n; pl.ho = ho; pl.wo = wo; pl.c_in = d.c_in; pl.c_out = d.c_out;
    pl.kdim = d.kh; pl.pad = d.pad;
    pl.pw = wo + d.kh - 1;
    if (pl.pw > 256) return false;
    pl.kc = patch_chunk(d.c_in, d.kh * d.kw);
    pl.chunks = (d.c_in + pl.kc - 1) / pl.kc;
    pl.apa = 128 / pl.kc;
    pl.accs_per_row = (d.kh + pl.apa - 1) / pl.apa;
    pl.tile_n = patch_chunk(d.c_out, d.kh * d.kw);
    pl.n_tiles = (d.c_out + pl.tile_n - 1) / pl.tile_n;
    int rpg = 512 / (pl.tile_n * pl.accs_per_row);
    if (rpg * pl.accs_per_row > 8) rpg = 8 / pl.accs_per_row;
    if (rpg > d.kh) rpg = d.kh;
    if (rpg < 1) return false;
    pl.rows_per_group = rpg;
    pl.row_groups = (d.kh + rpg - 1) / rpg;
    pl.num_groups = pl.n_tiles * pl.chunks * pl.row_groups;
    pl.rows_total = d.kh * d.kw * d.c_in;
    // Rows per pixel block: as many as keep one stage near 64 KB (three stages in flight).  Layers of one 32-channel chunk take
    // half: the error back-propagation of such layers leaves the other half of an SM's shared memory, and the two then share
    // SMs (ResNet-20 step at batch 128: 659 -> 647 us; wider layers fill the SM anyway and only load more halo rows).
    const int smem_kb = pl.kc <= 32 && pl.tile_n <= 32 ? 100 : 200;
    auto set_rows = [&](int r) {
        const int kp = (r * pl.pw + 31) / 32 * 32;
        int x_rows = (r + d.kh - 1) * pl.pw;
        const int x_read = (d.kh - 1) * (pl.pw + 1) + pl.apa + kp;
        if (x_read > x_rows) x_rows = x_read;
        pl.x_bytes = (x_rows * pl.kc + 1023) / 1024 * 1024;
        pl.e_bytes = (kp * pl.tile_n + 1023) / 1024 * 1024;
        pl.kp = kp;
        pl.r_rows = r;
        pl.blocks_per_img = (ho + r - 1) / r;
        pl.x_box_bytes = pl.kc * pl.pw * (r + d.kh - 1);
        pl.e_box_bytes = pl.tile_n * pl.pw * r;
        const int stages = (smem_kb * 1024) / (pl.x_bytes + pl.e_bytes);
        pl.num_stages = stages > 4 ? 4 : stages;
        const int total_blocks = d.n * pl.blocks_per_img;
        int splits = target_ctas / pl.num_groups;  // rounded down: a few CTAs beyond one wave would double the kernel's time
        if (splits > total_blocks) splits = total_blocks;
        if (splits < 1) splits = 1;
        int per = (total_blocks + splits - 1) / splits;
        const int max_per = 130000 / kp;  // keeps a CTA's int32 partial sums exact: rows * 127 * 128 < 2^31
        if (per > max_per) per = max_per;
        pl.blocks_per_split = per;
        pl.num_splits = per > 0 ? (total_blocks + per - 1) / per : 0;
    };
    int r = ho < 32 ? ho : 32;
    for (; r >= 1; --r) {
        set_rows(r);
        if (pl.x_bytes + pl.e_bytes <= smem_kb / 3 * 1024) break;
    }
    if (r < 1 || pl.num_stages < 2 || pl.blocks_per_split < 1) return false;
    // Small batches leave fewer blocks than CTAs: shorter blocks then, as long as the time a CTA saves is not spent on more
    // slices.  In SM cycles: a TMA row 4.5, an MMA 57 to 64; a slice is written and read back at 2,500 bytes per cycle.
    auto cost = [&]() {
        const double load = 4.5 * pl.pw * (2 * pl.r_rows + d.kh - 1);
        const double mma = pl.kp / 32 * pl.rows_per_group * pl.accs_per_row * (pl.tile_n > 114 ? 64.0 : 57.0);
        return pl.blocks_per_split * (load > mma ? load : mma) + (double)pl.num_splits * d.c_out * pl.rows_total * 8 / 2500.0;
    };
    int best_r = r;
    double best = cost();
    for (int rr = (r + 1) / 2; rr >= 1; rr = (rr + 1) / 2) {
        set_rows(rr);
        if (pl.num_stages >= 2 && pl.blocks_per_split >= 1 && cost() < 0.9 * best) {
            best = cost();
            best_r = rr;
        }
        if (rr == 1) break;
    }
    set_rows(best_r);
    // with fewer CTAs no more slices than with all of them (the workspace holds that many)
    WgradPatchPlan full;
    if (target_ctas < kWgradTargetCtas && plan_wgrad_patch(full, d, ho, wo) && pl.num_splits > full.num_splits) pl = full;
    return true;
}

// Plan of the per-tap weight gradient (strided and 1x1 filters, the filter-row path); false when the geometry is not
// supported.  With fewer CTAs than the device has, no more splits than with all of them (the workspace holds that many).
bool plan_wgrad(WgradParams &p, const eoq_conv_desc_t &d, const Geometry &g, int ctas)
{
    memset(&p, 0, sizeof(p));
    p.P = d.n * g.ho * g.wo;
    p.ho = g.ho;
    p.wo = g.wo;
    p.c_in = d.c_in;
    p.c_out = d.c_out;
    p.ntaps = g.taps;
    const bool row_window = use_row_window(d, g.wo);
    if (d.c_in == 8 && !row_window) return false;
    p.kc = row_window ? 8 * d.c_in : chunk_bytes(d.c_in);
    p.nc = chunk_bytes(d.c_out);
    p.chunks_per_tap = row_window ? 1 : d.c_in / p.kc;
    p.rows_total = g.taps * d.c_in;
    p.subs_per_mtile = kTileM / p.kc;
    // filter-row path: a filter row is 8 taps x c_in rows, 128 / (8 c_in) filter rows per M tile
    p.num_m_tiles = row_window ? (d.kh * p.kc + kTileM - 1) / kTileM : (p.rows_total + kTileM - 1) / kTileM;
    if (row_window) {
        p.ntaps = d.kh;
        p.row_window_kw = d.kw;
    }
    p.pixels_per_stage = 64;
    const int px = p.pixels_per_stage;
    const int total_stages = (p.P + px - 1) / px;
    // a 64-pixel stage adds at most 64 * 127 * 127 to an int32 partial sum
    const int max_stages_exact = 1024;
    // Columns, M tiles side by side in one CTA (they share the stage's error tile) and splits of the pixel range are chosen
    // together.  In SM cycles, as measured: a TMA row 3.1, an MMA 57 to 128, a column of an M tile in the epilogue 8; a slice
    // is written and read back at 2,500 bytes per cycle of the whole device.  With 64-bit atomics into one buffer and at
    // least 8 stages per CTA, the 1024 -> 256 layer of 14 x 14 pixels took 24.4 us at batch 32 (the atomics 17 of them).
    const int cap = ctas < kWgradTargetCtas ? ctas : kWgradTargetCtas;
    double best = 0;
    int best_splits = 0;
    for (int cuts = 1; cuts <= 8; cuts = cuts < 4 ? cuts + 1 : cuts * 2) {
        const int tn = ((d.c_out + cuts - 1) / cuts + p.nc - 1) / p.nc * p.nc;
        if (tn > 256) continue;
        if (cuts > 1 && tn >= d.c_out) break;
        const int n_tiles = (d.c_out + tn - 1) / tn, b_subs = tn / p.nc;
        for (int mpc = 1; mpc <= 8 && mpc <= p.num_m_tiles && mpc * tn <= 512; ++mpc) {
            const size_t stage_bytes = (size_t)px * (mpc * kTileM + tn);
            if (mpc > 1 && 3 * stage_bytes > 200 * 1024) break;
            const int groups = (p.num_m_tiles + mpc - 1) / mpc, tiles = groups * n_tiles;
            const int waves = (tiles + cap - 1) / cap;
            const double load = 3.1 * px * (mpc * p.subs_per_mtile + b_subs), mma = (px / 32) * mpc * (tn > 114 ? tn * 0.5 : 57.0);
            const double per_stage = load > mma ? load : mma, per_slice = (double)p.rows_total * d.c_out * 8 / 2500.0;
            // waves * (total / s) * per_stage + s * per_slice is smallest near s = sqrt(total * per_stage / per_slice)
            const int most = tiles > cap ? 1 : cap / tiles;
            int splits = (int)(sqrt((double)total_stages * per_stage / per_slice) + 0.5);
            splits = splits < 1 ? 1 : (splits > most ? most : splits);
            if (splits > total_stages) splits = total_stages;
            int per = (total_stages + splits - 1) / splits;
            if (per > max_stages_exact) per = max_stages_exact;
            splits = (total_stages + per - 1) / per;
            const double cost = waves * (per * per_stage + 8.0 * mpc * tn) + splits * per_slice;
            if (best_splits == 0 || cost < best) {
                best = cost;
                best_splits = splits;
                p.tile_n = tn;
                p.num_n_tiles = n_tiles;
                p.mtiles_per_cta = mpc;
                p.num_m_groups = groups;
                p.stages_per_split = per;
                p.num_k_splits = splits;
                const int stages = (int)(200 * 1024 / stage_bytes);
                p.num_stages = stages > 8 ? 8 : (stages < 2 ? 2 : stages);
            }
        }
    }
    if (cap < kWgradTargetCtas) {
        WgradParams full;
        plan_wgrad(full, d, g, kWgradTargetCtas);
        if (p.num_k_splits > full.num_k_splits) {
            p.stages_per_split = full.stages_per_split;
            p.num_k_splits = full.num_k_splits;
        }
    }
    p.src_stride = d.stride;
    p.base_h = -d.pad;
    if (row_window) {
        p.src_stride_w = 1;
        p.base_w = 0;
        for (int t = 0; t < d.kh; ++t) {
            p.tap_dh[t] = (unsigned char)t;
            p.tap_dw[t] = 0;
        }
    } else {
        p.src_stride_w = d.stride;
        p.base_w = d.x_wmargin - d.pad;
        for (int t = 0; t < g.taps; ++t) {
            p.tap_dh[t] = (unsigned char)(t / d.kw);
            p.tap_dw[t] = (unsigned char)(t % d.kw);
        }
    }
    return true;
}

// Plan of the filter-row weight gradient with its window rows in a ring; false when the geometry does not suit it (16 channels,
// or rows so wide that the ring does not hold two output rows: the per-tap kernel).
bool plan_wgrad_rows(WgradRowsPlan &pl, const eoq_conv_desc_t &d, const Geometry &g, int ctas)
{
    if (!use_row_window(d, g.wo) || d.c_in != 8 || g.wo > 256) return false;
    memset(&pl, 0, sizeof(pl));
    pl.n_img = d.n; pl.ho = g.ho; pl.wo = g.wo; pl.kh = d.kh; pl.kw = d.kw; pl.stride = d.stride; pl.pad = d.pad;
    pl.c_in = d.c_in; pl.c_out = d.c_out;
    pl.kc = 8 * d.c_in;
    pl.nc = chunk_bytes(d.c_out);
    const int per_tile = kTileM / pl.kc;
    pl.mtiles = (d.kh + per_tile - 1) / per_tile;
    if (pl.nc < 32 || d.c_out > 256 || pl.mtiles * d.c_out > 512) return false;
    pl.kp = (g.wo + 31) / 32 * 32;
    pl.span = pl.mtiles * per_tile;
    pl.rows_total = g.taps * d.c_in;
    const int most = pl.span > d.stride ? pl.span : d.stride;   // what the ring advances at the start of an image
    for (int stages = 4; stages >= 2; --stages) {
        // `stages` output rows in flight, with one start of an image among them (or each its own, in images of few rows)
        const int advance = g.ho >= stages - 1 ? (stages - 2) * d.stride + most : (stages - 1) * most;
        int slots = (200 * 1024 - stages * pl.kp * d.c_out) / (pl.kp * pl.kc);
        slots -= slots % per_tile;
        if (slots < advance + pl.span) continue;
        pl.num_stages = stages;
        pl.slots = advance + pl.span + per_tile - 1;
        pl.slots -= pl.slots % per_tile;
        break;
    }
    if (!pl.num_stages) return false;
    // a row adds at most wo * 127 * 127 to an int32 sum
    const int cap = ctas < kWgradTargetCtas ? ctas : kWgradTargetCtas, rows = d.n * g.ho, exact = 130000 / g.wo;
    int per = (rows + cap - 1) / cap;
    if (per > exact) per = exact;
    pl.rows_per_split = per;
    pl.num_splits = (rows + per - 1) / per;
    return true;
}

// int32 slices of partial sums the weight-gradient GEMM leaves, at most
int wgrad_slices(const eoq_conv_desc_t &d, const Geometry &g)
{
    WgradPatchPlan wp;
    if (plan_wgrad_patch(wp, d, g.ho, g.wo)) return wp.num_splits;
    WgradRowsPlan rp;
    if (plan_wgrad_rows(rp, d, g, kWgradTargetCtas)) return rp.num_splits;
    WgradParams p;
    return plan_wgrad(p, d, g, kWgradTargetCtas) ? p.num_k_splits : 0;
}

}  // namespace

// ================================================================================= handle

extern "C" int eoq_create(eoq_handle_t *handle, int device)
{
    if (!handle) return EOQ_ERR_BAD_ARG;
    *handle = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return EOQ_ERR_CUDA;
    if (!load_driver_entry_points()) return EOQ_ERR_CUDA;
    Handle *h = new (std::nothrow) Handle();
    if (!h) return EOQ_ERR_BAD_ARG;
    h->device = device;
    h->last_cuda_error = 0;
    h->dev = nullptr;
    h->launches = 0;
    h->profiling = false;
    h->force_timeout = false;
    h->gemm_only = false;
    h->hook = ReduceHook{nullptr, nullptr};
    h->num_records = 0;
    h->records = nullptr;
    // two attributes: cudaGetDeviceProperties took 2.5 of the call's 3.1 ms, and a training step creates five handles
    int major = 0;
    cudaError_t e = cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
    if (e == cudaSuccess) {
        h->gemm_ctas = h->sm_count;
        if (major != 10) {
            delete h;
            return EOQ_ERR_UNSUPPORTED;  // the kernels are sm_100a only
        }
        e = cudaMalloc(reinterpret_cast<void **>(&h->dev), round256(sizeof(DeviceState)) + kSqTiles * sizeof(int16_t));
    }
    if (e == cudaSuccess) e = cudaMemset(h->dev, 0, sizeof(DeviceState));
    h->tile_shift = reinterpret_cast<int16_t *>(reinterpret_cast<char *>(h->dev) + round256(sizeof(DeviceState)));
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        if (h->dev) cudaFree(h->dev);
        delete h;
        return EOQ_ERR_CUDA;
    }
    *handle = reinterpret_cast<eoq_handle_t>(h);
    return EOQ_OK;
}

extern "C" int eoq_destroy(eoq_handle_t handle)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h) return EOQ_ERR_BAD_ARG;
    cudaSetDevice(h->device);
    cudaDeviceSynchronize();
    if (h->dev) cudaFree(h->dev);
    if (h->records) {
        for (int i = 0; i < h->num_records; ++i) {
            cudaEventDestroy(h->records[i].begin);
            cudaEventDestroy(h->records[i].end);
        }
        delete[] h->records;
    }
    delete h;
    return EOQ_OK;
}

extern "C" int eoq_profile_start(eoq_handle_t handle)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h) return EOQ_ERR_BAD_ARG;
    if (!h->records) {
        h->records = new (std::nothrow) ProfRecord[kMaxProfRecords];
        if (!h->records) return EOQ_ERR_BAD_ARG;
    }
    for (int i = 0; i < h->num_records; ++i) {
        cudaEventDestroy(h->records[i].begin);
        cudaEventDestroy(h->records[i].end);
    }
    h->num_records = 0;
    h->profiling = true;
    return EOQ_OK;
}

extern "C" int eoq_profile_stop(eoq_handle_t handle, int launches[EOQ_PROF_KINDS], double milliseconds[EOQ_PROF_KINDS])
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !launches || !milliseconds) return EOQ_ERR_BAD_ARG;
    h->profiling = false;
    cudaError_t e = cudaDeviceSynchronize();
    for (int k = 0; k < EOQ_PROF_KINDS; ++k) {
        launches[k] = 0;
        milliseconds[k] = 0.0;
    }
    for (int i = 0; i < h->num_records && e == cudaSuccess; ++i) {
        float ms = 0.f;
        e = cudaEventElapsedTime(&ms, h->records[i].begin, h->records[i].end);
        launches[h->records[i].kind] += 1;
        milliseconds[h->records[i].kind] += ms;
    }
    return record(h, e);
}

extern "C" int eoq_profile_gemm_only(eoq_handle_t handle, int on)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h) return EOQ_ERR_BAD_ARG;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess && h->gemm_only && !on) {
        // the GEMMs that ran without their consumers left maxima in the reduction cells
        e = launch_reset_cells(h->dev, nullptr);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    h->gemm_only = on != 0;
    return record(h, e);
}

extern "C" int eoq_set_reduce_hook(eoq_handle_t handle, eoq_reduce_fn fn, void *user)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h) return EOQ_ERR_BAD_ARG;
    h->hook = ReduceHook{fn, user};
    return EOQ_OK;
}

extern "C" int eoq_set_gemm_ctas(eoq_handle_t handle, int ctas)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || ctas < 0) return EOQ_ERR_BAD_ARG;
    h->gemm_ctas = (ctas == 0 || ctas > h->sm_count) ? h->sm_count : ctas;
    return EOQ_OK;
}

extern "C" unsigned long long eoq_launch_count(eoq_handle_t handle)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    return h ? h->launches : 0ull;
}

namespace {

// Brackets one tensor-core kernel launch with events while profiling is on.
struct ProfScope {
    Handle *h;
    cudaStream_t s;
    ProfRecord *r;
    ProfScope(Handle *h_, int kind, cudaStream_t s_) : h(h_), s(s_), r(nullptr)
    {
        if (!h->profiling || h->num_records >= kMaxProfRecords) return;
        ProfRecord *c = &h->records[h->num_records];
        if (cudaEventCreate(&c->begin) != cudaSuccess) return;
        if (cudaEventCreate(&c->end) != cudaSuccess) {
            cudaEventDestroy(c->begin);
            return;
        }
        c->kind = kind;
        ++h->num_records;
        r = c;
        cudaEventRecord(r->begin, s);
    }
    ~ProfScope()
    {
        if (r) cudaEventRecord(r->end, s);
    }
};

}  // namespace

extern "C" int eoq_last_status(eoq_handle_t handle, void *stream, unsigned *bits)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !bits) return EOQ_ERR_BAD_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    unsigned v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, &h->dev->status, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&h->dev->status, 0, sizeof(unsigned), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && (v & EOQ_DEV_TIMEOUT)) {
        // a kernel that gave up may not have put the reduction cells back to zero
        e = launch_reset_cells(h->dev, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(&h->dev->ticket, 0, sizeof(unsigned), s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    *bits = v;
    return record(h, e);
}

extern "C" int eoq_last_cuda_error(eoq_handle_t handle)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    return h ? h->last_cuda_error : static_path_last_cuda_error();
}

extern "C" const char *eoq_status_string(int status)
{
    switch (status) {
        case EOQ_OK: return "ok";
        case EOQ_ERR_BAD_ARG: return "bad argument";
        case EOQ_ERR_ALIGNMENT: return "alignment (16-byte pointers, channels in multiples of 16)";
        case EOQ_ERR_UNSUPPORTED: return "unsupported geometry or device";
        case EOQ_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case EOQ_ERR_RANGE: return "scalar code out of range";
        case EOQ_ERR_CUDA: return "CUDA error";
        default: return "unknown status";
    }
}

// ================================================================================= workspace

extern "C" int eoq_workspace_size(const eoq_conv_desc_t *desc, int pass, size_t *bytes)
{
    Geometry g;
    if (!bytes) return EOQ_ERR_BAD_ARG;
    int st = check_desc(desc, &g);
    if (st != EOQ_OK) return st;
    const BorderClasses bc = border_classes(*desc, g);
    switch (pass) {
        case EOQ_PASS_FWD:  // b1 table, then the row-padded weights of the filter-row path
            *bytes = round256((size_t)bc.nrc * bc.ncc * desc->c_out * sizeof(int32_t)) +
                     (use_row_window(*desc, g.wo) ? round256((size_t)desc->c_out * desc->kh * 8 * desc->c_in) : 0);
            return EOQ_OK;
        // Sums behind room for a copy of the weights.  The 16-bit words of the sums fill half of theirs, and no kernel makes the copy
        // any more.  The size is part of the interface all the same: callers keep buffers of it, and the allocation-free entry point
        // accepts and refuses geometries by it.
        case EOQ_PASS_DGRAD:
            *bytes = round256(g.w_elems) + round256(g.in_elems * sizeof(int32_t));
            return EOQ_OK;
        case EOQ_PASS_WGRAD: {  // per-tap error sums, reduction cell, int64 sums, split-K slices
            const size_t slices = (size_t)wgrad_slices(*desc, g) * g.w_elems * sizeof(int32_t);
            *bytes = kTapReplicas * round256((size_t)desc->c_out * g.taps * sizeof(long long)) + 256 +
                     round256(g.w_elems * sizeof(long long)) + round256(slices);
            return EOQ_OK;
        }
        default: return EOQ_ERR_BAD_ARG;
    }
}

static int check_workspace(const eoq_conv_desc_t *desc, int pass, const void *ws, size_t ws_bytes)
{
    size_t need = 0;
    int st = eoq_workspace_size(desc, pass, &need);
    if (st != EOQ_OK) return st;
    if (need == 0) return EOQ_OK;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) || ws_bytes < need) return EOQ_ERR_WORKSPACE;
    return EOQ_OK;
}

// ================================================================================= forward

// Forward chain behind eoq_conv_fwd and eoq_conv_fwd_dev.  The scalars are the three host codes, or the device
// array `scal_dev`.  `prep` holds what eoq_weight_prep derives from the weights; when it is null the call derives it
// itself into `workspace` (two more kernels on the forward chain).
static int conv_fwd_impl(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *x, const int32_t *x_exp,
                         int32_t b1_c, int32_t gamma_c, int32_t b2_c, const int32_t *scal_dev, const int8_t *w,
                         const void *prep, const int8_t *shortcut, int relu, int8_t *x5, int16_t *x2, uint8_t *relu_mask,
                         int32_t *acc_dump, void *workspace, size_t workspace_bytes, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    Geometry g;
    if (!h || !x || !w || !x5) return EOQ_ERR_BAD_ARG;
    int st = check_desc(desc, &g);
    if (st != EOQ_OK) return st;
    if (!aligned16(x) || !aligned16(w) || !aligned16(x5) || !aligned16(shortcut) || !aligned16(x2) ||
        !aligned16(relu_mask) || !aligned16(acc_dump))
        return EOQ_ERR_ALIGNMENT;
    if (b1_c < -32768 || b1_c > 32767 || gamma_c < -32768 || gamma_c > 32767 || b2_c < -32768 || b2_c > 32767)
        return EOQ_ERR_RANGE;
    const eoq_conv_desc_t &d = *desc;
    // the accumulator with its b1 term must fit int32: taps * c_in * (127 + |b1|) * 127 < 2^31
    if ((double)g.taps * d.c_in * (127.0 + (b1_c < 0 ? -b1_c : b1_c)) * 127.0 >= 2147483647.0 - 16777216.0) return EOQ_ERR_RANGE;
    const bool row_window = use_row_window(d, g.wo);
    if (d.c_in == 8 && !row_window) return EOQ_ERR_UNSUPPORTED;
    // with device scalars b1 is unknown here: the table is applied whenever prepared weights are at hand
    const bool use_b1 = scal_dev ? prep != nullptr : b1_c != 0;
    if (scal_dev && !prep && row_window) return EOQ_ERR_BAD_ARG;
    if (!prep && (use_b1 || row_window) && (st = check_workspace(desc, EOQ_PASS_FWD, workspace, workspace_bytes)) != EOQ_OK) return st;
    if (prep && (reinterpret_cast<uintptr_t>(prep) & 255)) return EOQ_ERR_ALIGNMENT;
    char *prep_base = prep ? static_cast<char *>(const_cast<void *>(prep)) : static_cast<char *>(workspace);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int w_mem = d.w + 2 * d.x_wmargin;

    IgemmParams p;
    memset(&p, 0, sizeof(p));
    PatchPlan pl;
    memset(&pl, 0, sizeof(pl));
    const bool patch = d.stride == 1 && d.kh == d.kw && d.x_wmargin == 0 &&
                       plan_stride1(p, pl, d.n, d.c_in, g.ho, g.wo, d.kh, d.pad, d.c_out, h->sm_count, h->gemm_ctas);
    p.M = d.n * g.ho * g.wo;
    p.N = d.c_out;
    p.hq = g.ho;
    p.wq = g.wo;
    p.src_stride = d.stride;
    p.base_h = -d.pad;
    int8_t *w_rows = nullptr;
    RowsPlan rp;
    bool by_rows = false;
    if (patch) {
        for (int t = 0; t < g.taps; ++t) p.tap_b[t] = (unsigned char)t;
    } else if (row_window) {
        // K sub-tile = one filter row (8 pixels x c_in channels); the map's W axis already steps by the stride
        by_rows = plan_rows(p, rp, d, g, h->gemm_ctas);
        if (!by_rows) plan_igemm(p, 8 * d.c_in, d.kh, h->sm_count);
        p.src_stride_w = 1;
        p.base_w = 0;
        for (int t = 0; t < d.kh; ++t) {
            p.tap_dh[t] = (unsigned char)t;
            p.tap_dw[t] = 0;
            p.tap_b[t] = (unsigned char)t;
        }
        const BorderClasses bc0 = border_classes(d, g);
        w_rows = reinterpret_cast<int8_t *>(prep_base) + round256((size_t)bc0.nrc * bc0.ncc * d.c_out * sizeof(int32_t));
        if (!prep) {
            ProfScope prof(h, EOQ_PROF_FWD_AUX, s);
            cudaError_t e = launch_weight_pad_rows(w, w_rows, d.c_out, d.kh, d.kw, d.c_in, s);
            if (e != cudaSuccess) return record(h, e);
            count_launches(h, 1);
        }
    } else {
        plan_igemm(p, d.c_in, g.taps, h->sm_count);
        p.src_stride_w = d.stride;
        p.base_w = d.x_wmargin - d.pad;
        for (int t = 0; t < g.taps; ++t) {
            p.tap_dh[t] = (unsigned char)(t / d.kw);
            p.tap_dw[t] = (unsigned char)(t % d.kw);
            p.tap_b[t] = (unsigned char)t;
        }
        plan_few_tiles(p, h->gemm_ctas);
    }
    p.out_h = g.ho;
    p.out_w = g.wo;
    p.out_step = 1;
    p.epilogue = kEpiForward;
    p.x_exp = x_exp;
    p.b1_c = b1_c;
    p.gamma_c = gamma_c;
    p.b2_c = b2_c;
    p.scal_dev = scal_dev;
    p.k_total = g.taps * d.c_in;
    p.shortcut = shortcut;
    p.relu = relu ? 1 : 0;
    p.x5 = x5;
    p.x2 = x2;
    p.relu_mask = relu_mask;
    p.acc_out = acc_dump;
    p.dev = h->dev;
    if (use_b1) {
        const BorderClasses bc = border_classes(d, g);
        if (bc.nrc * bc.ncc > kMaxBorderClasses) return EOQ_ERR_UNSUPPORTED;
        p.b1_table = reinterpret_cast<const int32_t *>(prep_base);
        p.b1_nlo_h = bc.nlo_h; p.b1_nhi_h = bc.nhi_h; p.b1_nrc = bc.nrc;
        p.b1_nlo_w = bc.nlo_w; p.b1_nhi_w = bc.nhi_w; p.b1_ncc = bc.ncc;
        if (!prep) {
            ProfScope prof(h, EOQ_PROF_FWD_AUX, s);
            cudaError_t e = launch_b1_weight_table(w, reinterpret_cast<int32_t *>(prep_base), d, bc, s);
            if (e != cudaSuccess) return record(h, e);
            count_launches(h, 1);
        }
    }
    CUtensorMap map_a, map_b;
    if (patch) {
        if (!make_patch_map(&map_a, x, d.n, d.h, d.w, d.c_in, p.kc, pl.pw, pl.r_rows + d.kh - 1) ||
            !make_weight_map(&map_b, w, d.c_out, g.taps, d.c_in, p.kc, p.tile_n))
            return EOQ_ERR_UNSUPPORTED;
        const int ptiles = p.num_m_tiles * p.num_n_tiles;
        count_launches(h, 1);
        ProfScope prof(h, EOQ_PROF_IGEMM_FWD, s);
        const int grid = persistent_grid(ptiles, h->gemm_ctas);
        plan_epilogue(p, grid);
        return record(h, launch_igemm_patch(p, pl, map_a, map_b, grid, s));
    }
    if (by_rows) {
        if (!make_input_rows_map(&map_a, x, d.n, d.h, (size_t)w_mem * d.c_in, rp.row_pitch / 8, (rp.r_rows - 1) * d.stride + d.kh) ||
            !make_weight_map(&map_b, w_rows, d.c_out, d.kh, 8 * d.c_in, 8 * d.c_in, p.tile_n))
            return EOQ_ERR_UNSUPPORTED;
        count_launches(h, 1);
        ProfScope prof(h, EOQ_PROF_IGEMM_FWD, s);
        const int grid = persistent_grid(p.num_m_tiles, h->gemm_ctas), rows = (p.num_m_tiles + grid - 1) / grid * rp.r_rows;
        p.ep_groups = rows >= 3 && p.tile_n <= 64 ? 4 : (rows >= 2 || p.tile_n < 64 ? 2 : 1);
        if (p.tile_n / 16 < 4 / p.ep_groups) p.ep_groups = p.tile_n >= 32 ? 2 : 4;   // at least one 16-column group per warp
        return record(h, launch_igemm_rows(p, rp, map_a, map_b, grid, s));
    }
    if (row_window) {
        if (!make_row_window_map(&map_a, x, d.n, d.h, w_mem, d.c_in, d.x_wmargin - d.pad, g.wo, g.ho, d.stride, d.pad, p.a_rows) ||
            !make_weight_map(&map_b, w_rows, d.c_out, d.kh, 8 * d.c_in, 8 * d.c_in, p.tile_n))
            return EOQ_ERR_UNSUPPORTED;
    } else if (!make_im2col_map(&map_a, x, d.n, d.h, w_mem, d.c_in, d.x_wmargin - d.pad, -d.pad, g.wo, g.ho, d.stride, p.kc,
                                p.a_rows) ||
               !make_weight_map(&map_b, w, d.c_out, g.taps, d.c_in, p.kc, p.tile_n)) {
        return EOQ_ERR_UNSUPPORTED;
    }
    const int tiles = p.num_m_tiles * p.num_n_tiles;
    count_launches(h, 1);
    ProfScope prof(h, EOQ_PROF_IGEMM_FWD, s);
    const int grid = persistent_grid(tiles, h->gemm_ctas);
    plan_epilogue(p, grid);
    return record(h, launch_igemm(p, map_a, map_b, grid * p.split, s));
}

extern "C" int eoq_conv_fwd(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *x, const int32_t *x_exp,
                            int32_t b1_c, const int8_t *w, int32_t gamma_c, int32_t b2_c, const int8_t *shortcut,
                            int relu, int8_t *x5, int16_t *x2, uint8_t *relu_mask, int32_t *acc_dump, void *workspace,
                            size_t workspace_bytes, void *stream)
{
    return conv_fwd_impl(handle, desc, x, x_exp, b1_c, gamma_c, b2_c, nullptr, w, nullptr, shortcut, relu, x5, x2, relu_mask,
                         acc_dump, workspace, workspace_bytes, stream);
}

extern "C" int eoq_conv_fwd_dev(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *x, const int32_t *x_exp,
                                const int32_t *scalars, const int8_t *w, const void *w_prep, const int8_t *shortcut,
                                int relu, int8_t *x5, int16_t *x2, uint8_t *relu_mask, void *stream)
{
    if (!scalars || (reinterpret_cast<uintptr_t>(scalars) & 3)) return EOQ_ERR_BAD_ARG;
    return conv_fwd_impl(handle, desc, x, x_exp, 0, 128, 0, scalars, w, w_prep, shortcut, relu, x5, x2, relu_mask, nullptr,
                         nullptr, 0, stream);
}

extern "C" int eoq_weight_prep_size(const eoq_conv_desc_t *desc, size_t *bytes)
{
    return eoq_workspace_size(desc, EOQ_PASS_FWD, bytes);
}

extern "C" int eoq_weight_prep(eoq_handle_t handle, int num, const eoq_conv_desc_t *descs, const int8_t *const *w,
                               void *const *prep, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || num <= 0 || !descs || !w || !prep) return EOQ_ERR_BAD_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    // every argument is checked before the first launch
    for (int i = 0; i < num; ++i) {
        Geometry g;
        int st = check_desc(&descs[i], &g);
        if (st != EOQ_OK) return st;
        if (!w[i] || !prep[i]) return EOQ_ERR_BAD_ARG;
        if (!aligned16(w[i]) || (reinterpret_cast<uintptr_t>(prep[i]) & 255)) return EOQ_ERR_ALIGNMENT;
        const BorderClasses bc = border_classes(descs[i], g);
        if (bc.nrc * bc.ncc > kMaxBorderClasses) return EOQ_ERR_UNSUPPORTED;
    }
    for (int base = 0; base < num; base += kPrepChunk) {
        PrepBatch b;
        memset(&b, 0, sizeof(b));
        b.num = num - base < kPrepChunk ? num - base : kPrepChunk;
        int blocks = 0;
        for (int k = 0; k < b.num; ++k) {
            const eoq_conv_desc_t &d = descs[base + k];
            Geometry g;
            check_desc(&d, &g);
            PrepItem &it = b.item[k];
            it.w = w[base + k];
            it.table = static_cast<int32_t *>(prep[base + k]);
            it.d = d;
            it.ho = g.ho;
            it.wo = g.wo;
            it.bc = border_classes(d, g);
            it.w_rows = use_row_window(d, g.wo)
                            ? static_cast<int8_t *>(prep[base + k]) + round256((size_t)it.bc.nrc * it.bc.ncc * d.c_out * sizeof(int32_t))
                            : nullptr;
            b.first_block[k] = blocks;
            blocks += d.c_out;
        }
        b.first_block[b.num] = blocks;
        ProfScope prof(h, EOQ_PROF_FWD_AUX, s);
        cudaError_t e = launch_weight_prep(b, s);
        if (e != cudaSuccess) return record(h, e);
        count_launches(h, 1);
    }
    return EOQ_OK;
}

// ================================================================================= error back-propagation

// The error join that takes e4 as its first operand, run behind the dgrad (eoq_conv_dgrad_join_head): the join's first
// pass rides on Q_e, its second pass follows; `next` there is the head of the layer that consumes the joined error.
struct JoinCall {
    const int8_t *b;
    const int32_t *b_exp;
    const uint8_t *mask_b;
    int8_t *out;
    int32_t *out_exp;
    long long *sum_out;
    const NextHeadArgs *next;
};

// A strided 1x1 filter without padding reaches only the pixels on the stride grid: its one GEMM leaves compact sums
// [n][hq][wq][c_in] and Q_e scatters them into the full tensor (zeros elsewhere), so nothing is cleared.
static bool compact_sums(const eoq_conv_desc_t &d)
{
    return d.kh == 1 && d.kw == 1 && d.pad == 0 && d.stride > 1 && (size_t)d.n * d.h * d.w * (d.c_in / 16) <= 0xffffffffull;
}

// First tap of each class of a launch, in error pixels (what the im2col loads start from).
struct ClassCorners {
    int dh[kMaxClasses], dw[kMaxClasses];
};

// The residue classes (y mod stride, x mod stride) of the input pixels that some tap reaches: within a class the taps kh with
// (y + pad - kh) divisible by the stride form a unit-stride correlation over e3.  They write disjoint pixels, so up to kMaxClasses of
// them share a launch, each with its share of the CTAs.  launch(classes, corners) is called for every launch, its GEMMs planned.
template <typename Launch>
static int each_class_launch(const eoq_conv_desc_t &d, bool compact, int sm_count, int ctas, Launch launch)
{
    IgemmClasses cl;
    ClassCorners at;
    cl.num = 0;
    auto flush = [&]() -> int {
        if (cl.num == 0) return EOQ_OK;
        plan_classes(cl, ctas);
        const int st = launch(cl, at);
        cl.num = 0;
        return st;
    };
    for (int py = 0; py < d.stride && py < d.h; ++py)
        for (int px = 0; px < d.stride && px < d.w; ++px) {
            int dh[16], dw[16], kh_of[16], kw_of[16], nh = 0, nw = 0, min_h = 0, min_w = 0;
            for (int kh = 0; kh < d.kh; ++kh)
                if ((py + d.pad - kh) % d.stride == 0) {
                    // floor division is exact here; negative quotients are rows above the image
                    dh[nh] = (py + d.pad - kh) / d.stride;
                    kh_of[nh] = kh;
                    if (dh[nh] < min_h) min_h = dh[nh];
                    ++nh;
                }
            for (int kw = 0; kw < d.kw; ++kw)
                if ((px + d.pad - kw) % d.stride == 0) {
                    dw[nw] = (px + d.pad - kw) / d.stride;
                    kw_of[nw] = kw;
                    if (dw[nw] < min_w) min_w = dw[nw];
                    ++nw;
                }
            if (nh == 0 || nw == 0) continue;  // no tap reaches this class: its sums stay zero
            int st = EOQ_OK;
            if (cl.num == kMaxClasses && (st = flush()) != EOQ_OK) return st;
            at.dh[cl.num] = min_h;
            at.dw[cl.num] = min_w;
            IgemmParams &p = cl.p[cl.num++];
            memset(&p, 0, sizeof(p));
            p.hq = (d.h - py + d.stride - 1) / d.stride;
            p.wq = (d.w - px + d.stride - 1) / d.stride;
            p.M = d.n * p.hq * p.wq;
            p.N = d.c_in;
            p.b_mn = 1;   // (the weights stay where they are, as for the patch kernel)
            plan_igemm(p, d.c_out, nh * nw, sm_count);
            p.src_stride = 1;
            p.src_stride_w = 1;
            p.base_h = min_h;
            p.base_w = min_w;
            for (int a = 0; a < nh; ++a)
                for (int b = 0; b < nw; ++b) {
                    const int t = a * nw + b;
                    if (dh[a] - min_h > 255 || dw[b] - min_w > 255) return EOQ_ERR_UNSUPPORTED;
                    p.tap_dh[t] = (unsigned char)(dh[a] - min_h);
                    p.tap_dw[t] = (unsigned char)(dw[b] - min_w);
                    p.tap_b[t] = (unsigned char)(kh_of[a] * d.kw + kw_of[b]);
                }
            p.out_h = compact ? p.hq : d.h;
            p.out_w = compact ? p.wq : d.w;
            p.out_step = compact ? 1 : d.stride;
            p.out_off_h = py;
            p.out_off_w = px;
            p.epilogue = kEpiDgrad;
        }
    return flush();
}

// `next`: the error head of the layer that consumes e4, fused into Q_e (null for the plain call); `jc`: see JoinCall
static int conv_dgrad_impl(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3, const int32_t *e3_exp,
                           const int8_t *w, int8_t *e4, int32_t *e4_exp, int64_t *sum_e4, int32_t *acc_dump,
                           const NextHeadArgs *next, void *workspace, size_t workspace_bytes, void *stream,
                           const JoinCall *jc = nullptr)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    Geometry g;
    if (!h || !e3 || !e3_exp || !w || !e4 || !e4_exp) return EOQ_ERR_BAD_ARG;
    int st = check_desc(desc, &g);
    if (st != EOQ_OK) return st;
    if (!aligned16(e3) || !aligned16(w) || !aligned16(e4) || !aligned16(acc_dump)) return EOQ_ERR_ALIGNMENT;
    if (desc->c_in % 16) return EOQ_ERR_UNSUPPORTED;  // 8 channels exist for the network input, which takes no error
    if (next) {
        if (!next->mask || !next->gamma || !next->e3 || !next->e3_exp) return EOQ_ERR_BAD_ARG;
        if (!aligned16(next->e3) || (next->x2 && !aligned16(next->x2)) || (reinterpret_cast<uintptr_t>(next->mask) & 1))
            return EOQ_ERR_ALIGNMENT;
        // the compact sums of a strided 1x1 filter are not laid out like the error tensor
        if (desc->kh == 1 && desc->kw == 1 && desc->pad == 0 && desc->stride > 1) return EOQ_ERR_UNSUPPORTED;
    }
    JoinStatArgs jstat{};
    const JoinStatArgs *jstat_p = nullptr;
    if (jc) {
        if (!jc->b || !jc->b_exp || !jc->out || !jc->out_exp || (g.in_elems % 16)) return EOQ_ERR_BAD_ARG;
        if (!aligned16(jc->b) || !aligned16(jc->out) || (reinterpret_cast<uintptr_t>(jc->mask_b) & 1)) return EOQ_ERR_ALIGNMENT;
        if (jc->next) {
            if (!jc->next->mask || !jc->next->gamma || !jc->next->e3 || !jc->next->e3_exp) return EOQ_ERR_BAD_ARG;
            if (!aligned16(jc->next->e3) || (jc->next->x2 && !aligned16(jc->next->x2)) ||
                (reinterpret_cast<uintptr_t>(jc->next->mask) & 1))
                return EOQ_ERR_ALIGNMENT;
        }
        if (desc->kh == 1 && desc->kw == 1 && desc->pad == 0 && desc->stride > 1) return EOQ_ERR_UNSUPPORTED;
        if (!h->hook.fn) {   // with replicas the join runs as its own two passes, each followed by its exchange
            jstat = JoinStatArgs{jc->b, jc->b_exp, jc->mask_b, jc->next ? jc->next->mask : nullptr};
            jstat_p = &jstat;
        }
    }
    // what follows Q_e when a join was asked for
    auto join_after = [&](cudaError_t e, cudaStream_t st) -> int {
        if (e != cudaSuccess || !jc) return record(h, e);
        ProfScope prof(h, EOQ_PROF_GLUE, st);
        if (jstat_p) {
            count_launches(h, 1);
            return record(h, launch_join_second(e4, e4_exp, jc->b, jc->b_exp, jc->mask_b, g.in_elems, jc->out, jc->out_exp, jc->sum_out,
                                                jc->next, h->dev, h->sm_count, st));
        }
        count_launches(h, 2);
        const NextHeadArgs *n = jc->next;
        return record(h, launch_join(e4, e4_exp, jc->b, jc->b_exp, jc->mask_b, g.in_elems, jc->out, jc->out_exp, jc->sum_out,
                                     n ? n->mask : nullptr, n ? n->x2 : nullptr, n ? n->gamma : nullptr, n ? n->e3 : nullptr,
                                     n ? n->e3_exp : nullptr, n ? n->sum_e1 : nullptr, n ? n->sum_e1x2 : nullptr, h->dev, h->sm_count,
                                     st, h->hook));
    };
    if ((st = check_workspace(desc, EOQ_PASS_DGRAD, workspace, workspace_bytes)) != EOQ_OK) return st;
    const eoq_conv_desc_t &d = *desc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

    // the GEMMs leave their sums as 16-bit words in the workspace, or as int32 where the caller wants them
    uint16_t *const sums16 = acc_dump ? nullptr : reinterpret_cast<uint16_t *>(static_cast<char *>(workspace) + round256(g.w_elems));
    auto code_sums = [&](cudaStream_t st) {   // Q_e over the whole tensor, behind the GEMMs
        return acc_dump ? launch_sq_i32(acc_dump, e3_exp, -7, g.in_elems, e4, e4_exp, reinterpret_cast<long long *>(sum_e4), true, h->dev,
                                        h->sm_count, st, h->hook)
                        : launch_sq_sums(sums16, e3_exp, -7, g.in_elems, e4, e4_exp, reinterpret_cast<long long *>(sum_e4), h->dev,
                                         h->sm_count, st, h->hook, next, jstat_p);
    };
    cudaError_t e;

    // sums that the kernels behind the GEMM add into; it clears them (one the caller also names for the join or the head is
    // written there: the later value counts)
    if (sum_e4 && jc && (void *)sum_e4 == (void *)jc->sum_out) sum_e4 = nullptr;
    const NextHeadArgs *const any_next = jc ? jc->next : next;
    long long *const zero_sums[4] = {reinterpret_cast<long long *>(sum_e4), jc ? jc->sum_out : nullptr, any_next ? any_next->sum_e1 : nullptr,
                                     any_next ? any_next->sum_e1x2 : nullptr};

    if (d.stride == 1 && d.kh == d.kw && d.kh - 1 - d.pad >= 0) {
        // stride 1: one correlation of e3 with the flipped filter, padding k - 1 - pad
        IgemmParams p;
        memset(&p, 0, sizeof(p));
        PatchPlan pl;
        memset(&pl, 0, sizeof(pl));
        // the weights are read where they are, [c_out][tap][c_in]: the reduction (c_out) is their slow axis, so
        // they reach the MMA as MN-major atoms of b_row input channels
        p.b_mn = 1;
        if (plan_stride1(p, pl, d.n, d.c_out, d.h, d.w, d.kh, d.kh - 1 - d.pad, d.c_in, h->sm_count, h->gemm_ctas)) {
            for (int a = 0; a < d.kh; ++a)
                for (int b = 0; b < d.kw; ++b) p.tap_b[a * d.kw + b] = (unsigned char)((d.kh - 1 - a) * d.kw + (d.kw - 1 - b));
            p.out_h = d.h;
            p.out_w = d.w;
            p.out_step = 1;
            p.epilogue = kEpiDgrad;
            memcpy(p.zero_sums, zero_sums, sizeof(zero_sums));
            p.acc_out = acc_dump;
            p.sums16 = sums16;
            p.dev = h->dev;
            p.next_mask = next ? next->mask : nullptr;
            CUtensorMap map_a, map_b;
            if (!make_patch_map(&map_a, e3, d.n, g.ho, g.wo, d.c_out, p.kc, pl.pw, pl.r_rows + d.kh - 1) ||
                !make_weight_map(&map_b, w, d.c_out, g.taps, d.c_in, p.b_row, p.kc))
                return EOQ_ERR_UNSUPPORTED;
            const int ptiles = p.num_m_tiles * p.num_n_tiles;
            count_launches(h, 1);
            {
                ProfScope prof(h, EOQ_PROF_IGEMM_DGRAD, s);
                const int grid = persistent_grid(ptiles, h->gemm_ctas);
                plan_epilogue(p, grid);
                e = launch_igemm_patch(p, pl, map_a, map_b, grid, s);
            }
            if (e != cudaSuccess || h->gemm_only) return record(h, e);
            {
                ProfScope prof(h, EOQ_PROF_DGRAD_AUX, s);
                e = code_sums(s);
            }
            count_launches(h, 1);
            return join_after(e, s);
        }
    }
    // a class no tap reaches (e.g. the odd pixels of a strided 1x1 filter) keeps zero sums: clear first
    bool any_empty = false;
    for (int r = 0; r < d.stride; ++r) {
        bool hit_h = false, hit_w = false;
        for (int kh = 0; kh < d.kh; ++kh) hit_h |= (r + d.pad - kh) % d.stride == 0;
        for (int kw = 0; kw < d.kw; ++kw) hit_w |= (r + d.pad - kw) % d.stride == 0;
        any_empty |= (r < d.h && !hit_h) || (r < d.w && !hit_w);
    }
    const bool compact = !acc_dump && compact_sums(d);
    if (any_empty && !compact) {
        e = acc_dump ? cudaMemsetAsync(acc_dump, 0, g.in_elems * sizeof(int32_t), s)
                     : cudaMemsetAsync(sums16, 0, g.in_elems * sizeof(uint16_t), s);
        if (e != cudaSuccess) return record(h, e);
    }
    int classes = 0;
    st = each_class_launch(d, compact, h->sm_count, h->gemm_ctas, [&](IgemmClasses &cl, const ClassCorners &at) -> int {
        for (int k = 0; k < cl.num; ++k) {
            IgemmParams &p = cl.p[k];
            memcpy(p.zero_sums, zero_sums, sizeof(zero_sums));
            p.acc_out = acc_dump;
            p.sums16 = sums16;
            p.dev = h->dev;
            p.next_mask = next ? next->mask : nullptr;
            if (!make_im2col_map(&cl.map_a[k], e3, d.n, g.ho, g.wo, d.c_out, at.dw[k], at.dh[k], p.wq, p.hq, 1, p.kc, p.a_rows) ||
                !make_weight_map(&cl.map_b[k], w, d.c_out, g.taps, d.c_in, p.b_row, p.kc))
                return EOQ_ERR_UNSUPPORTED;
        }
        classes += cl.num;
        count_launches(h, 1);
        ProfScope prof(h, EOQ_PROF_IGEMM_DGRAD, s);
        const cudaError_t err = cl.num == 1 ? launch_igemm(cl.p[0], cl.map_a[0], cl.map_b[0], cl.first[1], s) : launch_igemm_classes(cl, s);
        if (err == cudaSuccess) return EOQ_OK;
        launch_reset_cells(h->dev, s);  // GEMMs already queued have touched the maximum cell
        return record(h, err);
    });
    if (st != EOQ_OK) return st;
    if (h->gemm_only) return EOQ_OK;
    if (classes == 0)   // no tap reaches any pixel: no GEMM ran
        for (long long *z : zero_sums)
            if (z && (e = cudaMemsetAsync(z, 0, sizeof(*z), s)) != cudaSuccess) return record(h, e);
    // Q_e over the whole tensor: the maximum is complete only now
    {
        ProfScope prof(h, EOQ_PROF_DGRAD_AUX, s);
        if (compact)
            e = launch_sq_sums_scatter(sums16, e3_exp, -7, d.n, d.h, d.w, d.c_in, d.stride, (d.h + d.stride - 1) / d.stride,
                                       (d.w + d.stride - 1) / d.stride, e4, e4_exp, reinterpret_cast<long long *>(sum_e4),
                                       h->dev, h->sm_count, s, h->hook);
        else
            e = code_sums(s);
    }
    count_launches(h, 1);
    return join_after(e, s);
}

extern "C" int eoq_conv_dgrad(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3,
                              const int32_t *e3_exp, const int8_t *w, int8_t *e4, int32_t *e4_exp, int64_t *sum_e4,
                              int32_t *acc_dump, void *workspace, size_t workspace_bytes, void *stream)
{
    return conv_dgrad_impl(handle, desc, e3, e3_exp, w, e4, e4_exp, sum_e4, acc_dump, nullptr, workspace, workspace_bytes, stream);
}

extern "C" int eoq_conv_dgrad_join_head(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3, const int32_t *e3_exp,
                                        const int8_t *w, int8_t *e4, int32_t *e4_exp, int64_t *sum_e4, const int8_t *b,
                                        const int32_t *b_exp, const uint8_t *mask_b, int8_t *out, int32_t *out_exp, int64_t *sum_out,
                                        const uint8_t *next_relu_mask, const int16_t *next_x2, const int32_t *next_gamma,
                                        int8_t *next_e3, int32_t *next_e3_exp, int64_t *next_sum_e1, int64_t *next_sum_e1x2,
                                        void *workspace, size_t workspace_bytes, void *stream)
{
    const NextHeadArgs next{next_relu_mask, next_x2, next_gamma, next_e3, next_e3_exp, reinterpret_cast<long long *>(next_sum_e1),
                            reinterpret_cast<long long *>(next_sum_e1x2)};
    const JoinCall jc{b, b_exp, mask_b, out, out_exp, reinterpret_cast<long long *>(sum_out), next_relu_mask ? &next : nullptr};
    return conv_dgrad_impl(handle, desc, e3, e3_exp, w, e4, e4_exp, sum_e4, nullptr, nullptr, workspace, workspace_bytes, stream, &jc);
}

extern "C" int eoq_conv_dgrad_head(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3, const int32_t *e3_exp,
                                   const int8_t *w, int8_t *e4, int32_t *e4_exp, int64_t *sum_e4, const uint8_t *next_relu_mask,
                                   const int16_t *next_x2, const int32_t *next_gamma, int8_t *next_e3, int32_t *next_e3_exp,
                                   int64_t *next_sum_e1, int64_t *next_sum_e1x2, void *workspace, size_t workspace_bytes,
                                   void *stream)
{
    const NextHeadArgs next{next_relu_mask, next_x2, next_gamma, next_e3, next_e3_exp, reinterpret_cast<long long *>(next_sum_e1),
                            reinterpret_cast<long long *>(next_sum_e1x2)};
    return conv_dgrad_impl(handle, desc, e3, e3_exp, w, e4, e4_exp, sum_e4, nullptr, &next, workspace, workspace_bytes, stream);
}

// ================================================================================= weight gradient

// The weight-gradient workspace: [tap sums][256 bytes with the maximum cell][int64 sums][split-K slices].
struct WgradSpace {
    long long *tap_sums;
    unsigned long long *max_cell;
    long long *acc;
    size_t acc_bytes;
    int32_t *parts;
};
static WgradSpace wgrad_space(const eoq_conv_desc_t &d, const Geometry &g, void *workspace)
{
    WgradSpace w;
    char *ws = static_cast<char *>(workspace);
    const size_t tap_bytes = kTapReplicas * round256((size_t)d.c_out * g.taps * sizeof(long long));   // (also 16-byte aligned cells)
    w.tap_sums = reinterpret_cast<long long *>(ws);
    w.max_cell = reinterpret_cast<unsigned long long *>(ws + tap_bytes);
    w.acc = reinterpret_cast<long long *>(ws + tap_bytes + 256);
    w.acc_bytes = round256(g.w_elems * sizeof(long long));
    w.parts = reinterpret_cast<int32_t *>(ws + tap_bytes + 256 + w.acc_bytes);
    return w;
}

static FinishItem finish_item(const eoq_conv_desc_t &d, const Geometry &g, const WgradSpace &w, const int8_t *e3, const int32_t *e3_exp,
                              int32_t b1_c, const int32_t *b1_dev, int8_t *gq, int32_t *g_exp, int num_parts)
{
    FinishItem it;
    memset(&it, 0, sizeof(it));
    it.e3 = e3;
    it.e3_exp = e3_exp;
    it.b1_dev = b1_dev;
    it.b1_c = b1_c;
    it.use_b1 = b1_dev != nullptr || b1_c != 0;   // a device-resident b1 may be anything: its term is always formed
    it.tap_sums = w.tap_sums;
    it.max_cell = w.max_cell;
    it.acc = w.acc;
    it.num_parts = num_parts;
    it.parts = w.parts;
    it.g = gq;
    it.g_exp = g_exp;
    it.n = g.w_elems;
    it.pixels = (unsigned long long)d.n * g.ho * g.wo;
    it.d = d;
    it.bc = border_classes(d, g);
    it.ho = g.ho;
    it.wo = g.wo;
    return it;
}

// The b1 error sums of the batch.
static int finish_taps(Handle *h, const FinishBatch &b, TapsOrder order, cudaStream_t s)
{
    ProfScope prof(h, EOQ_PROF_WGRAD_TAPS, s);
    count_launches(h, 1);
    return record(h, launch_finish_taps(b, order, s));
}

// Sums and Q_g of the batch, whose GEMMs and b1 error sums are in front on the stream.
static int finish_sums(Handle *h, const FinishBatch &b, cudaStream_t s)
{
    ProfScope prof(h, EOQ_PROF_WGRAD_AUX, s);
    count_launches(h, h->hook.fn ? 2 + b.num : 2);
    return record(h, launch_finish_sums(b, &h->dev->status, s, h->hook));
}

// Weight gradient behind eoq_conv_wgrad and eoq_conv_wgrad_dev: b1 is the host code b1_c, or the code at b1_dev.
// num_parts_out (eoq_conv_wgrad_gemm): the GEMM alone; the sums stay in the workspace for eoq_wgrad_finish and
// *num_parts_out tells it how many int32 slices there are.
static int conv_wgrad_impl(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3, const int32_t *e3_exp,
                           const int8_t *x, int32_t b1_c, const int32_t *b1_dev, int8_t *gq, int32_t *g_exp,
                           int64_t *acc_dump, void *workspace, size_t workspace_bytes, void *stream, int *num_parts_out = nullptr)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    Geometry g;
    const bool gemm_only = num_parts_out != nullptr || (h && h->gemm_only);
    if (!h || !e3 || !e3_exp || !x || (!num_parts_out && (!gq || !g_exp))) return EOQ_ERR_BAD_ARG;
    int st = check_desc(desc, &g);
    if (st != EOQ_OK) return st;
    if (!aligned16(e3) || !aligned16(x) || !aligned16(gq) || !aligned16(acc_dump)) return EOQ_ERR_ALIGNMENT;
    if (b1_c < -32768 || b1_c > 32767) return EOQ_ERR_RANGE;
    if ((st = check_workspace(desc, EOQ_PASS_WGRAD, workspace, workspace_bytes)) != EOQ_OK) return st;
    const eoq_conv_desc_t &d = *desc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

    const BorderClasses bc = border_classes(d, g);
    const bool use_b1 = b1_dev != nullptr || b1_c != 0;
    if (use_b1 && bc.nrc * bc.ncc > kMaxBorderClasses) return EOQ_ERR_UNSUPPORTED;
    const WgradSpace w = wgrad_space(d, g, workspace);
    // The b1 error sums run beside the GEMM (whose kernel leaves sums as [oc][tap][ic], the layout of g), launched behind it or in front;
    // then come the sums of its slices with Q_g.  A small layer is finished by one launch, which forms the b1 sums beside the GEMM too.
    FinishItem item = finish_item(d, g, w, e3, e3_exp, b1_c, b1_dev, gq, g_exp, 0);
    item.copy_out = reinterpret_cast<long long *>(acc_dump);
    FinishBatch batch;
    bool small = false, taps_first = false;
    // Fills in what the GEMM's plan says of its neighbours.  Its kernel clears the maximum's cell, and the tap sums' where they may be added up.
    auto begin = [&](int num_parts, auto &plan, bool beside) -> int {   // beside: the kernel can run beside them
        if (num_parts_out) *num_parts_out = num_parts;
        bool add = num_parts_out != nullptr;
        if (!gemm_only) {
            item.num_parts = num_parts;
            small = !h->profiling && finish_is_small(item, h->hook);   // (a profile brackets the b1 sums as a kind of their own)
            if (!small) plan_finish(batch, &item, 1, h->sm_count, h->gemm_ctas >= h->sm_count, h->hook);
            add = !small && use_b1 && batch.item[0].tap_add;
            taps_first = beside && use_b1 && !small && finish_taps_first(batch.item[0]);
        }
        plan.zero = add ? reinterpret_cast<int4 *>(w.tap_sums) : reinterpret_cast<int4 *>(w.max_cell);
        plan.zero_n16 = (unsigned)(reinterpret_cast<int4 *>(w.max_cell) + 1 - plan.zero);
        return taps_first ? finish_taps(h, batch, kTapsFirst, s) : EOQ_OK;
    };
    auto finish = [&](cudaError_t e, bool beside) -> int {
        if (e != cudaSuccess || gemm_only) return record(h, e);
        if (small) {
            count_launches(h, 1);
            return record(h, launch_finish_small(item, &h->dev->status, h->sm_count, beside && use_b1, s));
        }
        if (use_b1 && !taps_first && (st = finish_taps(h, batch, beside ? kTapsBeside : kTapsBehind, s)) != EOQ_OK) return st;
        return finish_sums(h, batch, s);
    };

    WgradPatchPlan wp;
    if (plan_wgrad_patch(wp, d, g.ho, g.wo, h->gemm_ctas < kWgradTargetCtas ? h->gemm_ctas : kWgradTargetCtas)) {
        wp.partials = w.parts;
        wp.dev = h->dev;
        CUtensorMap map_x, map_e;
        if (!make_patch_map(&map_x, x, d.n, d.h, d.w, d.c_in, wp.kc, wp.pw, wp.r_rows + d.kh - 1) ||
            !make_patch_map(&map_e, e3, d.n, g.ho, g.wo, d.c_out, wp.tile_n, wp.pw, wp.r_rows))
            return EOQ_ERR_UNSUPPORTED;
        if ((st = begin(wp.num_splits, wp, true)) != EOQ_OK) return st;
        wp.launch_early = use_b1 && !gemm_only && !taps_first;
        wp.wait_late = taps_first;
        count_launches(h, 1);
        cudaError_t e;
        {
            ProfScope prof(h, EOQ_PROF_WGRAD, s);
            e = launch_wgrad_patch(wp, map_x, map_e, s);
        }
        return finish(e, true);
    }

    const int w_mem = d.w + 2 * d.x_wmargin;
    WgradRowsPlan rp;
    if (plan_wgrad_rows(rp, d, g, h->gemm_ctas)) {
        rp.partials = w.parts;
        rp.dev = h->dev;
        CUtensorMap map_x, map_e;
        if (!make_matrix_map(&map_e, e3, (size_t)d.n * g.ho * g.wo, d.c_out, rp.nc, g.wo) ||
            !make_row_window_map(&map_x, x, d.n, d.h, w_mem, d.c_in, d.x_wmargin - d.pad, g.wo, g.ho, d.stride, d.pad, g.wo))
            return EOQ_ERR_UNSUPPORTED;
        if ((st = begin(rp.num_splits, rp, false)) != EOQ_OK) return st;
        count_launches(h, 1);
        cudaError_t e;
        {
            ProfScope prof(h, EOQ_PROF_WGRAD, s);
            e = launch_wgrad_rows(rp, map_x, map_e, s);
        }
        return finish(e, false);
    }

    WgradParams p;
    if (!plan_wgrad(p, d, g, h->gemm_ctas)) return EOQ_ERR_UNSUPPORTED;
    const bool row_window = p.row_window_kw != 0;
    p.partials = w.parts;
    p.dev = h->dev;

    cudaError_t e;
    CUtensorMap map_x, map_e;
    if (!make_matrix_map(&map_e, e3, (size_t)p.P, d.c_out, p.nc, p.pixels_per_stage)) return EOQ_ERR_UNSUPPORTED;
    if (row_window ? !make_row_window_map(&map_x, x, d.n, d.h, w_mem, d.c_in, d.x_wmargin - d.pad, g.wo, g.ho, d.stride, d.pad,
                                          p.pixels_per_stage)
                   : !make_im2col_map(&map_x, x, d.n, d.h, w_mem, d.c_in, d.x_wmargin - d.pad, -d.pad, g.wo, g.ho, d.stride,
                                      p.kc, p.pixels_per_stage))
        return EOQ_ERR_UNSUPPORTED;
    if ((st = begin(p.num_k_splits, p, true)) != EOQ_OK) return st;
    p.launch_early = use_b1 && !gemm_only && !taps_first;
    p.wait_late = taps_first;
    count_launches(h, 1);
    {
        ProfScope prof(h, EOQ_PROF_WGRAD, s);
        e = launch_wgrad(p, map_x, map_e, s);
    }
    return finish(e, true);
}

extern "C" int eoq_conv_wgrad(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3,
                              const int32_t *e3_exp, const int8_t *x, int32_t b1_c, int8_t *gq, int32_t *g_exp,
                              int64_t *acc_dump, void *workspace, size_t workspace_bytes, void *stream)
{
    return conv_wgrad_impl(handle, desc, e3, e3_exp, x, b1_c, nullptr, gq, g_exp, acc_dump, workspace, workspace_bytes, stream);
}

extern "C" int eoq_conv_wgrad_dev(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3,
                                  const int32_t *e3_exp, const int8_t *x, const int32_t *b1_c, int8_t *gq, int32_t *g_exp,
                                  void *workspace, size_t workspace_bytes, void *stream)
{
    // b1_c null: the layer has no bias in front of its convolution (the first layer of a network)
    return conv_wgrad_impl(handle, desc, e3, e3_exp, x, 0, b1_c, gq, g_exp, nullptr, workspace, workspace_bytes, stream);
}

extern "C" int eoq_conv_wgrad_gemm(eoq_handle_t handle, const eoq_conv_desc_t *desc, const int8_t *e3, const int32_t *e3_exp,
                                   const int8_t *x, void *workspace, size_t workspace_bytes, int *num_parts, void *stream)
{
    if (!num_parts) return EOQ_ERR_BAD_ARG;
    return conv_wgrad_impl(handle, desc, e3, e3_exp, x, 0, nullptr, nullptr, nullptr, nullptr, workspace, workspace_bytes, stream,
                           num_parts);
}

extern "C" int eoq_wgrad_finish(eoq_handle_t handle, int num, const eoq_conv_desc_t *descs, const int8_t *const *e3,
                                const int32_t *const *e3_exp, const int32_t *const *b1_c, int8_t *const *gq, int32_t *const *g_exp,
                                void *const *workspace, const size_t *workspace_bytes, const int *num_parts, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || num <= 0 || !descs || !e3 || !e3_exp || !b1_c || !gq || !g_exp || !workspace || !workspace_bytes || !num_parts)
        return EOQ_ERR_BAD_ARG;
    if (h->hook.fn) return EOQ_ERR_UNSUPPORTED;  // replicas exchange per layer: eoq_conv_wgrad_dev
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    for (int i = 0; i < num; ++i) {
        Geometry g;
        int st = check_desc(&descs[i], &g);
        if (st != EOQ_OK) return st;
        if (!e3[i] || !e3_exp[i] || !gq[i] || !g_exp[i] || num_parts[i] < 1) return EOQ_ERR_BAD_ARG;
        if (!aligned16(e3[i]) || !aligned16(gq[i])) return EOQ_ERR_ALIGNMENT;
        if ((st = check_workspace(&descs[i], EOQ_PASS_WGRAD, workspace[i], workspace_bytes[i])) != EOQ_OK) return st;
        const BorderClasses bc = border_classes(descs[i], g);
        if (b1_c[i] && bc.nrc * bc.ncc > kMaxBorderClasses) return EOQ_ERR_UNSUPPORTED;
    }
    for (int base = 0; base < num; base += kFinishChunk) {
        FinishItem items[kFinishChunk];
        const int count = num - base < kFinishChunk ? num - base : kFinishChunk;
        for (int k = 0; k < count; ++k) {
            const eoq_conv_desc_t &d = descs[base + k];
            Geometry g;
            check_desc(&d, &g);
            items[k] = finish_item(d, g, wgrad_space(d, g, workspace[base + k]), e3[base + k], e3_exp[base + k], 0, b1_c[base + k],
                                   gq[base + k], g_exp[base + k], num_parts[base + k]);
            items[k].tap_clear = 1;
        }
        if (count == 1 && !h->profiling && finish_is_small(items[0], h->hook)) {
            count_launches(h, 1);
            const int st = record(h, launch_finish_small(items[0], &h->dev->status, h->sm_count, false, s));
            if (st != EOQ_OK) return st;
            continue;
        }
        FinishBatch b;
        plan_finish(b, items, count, h->sm_count, h->gemm_ctas >= h->sm_count, h->hook);
        int st = b.tap_first[count] > 0 ? finish_taps(h, b, kTapsBehind, s) : EOQ_OK;
        if (st == EOQ_OK) st = finish_sums(h, b, s);
        if (st != EOQ_OK) return st;
    }
    return EOQ_OK;
}

// ================================================================================= tensor-pipe probe

extern "C" int eoq_probe_mma_i8(eoq_handle_t handle, int n_cols, int iters, int launches, double *tops,
                                double *cycles_per_mma, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !tops || n_cols < 16 || n_cols > 256 || (n_cols % 16) || iters < 1 || iters > (1 << 20) || launches < 1 ||
        launches > 100000)
        return EOQ_ERR_BAD_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaEvent_t a = nullptr, b = nullptr;
    cudaError_t e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    unsigned long long *cyc = &h->dev->probe_cycles;
    if (e == cudaSuccess) e = launch_probe_mma_i8(n_cols, iters, h->sm_count, h->dev, cyc, s);  // warm-up
    if (e == cudaSuccess) e = cudaMemsetAsync(cyc, 0, sizeof(unsigned long long), s);
    if (e == cudaSuccess) e = cudaEventRecord(a, s);
    for (int i = 0; i < launches && e == cudaSuccess; ++i) e = launch_probe_mma_i8(n_cols, iters, h->sm_count, h->dev, cyc, s);
    if (e == cudaSuccess) e = cudaEventRecord(b, s);
    if (e == cudaSuccess) e = cudaEventSynchronize(b);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
    unsigned long long cycles = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&cycles, cyc, sizeof(cycles), cudaMemcpyDeviceToHost);
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    if (e != cudaSuccess) return record(h, e);
    count_launches(h, launches + 1);
    const double ops = 2.0 * kTileM * n_cols * 32.0 * 4.0 * iters * (double)h->sm_count * launches;
    *tops = ms > 0.f ? ops / (ms * 1e-3) / 1e12 : 0.0;
    if (cycles_per_mma) *cycles_per_mma = (double)cycles / (4.0 * iters);
    return EOQ_OK;
}

// ================================================================================= plan report

extern "C" int eoq_describe_plan(eoq_handle_t handle, const eoq_conv_desc_t *desc, int pass, char *buf, size_t buf_bytes)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    Geometry g;
    if (!h || !buf || buf_bytes == 0) return EOQ_ERR_BAD_ARG;
    int st = check_desc(desc, &g);
    if (st != EOQ_OK) return st;
    const eoq_conv_desc_t &d = *desc;
    IgemmParams p;
    memset(&p, 0, sizeof(p));
    PatchPlan pl;
    memset(&pl, 0, sizeof(pl));
    buf[0] = 0;
    if (pass == EOQ_PASS_FWD) {
        if (d.stride == 1 && d.kh == d.kw && d.x_wmargin == 0 &&
            plan_stride1(p, pl, d.n, d.c_in, g.ho, g.wo, d.kh, d.pad, d.c_out, h->sm_count, h->gemm_ctas)) {
            snprintf(buf, buf_bytes, "kernel=igemm_patch tile_n=%d accumulators=%d m_tiles=%d n_tiles=%d weights=%s", p.tile_n,
                     p.tile_n <= 128 ? 2 : 1, p.num_m_tiles, p.num_n_tiles, pl.b_resident ? "resident" : "streamed");
            return EOQ_OK;
        }
        p.M = d.n * g.ho * g.wo;
        p.N = d.c_out;
        const bool rw = use_row_window(d, g.wo);
        RowsPlan rp;
        if (rw && plan_rows(p, rp, d, g, h->gemm_ctas)) {
            snprintf(buf, buf_bytes, "kernel=igemm_input_rows tile_n=%d rows_per_patch=%d patches=%d pixels=%d", p.tile_n, rp.r_rows, p.num_m_tiles,
                     rp.tile_px);
            return EOQ_OK;
        }
        plan_igemm(p, rw ? 8 * d.c_in : d.c_in, rw ? d.kh : g.taps, h->sm_count);
        if (!rw) plan_few_tiles(p, h->gemm_ctas);
        snprintf(buf, buf_bytes, "kernel=igemm%s tile_n=%d m_tiles=%d n_tiles=%d kc=%d stages=%d split=%d", rw ? "_filter_rows" : "",
                 p.tile_n, p.num_m_tiles, p.num_n_tiles, p.kc, p.num_stages, p.split);
        return EOQ_OK;
    }
    if (pass == EOQ_PASS_DGRAD) {
        p.epilogue = kEpiDgrad;
        p.b_mn = 1;
        if (d.stride == 1 && d.kh == d.kw && d.kh - 1 - d.pad >= 0 &&
            plan_stride1(p, pl, d.n, d.c_out, d.h, d.w, d.kh, d.kh - 1 - d.pad, d.c_in, h->sm_count, h->gemm_ctas)) {
            snprintf(buf, buf_bytes, "kernel=igemm_patch tile_n=%d accumulators=%d m_tiles=%d n_tiles=%d weights=%s%s", p.tile_n,
                     p.tile_n <= 128 ? 2 : 1, p.num_m_tiles, p.num_n_tiles, pl.b_resident ? "resident" : "streamed",
                     igemm_patch_lean(p, pl) ? " registers=72" : "");
            return EOQ_OK;
        }
        // as the call without a dump of the sums: a number per class, the classes of a launch apart by commas, launches by slashes
        struct List {
            char text[256];
            size_t used;
            void add(const char *separator, int v)
            {
                const int n = snprintf(text + used, sizeof(text) - used, "%s%d", separator, v);
                if (n > 0) used = used + n < sizeof(text) ? used + n : sizeof(text) - 1;
            }
        } tile_n = {}, m_tiles = {}, n_tiles = {}, ctas = {}, split = {};
        int classes = 0, launches = 0, kc = 0;
        st = each_class_launch(d, compact_sums(d), h->sm_count, h->gemm_ctas, [&](const IgemmClasses &cl, const ClassCorners &) -> int {
            const char *const next_launch = launches++ ? "/" : "";
            for (int k = 0; k < cl.num; ++k) {
                const char *const separator = k ? "," : next_launch;
                tile_n.add(separator, cl.p[k].tile_n);
                m_tiles.add(separator, cl.p[k].num_m_tiles);
                n_tiles.add(separator, cl.p[k].num_n_tiles);
                ctas.add(separator, cl.first[k + 1] - cl.first[k]);
                kc = cl.p[k].kc;
            }
            split.add(next_launch, cl.p[0].split);
            classes += cl.num;
            return EOQ_OK;
        });
        if (st != EOQ_OK) return st;
        snprintf(buf, buf_bytes, "kernel=igemm classes=%d tile_n=%s m_tiles=%s n_tiles=%s kc=%d split=%s launches=%d ctas=%s", classes, tile_n.text,
                 m_tiles.text, n_tiles.text, kc, split.text, launches, ctas.text);
        return EOQ_OK;
    }
    if (pass == EOQ_PASS_WGRAD) {
        WgradPatchPlan wp;
        if (plan_wgrad_patch(wp, d, g.ho, g.wo, h->gemm_ctas < kWgradTargetCtas ? h->gemm_ctas : kWgradTargetCtas))
            snprintf(buf, buf_bytes, "kernel=wgrad_patch groups=%d splits=%d tile_n=%d kc=%d", wp.num_groups, wp.num_splits, wp.tile_n,
                     wp.kc);
        else
            snprintf(buf, buf_bytes, "kernel=wgrad%s", use_row_window(d, g.wo) ? "_filter_rows" : "");
        return EOQ_OK;
    }
    return EOQ_ERR_BAD_ARG;
}

// ================================================================================= elementwise entry points

extern "C" int eoq_quantize(eoq_handle_t handle, int mode, const void *src, int src_is_float, const int32_t *src_exp,
                            size_t n, void *dst, int32_t *dst_exp, void *workspace, size_t workspace_bytes,
                            void *stream)
{
    (void)workspace;
    (void)workspace_bytes;
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !src || !dst || n == 0) return EOQ_ERR_BAD_ARG;
    if (mode != EOQ_Q && mode != EOQ_CQ && mode != EOQ_SQ) return EOQ_ERR_BAD_ARG;
    if (mode == EOQ_SQ && !dst_exp) return EOQ_ERR_BAD_ARG;
    if (!aligned16(src) || !aligned16(dst)) return EOQ_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, mode == EOQ_SQ && !(src_is_float && quantize_is_small(mode, n, h->hook)) ? 2 : 1);
    ProfScope prof(h, EOQ_PROF_OTHER, s);
    if (src_is_float)
        return record(h, launch_quantize_f32(mode, reinterpret_cast<const float *>(src), n, dst, dst_exp, h->tile_shift, h->dev,
                                             h->sm_count, s, h->hook));
    if (mode != EOQ_SQ || !src_exp) return EOQ_ERR_UNSUPPORTED;
    return record(h, launch_sq_i32(reinterpret_cast<const int32_t *>(src), src_exp, 0, n, reinterpret_cast<int8_t *>(dst),
                                   dst_exp, nullptr, false, h->dev, h->sm_count, s, h->hook));
}

static int err_prescale_impl(eoq_handle_t handle, const int8_t *e0, const int32_t *e0_exp, const uint8_t *relu_mask,
                             const int16_t *x2, size_t n_el, int32_t gamma_c, const int32_t *gamma_dev, int8_t *e3,
                             int32_t *e3_exp, int64_t *sum_e1, int64_t *sum_e1x2, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !e0 || !e0_exp || !e3 || !e3_exp || n_el == 0 || (n_el % 16)) return EOQ_ERR_BAD_ARG;
    if (!aligned16(e0) || !aligned16(e3) || !aligned16(x2) || (reinterpret_cast<uintptr_t>(relu_mask) & 1)) return EOQ_ERR_ALIGNMENT;
    if (gamma_c < -32768 || gamma_c > 32767) return EOQ_ERR_RANGE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    ProfScope prof(h, EOQ_PROF_ERR_HEAD, s);
    int kernels = 0;
    const bool force_timeout = h->force_timeout;
    h->force_timeout = false;
    const cudaError_t e = launch_err_prescale(e0, e0_exp, relu_mask, x2, n_el, gamma_c, gamma_dev, e3, e3_exp,
                                              reinterpret_cast<long long *>(sum_e1), reinterpret_cast<long long *>(sum_e1x2),
                                              h->dev, h->sm_count, s, &kernels, force_timeout, h->hook);
    count_launches(h, kernels);
    return record(h, e);
}

extern "C" int eoq_err_prescale(eoq_handle_t handle, const int8_t *e0, const int32_t *e0_exp, const uint8_t *relu_mask,
                                const int16_t *x2, size_t n_el, int32_t gamma_c, int8_t *e3, int32_t *e3_exp,
                                int64_t *sum_e1, int64_t *sum_e1x2, void *stream)
{
    return err_prescale_impl(handle, e0, e0_exp, relu_mask, x2, n_el, gamma_c, nullptr, e3, e3_exp, sum_e1, sum_e1x2, stream);
}

extern "C" int eoq_err_prescale_dev(eoq_handle_t handle, const int8_t *e0, const int32_t *e0_exp, const uint8_t *relu_mask,
                                    const int16_t *x2, size_t n_el, const int32_t *gamma_c, int8_t *e3, int32_t *e3_exp,
                                    int64_t *sum_e1, int64_t *sum_e1x2, void *stream)
{
    if (!gamma_c) return EOQ_ERR_BAD_ARG;
    return err_prescale_impl(handle, e0, e0_exp, relu_mask, x2, n_el, 128, gamma_c, e3, e3_exp, sum_e1, sum_e1x2, stream);
}

extern "C" int eoq_debug_force_wait_timeout(eoq_handle_t handle)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h) return EOQ_ERR_BAD_ARG;
    h->force_timeout = true;
    return EOQ_OK;
}

static int update_impl(eoq_handle_t handle, int num, int8_t *const *w, const int8_t *const *g,
                       const int32_t *const *g_exp, const size_t *n, int32_t lr_mant, int32_t lr_exp, int round_mode,
                       uint64_t seed, uint64_t step, uint64_t *step_dev, void *stream, int first = 0, bool last = true)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || num <= 0 || !w || !g || !g_exp || !n) return EOQ_ERR_BAD_ARG;
    if (first < 0) return EOQ_ERR_BAD_ARG;
    if (num > 256 || first > 256 - num) return EOQ_ERR_UNSUPPORTED;
    if (lr_mant < 1 || lr_mant > 255 || lr_exp < -64 || lr_exp > 64) return EOQ_ERR_RANGE;
    if (round_mode != EOQ_ROUND_RNE && round_mode != EOQ_ROUND_STOCHASTIC) return EOQ_ERR_BAD_ARG;
    UpdateTensor t[256];
    for (int i = 0; i < num; ++i) {
        if (!w[i] || !g[i] || !g_exp[i] || n[i] == 0) return EOQ_ERR_BAD_ARG;
        t[i].w = w[i];
        t[i].g = g[i];
        t[i].g_exp = g_exp[i];
        t[i].n = n[i];
        t[i].master = nullptr;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, update_launches(t, num, false));
    ProfScope prof(h, EOQ_PROF_UPDATE, s);
    return record(h, launch_update(t, num, lr_mant, lr_exp, round_mode == EOQ_ROUND_STOCHASTIC, seed, step,
                                   reinterpret_cast<unsigned long long *>(step_dev), h->dev, s, first, last));
}

extern "C" int eoq_update(eoq_handle_t handle, int num, int8_t *const *w, const int8_t *const *g,
                          const int32_t *const *g_exp, const size_t *n, int32_t lr_mant, int32_t lr_exp,
                          int round_mode, uint64_t seed, uint64_t step, void *stream)
{
    return update_impl(handle, num, w, g, g_exp, n, lr_mant, lr_exp, round_mode, seed, step, nullptr, stream);
}

extern "C" int eoq_update_dev(eoq_handle_t handle, int num, int8_t *const *w, const int8_t *const *g,
                              const int32_t *const *g_exp, const size_t *n, int32_t lr_mant, int32_t lr_exp,
                              int round_mode, uint64_t seed, uint64_t *step, void *stream)
{
    if (!step || (reinterpret_cast<uintptr_t>(step) & 7)) return EOQ_ERR_BAD_ARG;
    return update_impl(handle, num, w, g, g_exp, n, lr_mant, lr_exp, round_mode, seed, 0, step, stream);
}

extern "C" int eoq_update_part(eoq_handle_t handle, int first, int last, int num, int8_t *const *w, const int8_t *const *g,
                               const int32_t *const *g_exp, const size_t *n, int32_t lr_mant, int32_t lr_exp, int round_mode,
                               uint64_t seed, uint64_t *step, void *stream)
{
    if (!step || (reinterpret_cast<uintptr_t>(step) & 7)) return EOQ_ERR_BAD_ARG;
    return update_impl(handle, num, w, g, g_exp, n, lr_mant, lr_exp, round_mode, seed, 0, step, stream, first, last != 0);
}

extern "C" int eoq_update_wide(eoq_handle_t handle, int num, int32_t *const *master, int8_t *const *w, const int8_t *const *g,
                               const int32_t *const *g_exp, const size_t *n, int32_t lr_mant, int32_t lr_exp, int k_u, int k_m,
                               int round_mode, uint64_t seed, uint64_t step, uint64_t *step_dev, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || num <= 0 || !master || !w || !g || !g_exp || !n) return EOQ_ERR_BAD_ARG;
    if (num > 256) return EOQ_ERR_UNSUPPORTED;
    if (lr_mant < 1 || lr_mant > 255 || lr_exp < -64 || lr_exp > 64) return EOQ_ERR_RANGE;
    if (k_u < 2 || k_u > 24 || k_m < 8 || k_m > 24) return EOQ_ERR_UNSUPPORTED;
    if (round_mode != EOQ_ROUND_RNE && round_mode != EOQ_ROUND_STOCHASTIC) return EOQ_ERR_BAD_ARG;
    if (step_dev && (reinterpret_cast<uintptr_t>(step_dev) & 7)) return EOQ_ERR_BAD_ARG;
    UpdateTensor t[256];
    for (int i = 0; i < num; ++i) {
        if (!master[i] || !w[i] || !g[i] || !g_exp[i] || n[i] == 0) return EOQ_ERR_BAD_ARG;
        t[i].w = w[i];
        t[i].g = g[i];
        t[i].g_exp = g_exp[i];
        t[i].n = n[i];
        t[i].master = master[i];
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, update_launches(t, num, true));
    ProfScope prof(h, EOQ_PROF_UPDATE, s);
    return record(h, launch_update_wide(t, num, lr_mant, lr_exp, k_u, k_m, round_mode == EOQ_ROUND_STOCHASTIC, seed, step,
                                        reinterpret_cast<unsigned long long *>(step_dev), h->dev, s));
}

extern "C" int eoq_layout_convert(eoq_handle_t handle, const int8_t *src, int8_t *dst, int n, int c, int hh, int ww,
                                  int to_nhwc, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !src || !dst || n <= 0 || c <= 0 || hh <= 0 || ww <= 0 || n > 65535) return EOQ_ERR_BAD_ARG;
    count_launches(h, 1);
    return record(h, launch_layout_convert(src, dst, n, c, hh, ww, to_nhwc, reinterpret_cast<cudaStream_t>(stream)));
}

extern "C" int eoq_quantize_image(eoq_handle_t handle, const float *src, int n, int hh, int ww, int c_src, int c_dst,
                                  int wmargin, int8_t *dst, int32_t *dst_exp, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !src || !dst || !dst_exp || n <= 0 || hh <= 0 || ww <= 0 || c_src <= 0 || c_dst < c_src || wmargin < 0 ||
        wmargin > 64)
        return EOQ_ERR_BAD_ARG;
    if ((c_dst % 16 && c_dst != 8) || c_dst > 64 || !aligned16(src) || !aligned16(dst)) return EOQ_ERR_ALIGNMENT;
    count_launches(h, 2);
    ProfScope prof(h, EOQ_PROF_INPUT_Q, reinterpret_cast<cudaStream_t>(stream));
    return record(h, launch_quantize_image(src, n, hh, ww, c_src, c_dst, wmargin, dst, dst_exp, h->dev,
                                           reinterpret_cast<cudaStream_t>(stream), h->hook));
}

// ================================================================================= network glue

extern "C" int eoq_aux_maxpool_fwd(eoq_handle_t handle, const int8_t *x, int n, int hh, int ww, int c, int k, int stride, int pad,
                                   int8_t *y, uint8_t *arg, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !x || !y || !arg || n <= 0 || hh <= 0 || ww <= 0 || c <= 0 || k <= 0 || k > 15 || stride <= 0 || pad < 0 || pad >= k)
        return EOQ_ERR_BAD_ARG;
    if (c % 16 || !aligned16(x) || !aligned16(y) || !aligned16(arg)) return EOQ_ERR_ALIGNMENT;
    if ((size_t)n * hh * ww * (c / 16) > 0xffffffffull) return EOQ_ERR_UNSUPPORTED;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 1);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_maxpool_fwd(x, n, hh, ww, c, k, stride, pad, y, arg, s));
}

extern "C" int eoq_aux_maxpool_bwd(eoq_handle_t handle, const int8_t *e, const int32_t *e_exp, const uint8_t *arg, int n, int hh,
                                   int ww, int c, int k, int stride, int pad, int8_t *e_in, int32_t *e_in_exp, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !e || !e_exp || !arg || !e_in || !e_in_exp || n <= 0 || hh <= 0 || ww <= 0 || c <= 0 || k <= 0 || k > 15 ||
        stride <= 0 || pad < 0 || pad >= k)
        return EOQ_ERR_BAD_ARG;
    if (c % 16 || !aligned16(e) || !aligned16(arg) || !aligned16(e_in)) return EOQ_ERR_ALIGNMENT;
    if ((size_t)n * hh * ww * (c / 16) > 0x7fffffffull) return EOQ_ERR_UNSUPPORTED;   // 32-bit item index in the kernel
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 2);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_maxpool_bwd(e, e_exp, arg, n, hh, ww, c, k, stride, pad, e_in, e_in_exp, nullptr, nullptr, nullptr, nullptr,
                                        nullptr, h->dev, h->sm_count, s, h->hook));
}

extern "C" int eoq_aux_maxpool_bwd_head(eoq_handle_t handle, const int8_t *e, const int32_t *e_exp, const uint8_t *arg, int n, int hh,
                                        int ww, int c, int k, int stride, int pad, int8_t *e_in, int32_t *e_in_exp,
                                        const uint8_t *relu_mask, const int32_t *gamma, int8_t *e3, int32_t *e3_exp, int64_t *sum_e1,
                                        void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !e || !e_exp || !arg || !relu_mask || !gamma || !e3 || !e3_exp || n <= 0 || hh <= 0 || ww <= 0 || c <= 0 || k <= 0 ||
        k > 15 || stride <= 0 || pad < 0 || pad >= k)
        return EOQ_ERR_BAD_ARG;
    if (c % 16 || !aligned16(e) || !aligned16(arg) || !aligned16(e3) || (e_in && !aligned16(e_in)) ||
        (reinterpret_cast<uintptr_t>(relu_mask) & 1))
        return EOQ_ERR_ALIGNMENT;
    if ((size_t)n * hh * ww * (c / 16) > 0x7fffffffull) return EOQ_ERR_UNSUPPORTED;   // 32-bit item index in the kernel
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 2);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_maxpool_bwd(e, e_exp, arg, n, hh, ww, c, k, stride, pad, e_in, e_in_exp, relu_mask, gamma, e3, e3_exp,
                                        reinterpret_cast<long long *>(sum_e1), h->dev, h->sm_count, s, h->hook));
}

extern "C" int eoq_bn_workspace_size(int c, size_t *bytes)
{
    if (!bytes || c <= 0) return EOQ_ERR_BAD_ARG;
    *bytes = (bn_workspace_bytes(c) + 255) & ~(size_t)255;
    return EOQ_OK;
}

static int bn_check(Handle *h, size_t pixels, int c, const void *ws, size_t ws_bytes)
{
    if (!h || !ws || pixels == 0 || c <= 0) return EOQ_ERR_BAD_ARG;
    if (c % 16 || !aligned16(ws)) return EOQ_ERR_ALIGNMENT;
    if (c > 1024 || pixels > 0x7fffffffull) return EOQ_ERR_UNSUPPORTED;
    if (ws_bytes < bn_workspace_bytes(c)) return EOQ_ERR_WORKSPACE;
    return EOQ_OK;
}

extern "C" int eoq_bn_fwd(eoq_handle_t handle, const int32_t *acc, int acc_exp, size_t pixels, int c, const float *gamma,
                          const float *beta, float eps, int8_t *x5, uint8_t *relu_mask, void *workspace, size_t workspace_bytes,
                          void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!acc || !gamma || !beta || !x5 || !relu_mask || !(eps >= 0.0f) || acc_exp < -60 || acc_exp > 60) return EOQ_ERR_BAD_ARG;
    const int chk = bn_check(h, pixels, c, workspace, workspace_bytes);
    if (chk != EOQ_OK) return chk;
    if (!aligned16(acc) || !aligned16(x5) || (reinterpret_cast<uintptr_t>(relu_mask) & 1)) return EOQ_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 3);
    ProfScope prof(h, EOQ_PROF_OTHER, s);
    return record(h, launch_bn_fwd(acc, acc_exp, pixels, c, gamma, beta, eps, x5, relu_mask, reinterpret_cast<BnChannel *>(workspace),
                                   h->sm_count, s));
}

extern "C" int eoq_bn_bwd(eoq_handle_t handle, const int8_t *e, const int32_t *e_exp, const uint8_t *relu_mask, const int32_t *acc,
                          int acc_exp, size_t pixels, int c, const float *gamma, void *workspace, size_t workspace_bytes, float *da,
                          float *dgamma, float *dbeta, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!e || !e_exp || !relu_mask || !acc || !gamma || !da || !dgamma || !dbeta || acc_exp < -60 || acc_exp > 60)
        return EOQ_ERR_BAD_ARG;
    const int chk = bn_check(h, pixels, c, workspace, workspace_bytes);
    if (chk != EOQ_OK) return chk;
    if (!aligned16(acc) || !aligned16(e) || !aligned16(da) || (reinterpret_cast<uintptr_t>(relu_mask) & 1)) return EOQ_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 3);
    ProfScope prof(h, EOQ_PROF_OTHER, s);
    return record(h, launch_bn_bwd(e, e_exp, relu_mask, acc, acc_exp, pixels, c, gamma, reinterpret_cast<BnChannel *>(workspace), da,
                                   dgamma, dbeta, h->sm_count, s));
}

extern "C" int eoq_aux_avgpool_sum(eoq_handle_t handle, const int8_t *x, int n, int hw, int c, int32_t *sums, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !x || !sums || n <= 0 || hw <= 0 || c <= 0 || hw > (1 << 23)) return EOQ_ERR_BAD_ARG;
    if (c % 16 || !aligned16(x)) return EOQ_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 1);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_avgpool_sum(x, n, hw, c, sums, s));
}

extern "C" int eoq_aux_join(eoq_handle_t handle, const int8_t *a, const int32_t *a_exp, const int8_t *b, const int32_t *b_exp,
                            const uint8_t *mask_b, size_t n_el, int8_t *out, int32_t *out_exp, int64_t *sum_out, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !a || !a_exp || !b || !b_exp || !out || !out_exp || n_el == 0 || (n_el % 16)) return EOQ_ERR_BAD_ARG;
    if (!aligned16(a) || !aligned16(b) || !aligned16(out) || (reinterpret_cast<uintptr_t>(mask_b) & 1)) return EOQ_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 2);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_join(a, a_exp, b, b_exp, mask_b, n_el, out, out_exp, reinterpret_cast<long long *>(sum_out), nullptr, nullptr,
                                 nullptr, nullptr, nullptr, nullptr, nullptr, h->dev, h->sm_count, s, h->hook));
}

extern "C" int eoq_aux_join_head(eoq_handle_t handle, const int8_t *a, const int32_t *a_exp, const int8_t *b, const int32_t *b_exp,
                                 const uint8_t *mask_b, size_t n_el, int8_t *out, int32_t *out_exp, int64_t *sum_out,
                                 const uint8_t *relu_mask, const int16_t *x2, const int32_t *gamma, int8_t *e3, int32_t *e3_exp,
                                 int64_t *sum_e1, int64_t *sum_e1x2, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !a || !a_exp || !b || !b_exp || !out || !out_exp || !relu_mask || !gamma || !e3 || !e3_exp || n_el == 0 || (n_el % 16))
        return EOQ_ERR_BAD_ARG;
    if (!aligned16(a) || !aligned16(b) || !aligned16(out) || !aligned16(e3) || (x2 && !aligned16(x2)) ||
        (reinterpret_cast<uintptr_t>(mask_b) & 1) || (reinterpret_cast<uintptr_t>(relu_mask) & 1))
        return EOQ_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 2);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_join(a, a_exp, b, b_exp, mask_b, n_el, out, out_exp, reinterpret_cast<long long *>(sum_out), relu_mask, x2, gamma,
                                 e3, e3_exp, reinterpret_cast<long long *>(sum_e1), reinterpret_cast<long long *>(sum_e1x2), h->dev,
                                 h->sm_count, s, h->hook));
}

extern "C" int eoq_aux_head_workspace_size(int n, int c, int classes, size_t *bytes)
{
    if (!bytes || n <= 0 || c <= 0 || classes <= 0) return EOQ_ERR_BAD_ARG;
    *bytes = round256((size_t)n * c * sizeof(float)) * 2 + round256((size_t)n * classes * sizeof(float)) + round256((size_t)n * sizeof(double));
    return EOQ_OK;
}

extern "C" int eoq_aux_head(eoq_handle_t handle, const int32_t *sums, int n, int c, int hw, int classes, float *W, float *bias,
                            const int32_t *labels, float lr, float *loss, float *dpooled, float *logits, void *workspace,
                            size_t workspace_bytes, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !sums || !W || !bias || !labels || !dpooled || !logits || n <= 0 || c <= 0 || hw <= 0 || classes <= 0)
        return EOQ_ERR_BAD_ARG;
    if (c > 1536) return EOQ_ERR_UNSUPPORTED;
    size_t need = 0;
    eoq_aux_head_workspace_size(n, c, classes, &need);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < need) return EOQ_ERR_WORKSPACE;
    char *ws = static_cast<char *>(workspace);
    float *pooled = reinterpret_cast<float *>(ws);
    float *dl = reinterpret_cast<float *>(ws + 2 * round256((size_t)n * c * sizeof(float)));
    double *loss_n = reinterpret_cast<double *>(ws + 2 * round256((size_t)n * c * sizeof(float)) + round256((size_t)n * classes * sizeof(float)));
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, (head_folds_pooling(n) ? 3 : 4) + (lr != 0.0f ? 1 : 0));
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_head(sums, n, c, hw, classes, W, bias, labels, lr, loss, dpooled, logits, pooled, dl, loss_n, s));
}

extern "C" int eoq_aux_head_update(eoq_handle_t handle, int n, int c, int classes, float *W, float *bias, float lr, const void *workspace,
                                   size_t workspace_bytes, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !W || !bias || n <= 0 || c <= 0 || classes <= 0) return EOQ_ERR_BAD_ARG;
    size_t need = 0;
    eoq_aux_head_workspace_size(n, c, classes, &need);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < need) return EOQ_ERR_WORKSPACE;
    const char *ws = static_cast<const char *>(workspace);
    const float *pooled = reinterpret_cast<const float *>(ws);
    const float *dl = reinterpret_cast<const float *>(ws + 2 * round256((size_t)n * c * sizeof(float)));
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, 1);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_head_update(dl, pooled, n, c, classes, lr, W, bias, s));
}

extern "C" int eoq_aux_head_error(eoq_handle_t handle, const float *dpooled, int n, int c, int hw, int8_t *e, int32_t *e_exp,
                                  void *workspace, size_t workspace_bytes, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || !dpooled || !e || !e_exp || n <= 0 || c <= 0 || hw <= 0) return EOQ_ERR_BAD_ARG;
    if (c % 16 || !aligned16(e)) return EOQ_ERR_ALIGNMENT;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < (size_t)n * c * sizeof(float)) return EOQ_ERR_WORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    count_launches(h, head_error_is_single(n, c, h->hook) ? 1 : 2);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    return record(h, launch_head_error(dpooled, n, c, hw, e, e_exp, h->dev, h->sm_count, s, h->hook));
}

extern "C" int eoq_aux_scalar_update(eoq_handle_t handle, int num, int32_t *const *theta, int32_t *const *mirror,
                                     const int64_t *const *total, const int32_t *const *total_exp, const int *exp_bias,
                                     const int *tensor_id, int32_t *const *grad_out, int32_t lr_mant, int32_t lr_exp,
                                     int round_mode, uint64_t seed, const uint64_t *step, void *stream)
{
    Handle *h = reinterpret_cast<Handle *>(handle);
    if (!h || num <= 0 || !theta || !total || !total_exp || !exp_bias || !tensor_id) return EOQ_ERR_BAD_ARG;
    if (lr_mant < 1 || lr_mant > 255 || lr_exp < -64 || lr_exp > 64) return EOQ_ERR_RANGE;
    if (round_mode != EOQ_ROUND_RNE && round_mode != EOQ_ROUND_STOCHASTIC) return EOQ_ERR_BAD_ARG;
    for (int i = 0; i < num; ++i)
        if (!theta[i] || !total[i] || !total_exp[i]) return EOQ_ERR_BAD_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    ProfScope prof(h, EOQ_PROF_GLUE, s);
    for (int base = 0; base < num; base += kScalarChunk) {
        ScalarBatch b;
        memset(&b, 0, sizeof(b));
        b.num = num - base < kScalarChunk ? num - base : kScalarChunk;
        for (int k = 0; k < b.num; ++k) {
            ScalarItem &it = b.item[k];
            it.theta = theta[base + k];
            it.mirror = mirror ? mirror[base + k] : nullptr;
            it.total = reinterpret_cast<const long long *>(total[base + k]);
            it.exp = total_exp[base + k];
            it.exp_bias = exp_bias[base + k];
            it.tensor_id = tensor_id[base + k];
            it.grad_out = grad_out ? grad_out[base + k] : nullptr;
        }
        cudaError_t e = launch_scalar_update(b, lr_mant, lr_exp, round_mode == EOQ_ROUND_STOCHASTIC, seed,
                                             reinterpret_cast<const unsigned long long *>(step), 0, s);
        if (e != cudaSuccess) return record(h, e);
        count_launches(h, 1);
    }
    return EOQ_OK;
}
