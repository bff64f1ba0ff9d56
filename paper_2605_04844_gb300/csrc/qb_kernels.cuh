// qb_kernels.cuh -- kernel argument blocks and launchers of libquadbox.
#pragma once

#include "qb_internal.cuh"

namespace qb {

// Cameras processed together: records of camera c live at [c * n, (c+1) * n).
constexpr int kMaxGroupCams = 16;

struct CamSet {
    int n_cams;
    CamDev cam[kMaxGroupCams];
};

struct PreArgs {
    int n;  // Gaussians (records per camera)
    const float *means, *scales, *quats, *opac, *sh;
    bool raw;
    bool sh_vec4;    // sh rows may be read as float4 (16-byte aligned)
    bool quat_vec4;  // quats may be read as float4 (16-byte aligned)
    CamSet cams;
    int mode;
    bool clamp3s;
    float2 *xy;      // [n_cams * n] ...
    float2 *shape;   // (r, -e/2) of an elongated Gaussian's exact power form, else (0, 0)
    float4 *conic_o, *rgbd, *box;
    float *r3;
    int *meta;
    uint32_t *counts;
    uint2 *cc;         // [records] (tiles, cells)
    uint4 *rects;      // [records][2] packed sub-box rectangles (pack_rects), written where there are tiles
    uint32_t *depth_keys, *depth_vals;  // [records] depth-sort keys and record indices, or null
};

// Image geometry of one camera in a set of cameras rendered together.  Tile
// ids are global over the set (camera c owns [tile_base, tile_base + tiles));
// per-pixel arrays and the planar [3][H][W] image of camera c start at pixel
// pix_base (the image at float offset 3 * pix_base).  The render reads the
// camera's sorted values at vals + vals_base (its ranges are relative to it)
// and a value v names the record rec_base + v.
struct CamTile {
    int W, H, tiles_x, tiles_y;
    uint32_t tile_base;
    uint32_t rec_base;
    uint64_t pix_base;
    uint64_t vals_base;
};

// The camera owning global tile t in a device table of n cameras ordered by
// tile_base (binary search).
__device__ __forceinline__ int camera_in_table(const CamTile *table, int n, uint32_t t) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (table[mid].tile_base <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

struct TileSet {
    int n_cams;
    uint32_t total_tiles;
    CamTile cam[kMaxGroupCams];
};

// The full-key emit (a single frame, index order).
struct EmitArgs {
    int n;
    const float4 *rgbd;
    const uint32_t *counts, *offsets;
    const uint32_t *chunk_first;  // Gaussian holding output position c kEmitStride
    const uint4 *rects;
    uint32_t *vals;
    const uint64_t *n_pairs;
    uint64_t n_pairs_host;  // P when the host knows it, else UINT64_MAX
    uint64_t capacity;
    int mode;
    uint32_t *err;
    const uint32_t *failed;  // the scan's failure word: nothing is emitted when it is set
    uint32_t tiles_x;
};

// Geometry of the cells of one image, and the widths of the passes that sort
// their ids.
struct CellGeo {
    int tiles_x, tiles_y, cells_x, cells_y, ncells, ntiles;
    int cell_bits, digit_bits;  // digit_bits: of the widest pass (sort scratch layout)
    PassGeo passes;
};

// Device arrays of the cell binning (qb_cells.cu).
struct CellArrays {
    uint32_t *count;       // [ncells + 1] entries per cell and without a tile, then two finished-block counters
    uint32_t *start;       // [ncells + 2] first sorted entry of each cell (last: of those without a tile)
    uint32_t *row_start;   // [ncells + 1] first row of each cell
    uint32_t *row_cell;    // [rows]
    uint32_t *row_counts;  // [rows][32] entries per tile; after the prefix, those of the cell's earlier rows
    uint32_t *tile_total;  // [ntiles rounded up to 8]
    // entries (cell id; Gaussian | tile bits << 32), two buffers; keys_b is read
    // and written by sorts of two passes or more only
    uint32_t *keys_a, *keys_b;
    uint64_t *vals_a, *vals_b;
};
constexpr uint32_t kCellRow = 128;  // sorted entries per row
inline size_t cell_zero_words(int ncells) { return (size_t)ncells + 3; }
inline size_t cell_rows_max(uint64_t pair_capacity, int ncells) { return (size_t)(pair_capacity / kCellRow) + ncells; }

struct CellBin {
    int n;
    const uint32_t *perm;   // record of each emission position
    const uint32_t *coff;   // first entry of each emission position
    const uint32_t *chunk_first;
    const uint4 *rects;     // by record
    const uint64_t *n_pairs, *n_cells;  // (n_cells 0: too many pairs, or the scan failed)
    uint64_t n_cells_max;   // bound on *n_cells (the capacity, or P where the host knows it)
    uint64_t capacity;
    bool naive;             // emit by nested loops (QB_BIN_QUADBOX_NAIVE)
    uint32_t *err;
    void *sort_scratch;
    CellGeo geo;
    CellArrays arr;
    uint2 *ranges;          // [ntiles]
    uint32_t *vals;         // [P] sorted values
};

// Tiles filed by work into kOrderBuckets buckets, heaviest first: bucket
// j = kOrderBuckets - 1 - min(work / kOrderWidth, kOrderBuckets - 1) holds
// cnt[j] tiles at list[j * ntiles ...]; position p of the order is slot
// p - (cnt[0] + ... + cnt[j - 1]) of the bucket j that contains it.  The
// counts are zeroed before the tiles are filed, each tile exactly once.
constexpr int kOrderBuckets = 64;
constexpr uint32_t kOrderWidth = 16;  // entries of work per bucket
struct TileOrder {
    uint32_t *cnt;   // [kOrderBuckets], or null: no order
    uint32_t *list;  // [kOrderBuckets][ntiles]
};

__device__ __forceinline__ void order_file(const TileOrder &o, uint32_t ntiles, uint32_t tile, uint32_t work) {
    const uint32_t j = (uint32_t)kOrderBuckets - 1u - min(work / kOrderWidth, (uint32_t)kOrderBuckets - 1u);
    const uint32_t slot = atomicAdd(o.cnt + j, 1u);
    if (slot < ntiles) o.list[(size_t)j * ntiles + slot] = tile;
}

// The tile at position pos of the order, found by one warp (every warp of a
// block finds the same tile, with no shared memory or barrier): lane l reads
// buckets l and l + 32.  Position pos itself when no bucket holds it (never,
// when every tile was filed once).
static_assert(kOrderBuckets == 64, "order_pick reads two buckets per lane");
__device__ __forceinline__ uint32_t order_pick(const TileOrder &o, uint32_t ntiles, uint32_t pos) {
    const int lane = threadIdx.x & 31;
    const uint32_t c0 = o.cnt[lane], c1 = o.cnt[32 + lane];
    uint32_t i0 = c0, i1 = c1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t u0 = __shfl_up_sync(0xffffffffu, i0, d), u1 = __shfl_up_sync(0xffffffffu, i1, d);
        if (lane >= d) i0 += u0, i1 += u1;
    }
    i1 += __shfl_sync(0xffffffffu, i0, 31);  // inclusive prefixes of buckets lane and 32 + lane
    const uint32_t e0 = i0 - c0, e1 = i1 - c1;
    const bool h0 = pos >= e0 && pos < i0 && pos - e0 < ntiles;
    const bool h1 = pos >= e1 && pos < i1 && pos - e1 < ntiles;
    uint32_t t = pos;
    if (h0) t = o.list[(size_t)lane * ntiles + (pos - e0)];
    if (h1) t = o.list[(size_t)(32 + lane) * ntiles + (pos - e1)];
    const uint32_t m0 = __ballot_sync(0xffffffffu, h0), m1 = __ballot_sync(0xffffffffu, h1);
    const int src = m0 ? __ffs(m0) - 1 : (m1 ? __ffs(m1) - 1 : 0);
    t = __shfl_sync(0xffffffffu, t, src);
    return (m0 | m1) && t < ntiles ? t : pos;
}

struct RenderArgs {
    const uint2 *ranges;  // by global tile
    const uint32_t *vals;
    const float2 *xy;
    const float2 *shape;
    const float4 *conic_o, *rgbd;
    float bg[3];
    float *img;     // packed planar images
    float *tfinal;  // per pixel (all cameras)
    int *ncontrib;
    int *neval;
    TileSet ts;
    uint32_t *queue;     // persistent launch: tile counter (zeroed); null: one block per tile
    int tiles_per_fetch;
    int blocks_per_sm;   // persistent blocks per SM (0: occupancy limit)
    unsigned long long *counts;  // measurement only (single frame): [evaluated, power test passed] or null
    const CamTile *cam_table;    // persistent launch over ts.n_cams cameras from this device table, or null (ts.cam)
    // single frame, with order_out[0].cnt set: every tile is filed in both by
    // its largest last-contributor count (the backward's work)
    TileOrder order_out[2];
};

struct BwdArgs {
    const uint2 *ranges;
    const uint32_t *vals;
    const float2 *xy;
    const float2 *shape;
    const float4 *conic_o, *rgbd;
    float bg[3];
    const float *dL_dimg;  // packed like the images
    const float *tfinal;
    const int *ncontrib;
    double *g_screen;  // [records][9]: mu_x, mu_y, Sigma11, Sigma12, Sigma22, o, r, g, b
    TileSet ts;
    uint32_t *queue;
    int tiles_per_fetch;
    int blocks_per_sm;
    const CamTile *cam_table;  // as RenderArgs::cam_table
    TileOrder order;           // one block per tile: with cnt set, block b takes the tile at position b, else tile b
};

struct PreBwdArgs {
    int n;  // Gaussians
    const float *means, *scales, *quats, *opac, *sh;
    bool raw;
    CamSet cams;
    const int *meta;          // [n_cams * n]
    const double *g_screen;   // [n_cams * n][9]
    float *gm, *gs, *gq, *go, *gsh;
    uint32_t *list_count;     // one camera: zero before the launch; Gaussians listed
    uint32_t *list;           // one camera: [n], the Gaussians with a sum that is not zero
    bool sh_vec4, gsh_vec4;   // sh / gsh rows may be accessed as float4 (16-byte aligned)
};

cudaError_t launch_preprocess(const PreArgs &a, int deg, cudaStream_t s);
// partials: scan_partials_count(n) words of scratch (block status words and
// the block counter), 16-byte aligned, cleared by the launch; a look-back that
// waits too long raises kErrTimeout in *err.  launch_scan: the counts in index
// order (full-key path).  launch_scan_cells: (tiles, cells) in the order perm;
// *n_cells becomes 0 when the pairs exceed the capacity.  n_pairs_host, when
// not null, is a device address of mapped host memory that also gets P (n > 0).
cudaError_t launch_scan(const uint32_t *counts, int n, uint32_t *offsets, uint64_t *partials,
                        uint64_t *n_pairs, uint64_t *n_pairs_host, uint32_t *err, uint32_t *chunk_first,
                        uint32_t chunk_cap, cudaStream_t s);
cudaError_t launch_scan_cells(const uint2 *cc, const uint32_t *perm, int n, uint32_t *offsets, uint32_t *coff,
                              uint64_t *partials, uint64_t *n_pairs, uint64_t *n_pairs_host, uint64_t *n_cells,
                              uint64_t capacity, uint32_t *err, const uint32_t *order_failed, uint32_t *chunk_first,
                              uint32_t chunk_cap, cudaStream_t s);
// The word of a scan's scratch that is not zero after a look-back ran out (the
// offsets are then of no use), or null for n = 0.
const uint32_t *scan_failed(const uint64_t *partials, int n);
// The depth order of n Gaussians (keys and record indices from the
// preprocess) and the scan in that order.
struct OrderArgs {
    uint32_t *keys, *vals, *keys_alt, *vals_alt;
    void *sort_scratch;  // depth_sort_scratch_bytes(n)
    const uint2 *cc;     // by record
    uint32_t *offsets, *coff, *chunk_first;
    uint32_t chunk_cap;
    uint64_t *partials;  // as launch_scan_cells
    uint64_t *n_pairs, *n_pairs_host, *n_cells;  // n_pairs_host as launch_scan
    uint64_t capacity;
    uint32_t *err;
};
// *in_alt: the order lies in vals_alt.
cudaError_t launch_depth_order(const OrderArgs &a, int n, cudaStream_t s, bool *in_alt);
// Output positions per entry of the scan's chunk table (a divisor of every
// emit kernel's per-warp output range).
constexpr uint32_t kEmitStride = 128;
inline uint64_t chunk_table_size(uint64_t pair_capacity) { return pair_capacity / kEmitStride + 1; }
size_t scan_partials_count(int n);
cudaError_t launch_emit(const EmitArgs &a, uint64_t *keys, cudaStream_t s);
cudaError_t launch_expand_ranges(const uint2 *ranges, int ntiles, uint32_t *out, uint64_t n_out, cudaStream_t s);
// scan_fail: the failure word of the pairs' scan, or null; sort_scratch: of their sort.
cudaError_t launch_ranges(const uint64_t *keys, uint64_t n_max, const uint64_t *n_dev, uint2 *ranges, int ntiles,
                          const uint32_t *scan_fail, void *sort_scratch, cudaStream_t s);
// The depth-first binning after the depth order and the scan: the emit of
// (cell, Gaussian, tile bits) entries; then their sort by cell and the
// expansion to the sorted values and ranges.
CellGeo cell_geo(int W, int H, int digit_bits);
// Scratch of the cell sort for images of at most max_cells cells and any digit width.
size_t cell_sort_scratch_bytes(uint64_t pair_capacity, int max_cells);
cudaError_t launch_cell_emit(const CellBin &b, cudaStream_t s);
cudaError_t launch_cell_sort(const CellBin &b, cudaStream_t s);
// Sorts b's entries by cell (bucket offsets already in the scratch's table,
// look-back words and counters cleared); values only from the last pass.
// *in_b: the sorted values lie in vals_b.
cudaError_t cell_sort_passes(const CellBin &b, cudaStream_t s, bool *in_b);
cudaError_t launch_render(const RenderArgs &a, cudaStream_t s);
cudaError_t launch_l1_grad(const float *img, const float *target, float *dL, uint64_t n, float scale, double *loss,
                           cudaStream_t s);
cudaError_t launch_zero5(float *const p[5], const uint64_t n[5], cudaStream_t s);
cudaError_t launch_adam(float *p, const float *g, float *m, float *v, uint64_t n, float lr, float b1, float b2,
                        float eps, int t, cudaStream_t s);
cudaError_t launch_render_bwd(const BwdArgs &a, cudaStream_t s);
cudaError_t launch_preprocess_bwd(const PreBwdArgs &a, int deg, cudaStream_t s);

}  // namespace qb
