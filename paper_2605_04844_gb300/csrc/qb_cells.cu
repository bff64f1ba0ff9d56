// qb_cells.cu -- K3-K5 of the depth-first path (DuplicateWithKeys with QPass
// traversal, SortPairs and the tile ranges of Sec. 2 and 3.2), through cells
// of 8 x 4 tiles.
//
// Sorting every (tile, Gaussian) pair moves each pair through memory several
// times (emit, histogram, two digit passes: about 40 bytes and a dozen
// instructions per pair).  A Gaussian's tiles lie in few cells, 8 to 24 tiles
// of it per cell on the frames measured, so here one entry stands for all its tiles in a
// cell: (cell id; Gaussian | tile bits << 32).  The entries are emitted in
// depth order and sorted by cell, one digit pass at 1080p over a twelfth of
// the elements, and only then expanded:
//   cell_count    per row (at most kCellRow consecutive entries of one cell) the number of
//                 entries of each of the cell's 32 tiles: the tile bits of 32
//                 entries, transposed across a warp, are one word per tile;
//   cell_prefix   per cell the exclusive prefix over its rows, the tiles'
//                 totals, and from these the ranges of all tiles;
//   cell_expand   per row, each tile's Gaussians to the tile's list, 32
//                 entries at a time: a ballot per tile gives the compacted
//                 positions, so a tile's stores are contiguous.
// The result (values in tile order, depth order within a tile; the ranges)
// is the one of the stable sort of all pairs by tile id.
// One GB300, start of the frame to its sorted values without the depth order:
// 1M Gaussians at 1080p (34.8M pairs, 2.7M entries), emit + histogram + two
// pair passes 0.54 ms, now 0.21; 3-sigma boxes (100.8M pairs, 5.0M entries)
// 1.36 -> 0.35 ms; 3840 x 2160 (126M pairs, 6.4M entries) 1.9 -> 0.53 ms.
#include <algorithm>

#include "qb_scan.cuh"
#include "qb_sweep.cuh"

namespace qb {

constexpr int kCellWarps = 8;          // warps per emit block
// Entries per warp and step: at most kCellChunk (512: 26 instead of 20 us for
// 400k entries), and no more than spread the entries over all warps of the
// grid, in steps of kEmitStride (10k Gaussians at 256 x 256 15.6 -> 12.7 us,
// 200k at 1001 x 701 18.8 -> 16.5; steps of 64 10.2 and 17.5, but the scan's
// larger table cost 3 us of 17 at 3840 x 2160).
constexpr uint32_t kCellChunk = 256;
constexpr int kCellHistMax = 4096;     // cells a block's histogram holds in shared memory
static_assert(kCellChunk % kEmitStride == 0, "a warp's range starts on the scan's chunk table");

CellGeo cell_geo(int W, int H, int digit_bits) {
    CellGeo g;
    g.tiles_x = (W + kTile - 1) / kTile;
    g.tiles_y = (H + kTile - 1) / kTile;
    g.ntiles = g.tiles_x * g.tiles_y;
    g.cells_x = (g.tiles_x + kCellX - 1) / kCellX;
    g.cells_y = (g.tiles_y + kCellY - 1) / kCellY;
    g.ncells = g.cells_x * g.cells_y;
    g.cell_bits = 0;
    while ((1 << g.cell_bits) < g.ncells + 1) ++g.cell_bits;  // id ncells: entries without a tile
    g.passes = pass_geo(g.cell_bits, digit_bits);
    g.digit_bits = std::max(g.passes.bits[0], 4);  // (a pass of fewer than 4 bits runs with 16 digits)
    return g;
}

size_t cell_sort_scratch_bytes(uint64_t pair_capacity, int max_cells) {
    size_t words = 0;  // look-back words per tile of the passes together
    for (int bits = 1; bits == 1 || (1 << (bits - 1)) < max_cells + 1; ++bits)
        for (int d = 8; d <= kMaxDigitBits; ++d) {
            const PassGeo g = pass_geo(bits, d);
            words = std::max(words, (size_t)g.passes << std::max(g.bits[0], 4));
        }
    return align256(kSortHeader + sort_tiles(pair_capacity) * words * 4);
}

__device__ __forceinline__ uint64_t cell_value(uint32_t gid, uint32_t bits) { return ((uint64_t)bits << 32) | gid; }

__device__ __forceinline__ uint32_t tiles_in_cell(const uint4 &w0, const uint4 &w1, int cx, int cy) {
    return cell_bits_of(unpack_rect(w0.x, w0.y), cx, cy) | cell_bits_of(unpack_rect(w0.z, w0.w), cx, cy) |
           cell_bits_of(unpack_rect(w1.x, w1.y), cx, cy) | cell_bits_of(unpack_rect(w1.z, w1.w), cx, cy);
}

// 32 Gaussians of a warp: their cells' bounding boxes and tile rectangles.
struct CellTable {
    int4 box[32];    // range position of its first entry, first cell x | y << 16, cells per row, Gaussian
    float2 inv[32];  // 1 / cells per row; entries of a Gaussian that skips cells (cell_entries), else 0
    uint4 rects[32][2];
};

// Entries [C, C + L) in emission order, by one warp: the Gaussian whose run
// holds entry C comes from the scan's table; the following ones are taken 32
// at a time, one per lane, and the range is produced 32 consecutive entries at
// a time: lane q finds the Gaussian of its entry from a ballot of the run
// starts in its group (every Gaussian with entries comes before those without
// in depth order, so run starts and lanes correspond), and the entry's cell by
// a division by its box's width.
__device__ __forceinline__ void cell_emit_range(const CellBin &b, uint64_t E, uint64_t C, int32_t L, CellTable &S,
                                                uint32_t *hist) {
    const int lane = threadIdx.x & 31;
    const uint32_t le_mask = lanemask_le();
    const uint32_t none = (uint32_t)b.geo.ncells;
    int64_t j0 = b.chunk_first[C / kEmitStride];
    int32_t done_to = 0;  // range positions [0, done_to) produced
    // The loads of a batch are taken ahead of it, the Gaussians and their runs
    // (which the rectangles wait for) two batches, the rectangles one: a warp's
    // half dozen batches would otherwise cost two memory latencies each.
    struct Run {
        uint32_t gid, at, end;  // (entries: E beyond the last Gaussian)
    };
    auto load_run = [&](int64_t j) {
        Run r{0u, (uint32_t)E, (uint32_t)E};
        if (j < b.n) {
            r.gid = b.perm[j];
            r.at = b.coff[j];
            if (j + 1 < b.n) r.end = b.coff[j + 1];
        }
        return r;
    };
    auto load_rects = [&](const Run &r, uint4 &w0, uint4 &w1) {
        w0 = w1 = make_uint4(1u | (1u << 16), 0u, 1u | (1u << 16), 0u);  // empty rectangles
        if (r.end > r.at) {
            w0 = b.rects[2 * (size_t)r.gid];
            w1 = b.rects[2 * (size_t)r.gid + 1];
        }
    };
    Run cur_run = load_run(j0 + lane), next_run = load_run(j0 + 32 + lane);
    uint4 w0, w1;
    load_rects(cur_run, w0, w1);
    while (done_to < L && j0 < b.n) {
        // the run of position j0 + lane, relative to C
        const int64_t rel = (int64_t)cur_run.at - (int64_t)C, end = (int64_t)cur_run.end - (int64_t)C;
        const uint32_t gid = cur_run.gid;
        const bool relevant = end > rel && rel < L && end > 0;
        __syncwarp();
        if (relevant) {
            const Rect r[4] = {unpack_rect(w0.x, w0.y), unpack_rect(w0.z, w0.w), unpack_rect(w1.x, w1.y),
                               unpack_rect(w1.z, w1.w)};
            const Rect box = cell_box(r);
            const int bw = box.x1 - box.x0 + 1, cells = bw * (box.y1 - box.y0 + 1);
            S.box[lane] = make_int4((int32_t)rel, box.x0 | (box.y0 << 16), bw, (int)gid);
            S.inv[lane] = make_float2(1.0f / (float)bw, cells != (int)(end - rel) ? (float)cells : 0.f);
            S.rects[lane][0] = w0;
            S.rects[lane][1] = w1;
        }
        cur_run = next_run;
        load_rects(cur_run, w0, w1);
        next_run = load_run(j0 + 64 + lane);
        // where the lane's run starts among the positions still to come
        const int32_t start = relevant && rel > done_to ? (int32_t)rel : INT32_MAX;
        // the Gaussian of position done_to
        int cur = __popc(__ballot_sync(0xffffffffu, rel <= done_to)) - 1;
        const int64_t last_end = __shfl_sync(0xffffffffu, end, 31);
        const int32_t batch_end = (int32_t)(last_end < (int64_t)L ? last_end : (int64_t)L);
        __syncwarp();
        for (int32_t c0 = done_to; c0 < batch_end; c0 += 32) {
            // runs that start in this group (the first position's is cur already)
            const uint32_t ahead = (uint32_t)(start - c0);
            const uint32_t M = __reduce_or_sync(0xffffffffu, ahead < 32u ? 1u << ahead : 0u);
            const int32_t p = c0 + lane;
            if (p < batch_end) {
                const int idx = cur + __popc(M & le_mask);
                const int4 B = S.box[idx];
                const float2 inv = S.inv[idx];
                const uint4 w0 = S.rects[idx][0], w1 = S.rects[idx][1];
                uint32_t k = (uint32_t)(p - B.x);
                const int x0 = B.y & 0xffff, y0 = B.y >> 16;
                uint32_t q, r;
                if (inv.y != 0.f) {  // entry k is the k-th of the box's cells that hold a tile
                    uint32_t c = 0;
                    for (uint32_t left = k + 1; c < (uint32_t)inv.y; ++c) {
                        seg_divide(c, (uint32_t)B.z, inv.x, q, r);
                        if (tiles_in_cell(w0, w1, x0 + (int)r, y0 + (int)q) && --left == 0u) break;
                    }
                    k = c;
                }
                seg_divide(k, (uint32_t)B.z, inv.x, q, r);
                const int cx = x0 + (int)r, cy = y0 + (int)q;
                const uint32_t bits = tiles_in_cell(w0, w1, cx, cy);
                const uint32_t cell = bits ? (uint32_t)(cy * b.geo.cells_x + cx) : none;
                b.arr.keys_a[C + p] = cell;
                b.arr.vals_a[C + p] = cell_value((uint32_t)B.w, bits);
                atomicAdd(hist + cell, 1u);
            }
            cur += __popc(M);
        }
        done_to = max(done_to, batch_end);
        j0 += 32;
    }
}

// The same for QuadBox-dagger (no QPass): one thread per Gaussian runs nested
// loops over the cells of each sub-box and skips those an earlier one holds.
__device__ __forceinline__ void cell_emit_naive(const CellBin &b, int64_t j, uint32_t *hist) {
    const uint32_t gid = b.perm[j];
    const uint32_t off = b.coff[j];
    const uint32_t end = j + 1 < b.n ? b.coff[j + 1] : (uint32_t)*b.n_cells;
    if (end == off) return;
    const uint4 w0 = b.rects[2 * (size_t)gid], w1 = b.rects[2 * (size_t)gid + 1];
    const Rect r[4] = {cell_rect(unpack_rect(w0.x, w0.y)), cell_rect(unpack_rect(w0.z, w0.w)),
                       cell_rect(unpack_rect(w1.x, w1.y)), cell_rect(unpack_rect(w1.z, w1.w))};
    uint32_t at = off;
    for (int q = 0; q < 4; ++q) {
        if (rect_empty(r[q])) continue;
        for (int cy = r[q].y0; cy <= r[q].y1; ++cy)
            for (int cx = r[q].x0; cx <= r[q].x1; ++cx) {
                bool seen = false;
                for (int p = 0; p < q; ++p) seen |= in_rect(r[p], cx, cy);
                if (seen || at >= end) continue;
                const uint32_t cell = (uint32_t)(cy * b.geo.cells_x + cx);
                b.arr.keys_a[at] = cell;
                b.arr.vals_a[at] = cell_value(gid, tiles_in_cell(w0, w1, cx, cy));
                atomicAdd(hist + cell, 1u);
                ++at;
            }
    }
}

// From the cells' entry counts, run by one block: the first entry and first
// row of each cell, and every sort pass's exclusive bucket offsets.  A digit
// d of pass p (width b, shift h) covers the runs of 2^h consecutive cells
// that start at u 2^(b+h) + d 2^h; each run's sum is a difference of two
// offsets.  s_dsum has room for 2^kMaxDigitBits digit sums.
__device__ __forceinline__ void cell_prepare(const CellBin &b, uint32_t *s_dsum) {
    constexpr int U = 4;
    const int ncells = b.geo.ncells, ids = ncells + 1;  // (id ncells: entries without a tile, no rows)
    uint32_t entries = 0, rows = 0;  // before this step's cells
    for (int c0 = 0; c0 < ids; c0 += U * (int)blockDim.x) {
        uint32_t v[U], sum = 0, rsum = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + (int)threadIdx.x * U + u;
            v[u] = c < ids ? __ldcg(b.arr.count + c) : 0u;
            sum += v[u];
            rsum += c < ncells ? (v[u] + kCellRow - 1) / kCellRow : 0u;
        }
        uint32_t total, rtotal;
        uint32_t e = entries + block_incl_scan<uint32_t>(sum, &total) - sum;
        uint32_t r = rows + block_incl_scan<uint32_t>(rsum, &rtotal) - rsum;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + (int)threadIdx.x * U + u;
            if (c < ids) {
                b.arr.start[c] = e;
                b.arr.row_start[c] = r;  // [ncells]: the rows there are
            }
            e += v[u];
            r += c < ncells ? (v[u] + kCellRow - 1) / kCellRow : 0u;
        }
        entries += total;
        rows += rtotal;
    }
    if (threadIdx.x == 0) b.arr.start[ids] = entries;
    __threadfence_block();
    __syncthreads();
    uint32_t *table = sort_hist_at(b.sort_scratch);
    const volatile uint32_t *start = b.arr.start;
    for (int p = 0; p < b.geo.passes.passes; ++p) {
        const int bits = b.geo.passes.bits[p], sh = b.geo.passes.shift[p];
        const int Rp = 1 << bits, period = Rp << sh;
        const int runs = Rp * ((ids + period - 1) / period);
        for (int d = threadIdx.x; d < Rp; d += blockDim.x) s_dsum[d] = 0u;
        __syncthreads();
        for (int i = threadIdx.x; i < runs; i += blockDim.x) {
            const int d = i & (Rp - 1), u = i >> bits;
            const int c = u * period + (d << sh);
            if (c >= ids) continue;
            const uint32_t v = start[min(ids, c + (1 << sh))] - start[c];
            if (v) atomicAdd(&s_dsum[d], v);
        }
        __syncthreads();
        const int per = (Rp + (int)blockDim.x - 1) / (int)blockDim.x;
        const int d0 = (int)threadIdx.x * per, d1 = min(Rp, d0 + per);
        uint32_t sum = 0;
        for (int d = d0; d < d1; ++d) sum += s_dsum[d];
        uint32_t tot;
        uint32_t r = block_incl_scan<uint32_t>(sum, &tot) - sum;
        for (int d = d0; d < d1; ++d) {
            table[p * kHistStride + d] = r;
            r += s_dsum[d];
        }
        __syncthreads();
    }
}

// The emit, with a histogram of the cells (in shared memory up to
// kCellHistMax cells) whose last block makes the cells' offsets.  It also
// zeroes the look-back words and counters of the sort's passes, sized by the
// entries there are and not by the capacity.
//
// Bound by issue slots.  Decomposing every Gaussian's cells into QPass runs
// took 41M warp instructions and 79 us for 1M Gaussians at 1080p (2.7M entries);
// now 48 us (20 us for 200k at 1001 x 701, was 49).  (A thread per Gaussian that runs through a small box, and a block's
// warps sharing the large ones, took 72 us, and 104 instead of 48 for 3M at
// 1440p seen from inside, where the nearest Gaussians' boxes fill the image.)
template <bool NAIVE>
__global__ void __launch_bounds__(kCellWarps * 32) cell_emit_kernel(CellBin b) {
    extern __shared__ __align__(16) uint8_t smem[];
    CellTable *s_tab = reinterpret_cast<CellTable *>(smem);
    uint32_t *s_hist = reinterpret_cast<uint32_t *>(smem + (NAIVE ? 0 : kCellWarps * sizeof(CellTable)));
    __shared__ bool s_last;
    const int tid = threadIdx.x, wid = tid >> 5;
    const bool in_smem = b.geo.ncells < kCellHistMax;
    const uint64_t E = *b.n_cells;  // (0 after a scan that failed)
    if (blockIdx.x == 0 && tid == 0 && *b.n_pairs > b.capacity) atomicOr(b.err, kErrCapacity);
    if (in_smem)
        for (int c = tid; c <= b.geo.ncells; c += blockDim.x) s_hist[c] = 0u;
    const uint64_t threads = (uint64_t)gridDim.x * blockDim.x, gt = (uint64_t)blockIdx.x * blockDim.x + tid;
    for (int p = 0; p < b.geo.passes.passes; ++p) {
        uint32_t *lb = sort_lookback_at(b.sort_scratch, b.capacity, b.geo.digit_bits, p);
        // (a pass of fewer than 4 bits still runs with 16 digits)
        const uint64_t words = ((E + kSortTile - 1) / kSortTile) << max(b.geo.passes.bits[p], 4);
        for (uint64_t i = gt; i < words; i += threads) lb[i] = 0u;
        if (gt == 0) *sort_counter_at(b.sort_scratch, p) = 0u;
    }
    if (gt == 0) *sort_failed_at(b.sort_scratch) = 0u;
    __syncthreads();
    uint32_t *hist = in_smem ? s_hist : b.arr.count;
    if constexpr (NAIVE) {
        if (E > 0)
            for (uint64_t j = gt; j < (uint64_t)b.n; j += threads) cell_emit_naive(b, (int64_t)j, hist);
    } else {
        const uint64_t warps = (uint64_t)gridDim.x * kCellWarps;
        const uint64_t even = (E + warps * kEmitStride - 1) / (warps * kEmitStride) * kEmitStride;
        const uint64_t chunk = min((uint64_t)kCellChunk, even);
        for (uint64_t C = ((uint64_t)blockIdx.x * kCellWarps + wid) * chunk; C < E; C += warps * chunk)
            cell_emit_range(b, E, C, (int32_t)min(chunk, E - C), s_tab[wid], hist);
    }
    if (in_smem) {
        __syncthreads();
        for (int c = tid; c <= b.geo.ncells; c += blockDim.x) {
            const uint32_t v = s_hist[c];
            if (v) atomicAdd(b.arr.count + c, v);
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(b.arr.count + b.geo.ncells + 1, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    cell_prepare(b, reinterpret_cast<uint32_t *>(smem));  // the table and histogram are no longer needed
}

cudaError_t launch_cell_emit(const CellBin &b, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(b.arr.count, 0, 4 * cell_zero_words(b.geo.ncells), s);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t hist = b.geo.ncells < kCellHistMax ? 4 * ((size_t)b.geo.ncells + 1) : 0;
    const size_t dsum = (size_t)4 << kMaxDigitBits;
    if (b.naive) {
        const size_t smem = std::max(hist, dsum);
        const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>(((uint64_t)b.n + 255) / 256, (uint64_t)sms * 8));
        note_launch("cell_emit_naive_kernel", s),
            cell_emit_kernel<true><<<(unsigned)blocks, kCellWarps * 32, smem, s>>>(b);
        return cudaGetLastError();
    }
    const size_t smem = std::max(kCellWarps * sizeof(CellTable) + hist, dsum);
    const uint64_t want = (b.n_cells_max + kCellWarps * kEmitStride - 1) / (kCellWarps * kEmitStride);
    const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)sms * 6));
    note_launch("cell_emit_kernel", s), cell_emit_kernel<false><<<(unsigned)blocks, kCellWarps * 32, smem, s>>>(b);
    return cudaGetLastError();
}

// Bit i of lane t's result is bit t of lane i's x (a 32 x 32 bit transpose).
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        // columns whose index has bit j clear
        const uint32_t m = j == 16 ? 0x0000ffffu : j == 8 ? 0x00ff00ffu : j == 4 ? 0x0f0f0f0fu
                                                          : j == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
        x = (lane & j) ? (x & ~m) | ((y >> j) & m) : (x & m) | ((y & m) << j);
    }
    return x;
}

// The cell that owns row r, found by one warp (32-ary search of row_start).
__device__ __forceinline__ int cell_of_row(const uint32_t *row_start, int ncells, uint32_t r, int lane) {
    int lo = 0, hi = ncells - 1;  // row_start[lo] <= r, answer in [lo, hi]: the last cell with row_start <= r
    while (hi > lo) {
        const int span = hi - lo;
        const int probe = lo + (int)(((int64_t)span * (lane + 1) + 31) / 32);  // 32 probes in (lo, hi]
        const uint32_t m = __ballot_sync(0xffffffffu, row_start[probe] <= r);
        const int k = m ? 31 - __clz(m) : -1;  // highest probe at or below r
        const int new_lo = k >= 0 ? lo + (int)(((int64_t)span * (k + 1) + 31) / 32) : lo;
        const int new_hi = k < 31 ? lo + (int)(((int64_t)span * (k + 2) + 31) / 32) - 1 : hi;
        lo = new_lo;
        hi = max(new_lo, new_hi);
    }
    return lo;
}

// The tile of bit `lane` of a cell, or -1 beyond the image.
__device__ __forceinline__ int tile_of_lane(const CellGeo &g, int cell, int lane) {
    const int cy = cell / g.cells_x, cx = cell - cy * g.cells_x;
    const int tx = (cx << kCellXShift) + (lane & (kCellX - 1)), ty = (cy << kCellYShift) + (lane >> kCellXShift);
    return tx < g.tiles_x && ty < g.tiles_y ? ty * g.tiles_x + tx : -1;
}

constexpr int kRowWarps = 8;  // warps per block of the row kernels

__global__ void __launch_bounds__(kRowWarps * 32) cell_count_kernel(CellGeo g, CellArrays a,
                                                                    const uint64_t *__restrict__ vals) {
    const int lane = threadIdx.x & 31;
    const uint32_t rows = a.row_start[g.ncells];
    for (uint32_t r = blockIdx.x * kRowWarps + (threadIdx.x >> 5); r < rows; r += gridDim.x * kRowWarps) {
        const int cell = cell_of_row(a.row_start, g.ncells, r, lane);
        const uint32_t first = a.start[cell] + (r - a.row_start[cell]) * kCellRow;
        const uint32_t end = min(first + kCellRow, a.start[cell + 1]);
        uint32_t bits[kCellRow / 32];
#pragma unroll
        for (int k = 0; k < (int)kCellRow / 32; ++k) {
            const uint32_t i = first + 32 * k + lane;
            bits[k] = i < end ? (uint32_t)(vals[i] >> 32) : 0u;
        }
        uint32_t c = 0;
#pragma unroll
        for (int k = 0; k < (int)kCellRow / 32; ++k) c += __popc(warp_transpose(bits[k], lane));
        a.row_counts[(size_t)r * 32 + lane] = tile_of_lane(g, cell, lane) >= 0 ? c : 0u;
        if (lane == 0) a.row_cell[r] = (uint32_t)cell;
    }
}

// Block c turns cell c's rows into their exclusive prefix (a warp takes a
// contiguous part of the rows) and writes the totals of its tiles; the last
// block scans the totals into the ranges ([0, 0) for an empty tile).
constexpr int kPrefixThreads = 512;
__global__ void __launch_bounds__(kPrefixThreads, 3) cell_prefix_kernel(CellGeo g, CellArrays a, uint2 *__restrict__ ranges,
                                                           const uint64_t *n_pairs, const uint64_t *n_cells,
                                                           const uint32_t *sort_failed) {
    __shared__ uint32_t s_part[kPrefixThreads / 32][32];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int cell = blockIdx.x;
    const bool failed = *sort_failed != 0u;
    const uint32_t r0 = a.row_start[cell], nr = a.row_start[cell + 1] - r0;
    const uint32_t per = (nr + nw - 1) / nw;
    const uint32_t w0 = min(nr, wid * per), w1 = min(nr, w0 + per);
    uint32_t *rows = a.row_counts + (size_t)r0 * 32 + lane;
    uint32_t sum = 0;
#pragma unroll 8
    for (uint32_t r = w0; r < w1; ++r) sum += __ldcg(rows + (size_t)r * 32);
    s_part[wid][lane] = sum;
    __syncthreads();
    uint32_t run = 0, total = 0;
    for (int w = 0; w < nw; ++w) {
        const uint32_t v = s_part[w][lane];
        run += w < wid ? v : 0u;
        total += v;
    }
    for (uint32_t r = w0; r < w1; r += 8) {
        uint32_t v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = r + k < w1 ? __ldcg(rows + (size_t)(r + k) * 32) : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (r + k < w1) rows[(size_t)(r + k) * 32] = run;
            run += v[k];
        }
    }
    if (wid == 0) {
        const int t = tile_of_lane(g, cell, lane);
        if (t >= 0) a.tile_total[t] = total;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.count + g.ncells + 2, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // exclusive scan over the tiles, eight consecutive ones per thread
    uint64_t before = 0;
    for (int t0 = 0; t0 < g.ntiles; t0 += 8 * (int)blockDim.x) {
        const int t = t0 + 8 * (int)threadIdx.x;
        uint32_t v[8], s = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[k] = t + k < g.ntiles ? __ldcg(a.tile_total + t + k) : 0u;
            s += v[k];
        }
        uint32_t tot;
        uint32_t e = (uint32_t)before + block_incl_scan<uint32_t>(s, &tot) - s;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (t + k < g.ntiles) ranges[t + k] = v[k] ? make_uint2(e, e + v[k]) : make_uint2(0u, 0u);
            e += v[k];
        }
        before += tot;
    }
    // After a look-back time-out the sorted entries are undefined, and some of
    // them whatever the buffer held: nothing is expanded.  (Nor if the tiles'
    // totals did not add up to the pairs there are.)
    if (failed || (*n_cells > 0 && before != *n_pairs)) {
        __syncthreads();  // the ranges above were written by other threads
        for (int t = threadIdx.x; t < g.ntiles; t += blockDim.x) ranges[t] = make_uint2(0u, 0u);
        if (threadIdx.x == 0) a.row_start[g.ncells] = 0u;
    }
}

// The stores bound it: each carries a dozen to 20 words of one tile at any
// alignment, and the memory-side queue is full (the largest stall) at 4.5 TB/s
// of sectors.  What else goes through that queue is kept small: the 32 tiles'
// places come from shared memory four at a time, not by 32 shuffles (1M
// Gaussians at 1080p 81 -> 77 us, with 3-sigma boxes 203 -> 193).  Staging a
// row's values in shared memory to write whole 128-byte lines was slower (122,
// 245 us): the values then pass the queue three times.
__global__ void __launch_bounds__(kRowWarps * 32) cell_expand_kernel(CellGeo g, CellArrays a,
                                                                     const uint64_t *__restrict__ in,
                                                                     const uint2 *__restrict__ ranges,
                                                                     uint32_t *__restrict__ vals) {
    __shared__ __align__(16) uint32_t s_base[kRowWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
    const uint32_t rows = a.row_start[g.ncells];
    for (uint32_t r = blockIdx.x * kRowWarps + w; r < rows; r += gridDim.x * kRowWarps) {
        const int cell = (int)a.row_cell[r];
        const uint32_t first = a.start[cell] + (r - a.row_start[cell]) * kCellRow;
        const uint32_t end = min(first + kCellRow, a.start[cell + 1]);
        uint64_t e[kCellRow / 32];
#pragma unroll
        for (int k = 0; k < (int)kCellRow / 32; ++k) {
            const uint32_t i = first + 32 * k + lane;
            e[k] = i < end ? in[i] : 0ull;
        }
        const int t = tile_of_lane(g, cell, lane);
        const uint32_t have = __ballot_sync(0xffffffffu, t >= 0);
        uint32_t base = t >= 0 ? ranges[t].x + a.row_counts[(size_t)r * 32 + lane] : 0u;
#pragma unroll
        for (int k = 0; k < (int)kCellRow / 32; ++k) {
            if (first + 32 * k >= end) break;  // warp-uniform
            const uint32_t gid = (uint32_t)e[k], bits = (uint32_t)(e[k] >> 32) & have;
            __syncwarp();  // the places of the 32 entries before have been read
            s_base[w][lane] = base;
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 32; q += 4) {
                const uint4 to4 = *reinterpret_cast<const uint4 *>(&s_base[w][q]);
                const uint32_t to[4] = {to4.x, to4.y, to4.z, to4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool on = (bits >> (q + j)) & 1u;
                    const uint32_t m = __ballot_sync(0xffffffffu, on);
                    if (on) vals[to[j] + __popc(m & lt)] = gid;
                }
            }
            base += __popc(warp_transpose(bits, lane));
        }
    }
}

cudaError_t launch_cell_sort(const CellBin &b, cudaStream_t s) {
    bool in_b = false;
    cudaError_t e = cell_sort_passes(b, s, &in_b);
    if (e != cudaSuccess) return e;
    const uint64_t *sorted = in_b ? b.arr.vals_b : b.arr.vals_a;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t rows = cell_rows_max(b.n_cells_max, b.geo.ncells);
    const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>((rows + kRowWarps - 1) / kRowWarps, (uint64_t)sms * 8));
    note_launch("cell_count_kernel", s),
        cell_count_kernel<<<(unsigned)blocks, kRowWarps * 32, 0, s>>>(b.geo, b.arr, sorted);
    note_launch("cell_prefix_kernel", s),
        cell_prefix_kernel<<<b.geo.ncells, kPrefixThreads, 0, s>>>(b.geo, b.arr, b.ranges, b.n_pairs, b.n_cells,
                                                                sort_failed_at(b.sort_scratch));
    note_launch("cell_expand_kernel", s),
        cell_expand_kernel<<<(unsigned)blocks, kRowWarps * 32, 0, s>>>(b.geo, b.arr, sorted, b.ranges, b.vals);
    return cudaGetLastError();
}

}  // namespace qb
