// qb_internal.cuh -- shared device helpers and workspace layout of libquadbox.
// Method: QuadBox (arXiv 2605.04844); see include/quadbox.h for the ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/quadbox.h"

namespace qb {

constexpr int kTile = 16;             // 16 x 16 pixel tiles (Sec. 2)
constexpr int kTileShift = 4;
constexpr float kAlphaMin = 1.0f / 255.0f;  // alpha_min (Sec. 3.1.1)
constexpr float kAlphaMax = 0.99f;          // opacity cap (3DGS convention)
constexpr float kTStop = 1e-4f;             // transmittance stop (3DGS convention)
constexpr float kDilation = 0.3f;           // low-pass dilation of Sigma^2D
constexpr int kDepthBits = 31;              // key = (tile << 31) | depth bits
constexpr uint32_t kErrCapacity = 1u;
constexpr uint32_t kErrTimeout = 2u;
constexpr int kMaxDigitBits = 11;
constexpr int kDepthDigitBits = 8;  // the depth-order sort: 31 bits in 4 passes (8 + 8 + 8 + 7)
constexpr int kMaxPasses = 8;              // ceil(64 / 8)

// meta bits
constexpr int kMetaVisible = 1;
constexpr int kMetaOrient = 2;
constexpr int kMetaClampShift = 2;
constexpr int kMetaNonFinite = 32;  // a colour channel is infinite or NaN

struct CamDev {
    float V[12];  // rows 0..2 of the world->view matrix
    float fx, fy, cx, cy;
    float limx, limy;  // 1.3 * tan_fov
    float campos[3];
    float znear;
    int W, H;
};

// Workspace offsets (bytes) of a frame; all 256-byte aligned.
struct Layout {
    size_t xy, shape, conic_o, rgbd, box, r3, meta, counts, offsets;
    size_t rects;  // [n] packed sub-box tile rectangles (pack_rects)
    size_t cc;     // [n] (tile count, cell count)
    size_t coff;   // [n] cell offsets in emission order (DEPTH_FIRST)
    size_t chunk_first;  // the emit's chunk table
    size_t scan_part;
    size_t keys0, keys1, vals0, vals1;
    size_t sort_scratch, sort_scratch_bytes;
    size_t dkeys0, dkeys1, dvals0, dvals1, dsort_scratch;  // depth order of the Gaussians
    size_t ranges, tfinal, ncontrib, neval;
    size_t cell_zero;    // cell counts and finished-block counters (CellLayout)
    size_t cell_start, row_start, row_cell, row_counts, tile_total;  // CellArrays (the rows inside vals1)
    size_t order_cnt;   // [2][kOrderBuckets]: tile orders by the backward's work (TileOrder)
    size_t order_list;  // [2][kOrderBuckets][tiles]
    size_t bwd_list, bwd_count;  // Gaussians with a screen-space gradient; their number (just before gscreen)
    size_t gscreen;  // [n][9] screen-space gradients
    size_t state;  // u64 n_pairs, u32 err_flags, padding
    size_t total;
};

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Sets the message qb_last_error() returns on the calling thread.
void set_last_error(const char *msg);
// Counts one kernel launch of the library (qb_kernel_launches) and reports
// it to the launch hook, if one is set, just before the launch on stream s.
void note_launch(const char *kernel, cudaStream_t s);
// A number of the calling thread's CUDA context that no other context of the
// process has or had (a cudaDeviceReset makes a new one), or 0 if it cannot be
// told.  What is kept from one call for the next is kept under it.
uint64_t context_id();
// Raises kernel func's dynamic shared-memory limit in the current context to
// at least bytes; the limit set is remembered per (kernel, context), and the
// calls are safe from several host threads.
cudaError_t ensure_dyn_smem(const void *func, size_t bytes);

// ---- sort -------------------------------------------------------------------
// Digit geometry of an LSD radix sort on bits [0, end_bit) with digits of at
// most digit_bits: ceil(end_bit / digit_bits) passes whose widths differ by at
// most one (13 bits at 8: 7 + 6), pass p on bits [shift[p], shift[p] + bits[p]).
struct PassGeo {
    int passes;
    int shift[kMaxPasses], bits[kMaxPasses];
};

__host__ __device__ inline PassGeo pass_geo(int end_bit, int digit_bits) {
    PassGeo g;
    g.passes = end_bit > 0 ? (end_bit + digit_bits - 1) / digit_bits : 0;
    int sh = 0;
    for (int p = 0; p < kMaxPasses; ++p) {
        const int w = p < g.passes ? end_bit / g.passes + (p < end_bit % g.passes ? 1 : 0) : 0;
        g.shift[p] = sh;
        g.bits[p] = w;
        sh += w;
    }
    return g;
}

size_t sort_scratch_bytes(uint64_t n, int end_bit, int digit_bits);
// Sorts pairs on bits [0, end_bit).  n_dev: device count (<= n_max) or null
// when n_max is exact.  Returns the number of passes; result lies in the alt
// buffers when the pass count is odd.
cudaError_t sort_pairs(uint64_t *keys, uint32_t *vals, uint64_t *keys_alt, uint32_t *vals_alt,
                       uint64_t n_max, const uint64_t *n_dev, int end_bit, int digit_bits,
                       void *scratch, uint32_t *err_flags, cudaStream_t stream, int *passes_out);
// The depth order's sort: 32-bit keys on kDepthBits bits in digits of
// kDepthDigitBits; scratch of depth_sort_scratch_bytes(n).
size_t depth_sort_scratch_bytes(uint64_t n);
cudaError_t sort_pairs(uint32_t *keys, uint32_t *vals, uint32_t *keys_alt, uint32_t *vals_alt,
                       uint64_t n_max, const uint64_t *n_dev, int end_bit, int digit_bits,
                       void *scratch, uint32_t *err_flags, cudaStream_t stream, int *passes_out);
// ---- device helpers -----------------------------------------------------------
// Gaussians whose stretching factor f (Eq. f-closed) has f^2 below this take
// the render's exact power form: with r = b / a = -Sigma12 / Sigma22 and
// u = dx + r dy, d^T Lambda d = a u^2 + dy^2 / Sigma22, a sum of two
// non-negative terms, where a dx^2 + 2 b dx dy + c dy^2 of a thin Gaussian
// cancels its large terms in float32 (an error of about 2^-24 (a dx^2 +
// 2 |b dx dy| + c dy^2), up to 10^5 times the result along a needle).
constexpr float kElongatedF2 = 0.01f;  // f < 0.1: aspect ratio above 10 : 1

// Exponents below this give alpha = o e^power < (1/255) e^-0.001: the 1e-3
// margin is far wider than the float32 error of the alpha test and of the
// fast logarithm (2^-21.4 absolute near 1, else 3 ulp: 1.5e-6 at o = 1, 6e-6
// at o = 10^6), so skipping them first never changes a decision of that test.
// EXACT takes logf itself: the counted render reports how many
// exponents pass, and a last bit of the threshold can move that number.
template <bool EXACT = false>
__device__ __forceinline__ float skip_threshold(float o) {
    return -(EXACT ? logf(255.0f * o) : __logf(255.0f * o)) - 1e-3f;
}

// e^x of both lanes as 2^(x log2 e), for the exponents of the compositing
// (at least skip_threshold, so the result is no subnormal and ex2's
// flush-to-zero form gives what its other form gives, without the rescaling
// that one needs; NaN stays NaN).
__device__ __forceinline__ float2 exp2_of(float2 x) {
    const float2 t = __fmul2_rn(x, make_float2(1.4426950408889634f, 1.4426950408889634f));
    float2 r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(t.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(t.y));
    return r;
}

// Whether some point of the pixel rectangle [x0, x1] x [y0, y1] can give the
// Gaussian (mu^2D, conic (a, b, c)) an exponent above t, i.e. whether the
// rectangle meets the ellipse q(d) = a dx^2 + 2 b dx dy + c dy^2 <= -2t,
// d = mu^2D - pixel.  q is convex with its minimum at d = 0, so over the
// rectangle it is smallest on an edge that faces d = 0 (or there, inside): at
// the 1D minimiser, clamped, on the lines through the rectangle's point
// nearest to 0 in x and in y.  The test is conservative: the radius gets a 1 %
// + 0.01 margin, far above the float32 error of q and of the kernels'
// exponents.  A degenerate conic always meets the rectangle.
//
// An elongated conic (shape = (r, -e/2) with r = b / a, e = 1 / Sigma22, not
// (0, 0)) is evaluated as a (dx + r dy)^2 + e dy^2, as the kernels do: both
// terms are non-negative, and what rounding costs is the error of dx + r dy,
// at most 3 x 2^-24 (|dx| + |r dy|) here and in the kernels' exponent together.
// It counts by sqrt(a) and sqrt(a) |r| <= sqrt(c), each at most 1 / sqrt(0.3)
// (Sigma's eigenvalues are at least the dilation): the Mahalanobis distance is
// off by less than d = 3.3e-7 D, D = |dx| + |dy|.  (R + d)^2 <= 1.01 R^2 +
// 101 d^2 for every radius R, so 1.2e-11 D^2 more in the squared radius covers it:
// 0.01 at 30000 pixels from mu^2D, everything from 10^6 on.  (Images are up to
// 32768 pixels and mu^2D may lie any distance outside; with the margin alone, 2 %
// of the rectangles that a needle reaches were missed at 10^7 pixels.)  The edge
// minimisers' rounding enters q squared, relative to D, and is far smaller.
// Before elongated conics were tested they met every rectangle: of the 19.4M
// entries staged for 3M Gaussians at 1440p seen from inside, where thin ones
// abound, 16.9M were walked and 2.8M reached a running pixel.
__device__ __forceinline__ bool ellipse_meets_rect(float mx, float my, float a, float b, float c, float t,
                                                   float2 shape, float x0, float y0, float x1, float y1) {
    if (!(a > 0.f && c > 0.f)) return true;
    float r2 = fmaxf(-2.f * t, 0.f) * 1.01f + 1e-2f;
    const float ul = mx - x1, uh = mx - x0, vl = my - y1, vh = my - y0;
    const bool elongated = shape.y != 0.f;
    const float ir = elongated ? shape.x : __fdividef(b, a);
    // on the vertical line dx = u1, and on the horizontal line dy = v2
    const float u1 = fminf(fmaxf(0.f, ul), uh), v1 = fminf(fmaxf(-__fdividef(b, c) * u1, vl), vh);
    const float v2 = fminf(fmaxf(0.f, vl), vh), u2 = fminf(fmaxf(-ir * v2, ul), uh);
    float q1, q2;
    if (elongated) {
        const float D = fabsf(u1) + fabsf(v2);
        r2 = fmaf(D * 1.2e-11f, D, r2);
        const float e = -2.f * shape.y, w1 = fmaf(ir, v1, u1), w2 = fmaf(ir, v2, u2);
        q1 = fmaf(a * w1, w1, e * v1 * v1);
        q2 = fmaf(a * w2, w2, e * v2 * v2);
    } else {
        q1 = fmaf(a * u1, u1, fmaf(2.f * b * u1, v1, c * v1 * v1));
        q2 = fmaf(a * u2, u2, fmaf(2.f * b * u2, v2, c * v2 * v2));
    }
    return !(fminf(q1, q2) > r2);
}

struct Rect {
    int x0, y0, x1, y1;  // inclusive tile bounds; empty if x0 > x1 || y0 > y1
};

__device__ __forceinline__ bool rect_empty(const Rect &r) { return r.x0 > r.x1 || r.y0 > r.y1; }

__device__ __forceinline__ Rect empty_rect() { return Rect{1, 1, 0, 0}; }

// Closed pixel interval [lo, hi] -> tiles of the pixel centres it holds,
// clipped to [0, npx-1].  Single IEEE float operations only (no contraction
// is possible: no products), so the integers are reproducible off-device.
__device__ __forceinline__ bool tiles_of(float lo, float hi, int npx, int &t0, int &t1) {
    float p0 = fmaxf(ceilf(lo), 0.0f);
    float p1 = fminf(floorf(hi), (float)(npx - 1));
    if (!(p0 <= p1)) return false;
    t0 = ((int)p0) >> kTileShift;
    t1 = ((int)p1) >> kTileShift;
    return true;
}

__device__ __forceinline__ Rect intersect(const Rect &a, const Rect &b) {
    Rect r{max(a.x0, b.x0), max(a.y0, b.y0), min(a.x1, b.x1), min(a.y1, b.y1)};
    return rect_empty(r) ? empty_rect() : r;
}

// The per-mode tile rectangles of one Gaussian (up to four sub-boxes).
// Quadrant order I (+x,+y), II (-x,+y), III (-x,-y), IV (+x,-y); orient = 1
// when Sigma12 >= 0, i.e. the major axis runs through quadrants I and III.
// Sub-boxes share the corner mu^2D (Sec. 3.1.2).
__device__ __forceinline__ int box_rects(float mx, float my, float4 box, float r3, bool orient, int mode,
                                         bool clamp3s, int W, int H, Rect out[4]) {
    out[0] = out[1] = out[2] = out[3] = empty_rect();
    Rect r3s;
    // __fadd_rn/__fsub_rn: one rounding each, never fused with a product.
    bool ok = tiles_of(__fsub_rn(ceilf(mx), r3), __fadd_rn(floorf(mx), r3), W, r3s.x0, r3s.x1) &
              tiles_of(__fsub_rn(ceilf(my), r3), __fadd_rn(floorf(my), r3), H, r3s.y0, r3s.y1);
    if (!ok) r3s = empty_rect();
    if (mode == QB_BIN_AABB3S) {
        out[0] = r3s;
        return rect_empty(r3s) ? 0 : 1;
    }
    if (clamp3s && rect_empty(r3s)) return 0;
    if (mode == QB_BIN_ADR) {
        Rect r;
        bool oka = tiles_of(__fsub_rn(mx, box.x), __fadd_rn(mx, box.x), W, r.x0, r.x1) &
                   tiles_of(__fsub_rn(my, box.y), __fadd_rn(my, box.y), H, r.y0, r.y1);
        if (!oka) return 0;
        out[0] = clamp3s ? intersect(r, r3s) : r;
        return rect_empty(out[0]) ? 0 : 1;
    }
    int nonempty = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        bool same = (q == 0 || q == 2);
        bool major = orient ? same : !same;
        if (mode == QB_BIN_DUALBOX && !major) continue;
        float ex = major ? box.x : box.z, ey = major ? box.y : box.w;
        bool px = (q == 0 || q == 3), py = (q == 0 || q == 1);
        float xlo = px ? mx : __fsub_rn(mx, ex), xhi = px ? __fadd_rn(mx, ex) : mx;
        float ylo = py ? my : __fsub_rn(my, ey), yhi = py ? __fadd_rn(my, ey) : my;
        Rect r;
        bool okq = tiles_of(xlo, xhi, W, r.x0, r.x1) & tiles_of(ylo, yhi, H, r.y0, r.y1);
        if (!okq) continue;
        out[q] = clamp3s ? intersect(r, r3s) : r;
        nonempty += rect_empty(out[q]) ? 0 : 1;
    }
    return nonempty;
}

// QPass (Sec. 3.2): global tile range of the sub-boxes, scan lines along its
// shorter axis; per line, min/max merge of the other-axis ranges of the
// sub-boxes whose range overlaps the line.  Returns the number of lines and
// the scan geometry; line_interval() gives a line's [lo, hi].
struct QPass {
    Rect b[4];
    int s0, s1;    // scan-line range
    bool columns;  // true: lines are tile columns (x), intervals along y
};

__device__ __forceinline__ bool qpass_setup(const Rect rects[4], QPass &qp) {
    int gx0 = 1 << 30, gy0 = 1 << 30, gx1 = -1, gy1 = -1;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        qp.b[q] = rects[q];
        if (rect_empty(rects[q])) continue;
        gx0 = min(gx0, rects[q].x0);
        gy0 = min(gy0, rects[q].y0);
        gx1 = max(gx1, rects[q].x1);
        gy1 = max(gy1, rects[q].y1);
    }
    if (gx1 < 0) return false;
    qp.columns = (gx1 - gx0) <= (gy1 - gy0);
    qp.s0 = qp.columns ? gx0 : gy0;
    qp.s1 = qp.columns ? gx1 : gy1;
    return true;
}

__device__ __forceinline__ void qpass_line(const QPass &qp, int s, int &lo, int &hi) {
    lo = 1 << 30;
    hi = -1;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const Rect &r = qp.b[q];
        int a0 = qp.columns ? r.x0 : r.y0, a1 = qp.columns ? r.x1 : r.y1;
        int o0 = qp.columns ? r.y0 : r.x0, o1 = qp.columns ? r.y1 : r.x1;
        bool hit = (s >= a0) & (s <= a1);  // empty boxes have a0 > a1
        lo = hit ? min(lo, o0) : lo;
        hi = hit ? max(hi, o1) : hi;
    }
}

// Runs of consecutive scan lines whose merged interval is the same: the
// interval of a line changes only where a sub-box's range on the scan axis
// begins or ends, so the QPass output is a union of at most 7 disjoint
// rectangles ("segments"), each visited line by line exactly as QPass does.
struct QSeg {
    int s0, lo;   // first line, first tile on the other axis
    int nl, len;  // lines in the run, interval length
};

// The runs are found in order and stored in fixed slots (so the array stays
// in registers): slot k holds the k-th run, an empty one (no sub-box overlaps
// its lines) with nl = len = 0.  The lines [s0, s1] have at most six interior
// breakpoints (each sub-box begins or ends at most once), so seven slots hold
// every run.  Returns the number of slots used.
__device__ __forceinline__ int qpass_segments(const QPass &qp, QSeg seg[7]) {
    int used = 0;
    int cur = qp.s0;
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        seg[k] = QSeg{0, 0, 0, 0};
        if (cur > qp.s1) continue;
        int next = qp.s1 + 1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const Rect &r = qp.b[q];
            if (rect_empty(r)) continue;
            const int a0 = qp.columns ? r.x0 : r.y0, a1 = qp.columns ? r.x1 : r.y1;
            if (a0 > cur) next = min(next, a0);
            if (a1 + 1 > cur) next = min(next, a1 + 1);
        }
        int lo, hi;
        qpass_line(qp, cur, lo, hi);
        if (hi >= lo) seg[k] = QSeg{cur, lo, next - cur, hi - lo + 1};
        used = k + 1;
        cur = next;
    }
    return used;
}

__device__ __forceinline__ bool seg_empty(const QSeg &g) { return g.nl <= 0 || g.len <= 0; }

__device__ __forceinline__ Rect both(const Rect &a, const Rect &b) {
    return Rect{max(a.x0, b.x0), max(a.y0, b.y0), min(a.x1, b.x1), min(a.y1, b.y1)};
}

__device__ __forceinline__ int rect_area(const Rect &r) { return max(r.x1 - r.x0 + 1, 0) * max(r.y1 - r.y0 + 1, 0); }

// Tiles (or cells) in the union of the sub-box rectangles, by inclusion and
// exclusion: what a QPass traversal counts (its merged line intervals hold no
// tile outside the union, because the sub-boxes share the corner mu^2D), in
// about 130 branch-free integer operations where the run decomposition
// (qpass_segments) takes several hundred.
__device__ __forceinline__ uint32_t union_count(const Rect r[4]) {
    const Rect r01 = both(r[0], r[1]), r02 = both(r[0], r[2]), r03 = both(r[0], r[3]);
    const Rect r12 = both(r[1], r[2]), r13 = both(r[1], r[3]), r23 = both(r[2], r[3]);
    const int one = rect_area(r[0]) + rect_area(r[1]) + rect_area(r[2]) + rect_area(r[3]);
    const int two = rect_area(r01) + rect_area(r02) + rect_area(r03) + rect_area(r12) + rect_area(r13) + rect_area(r23);
    const int three = rect_area(both(r01, r[2])) + rect_area(both(r01, r[3])) + rect_area(both(r23, r[0])) +
                      rect_area(both(r23, r[1]));
    return (uint32_t)(one - two + three - rect_area(both(r01, r23)));
}

// The depth-first path bins Gaussians into cells of kCellX x kCellY tiles
// first (qb_cells.cu): the cells a Gaussian's tiles lie in, and per cell one
// bit per tile.
constexpr int kCellXShift = 3, kCellYShift = 2;
constexpr int kCellX = 1 << kCellXShift, kCellY = 1 << kCellYShift;
static_assert(kCellX * kCellY == 32, "a cell's tiles are the bits of one word");

// The cells a tile rectangle touches.  An empty rectangle stays empty:
// intersections are stored as empty_rect() (1, 1, 0, 0), whose corners would
// meet after the shift, so it is kept apart.
__device__ __forceinline__ Rect cell_rect(const Rect &r) {
    if (rect_empty(r)) return empty_rect();
    return Rect{r.x0 >> kCellXShift, r.y0 >> kCellYShift, r.x1 >> kCellXShift, r.y1 >> kCellYShift};
}

// The tiles of rectangle r inside cell (cx, cy), bit (ty % kCellY) kCellX +
// tx % kCellX.
__device__ __forceinline__ uint32_t cell_bits_of(const Rect &r, int cx, int cy) {
    const int x0 = max(r.x0 - (cx << kCellXShift), 0), x1 = min(r.x1 - (cx << kCellXShift), kCellX - 1);
    const int y0 = max(r.y0 - (cy << kCellYShift), 0), y1 = min(r.y1 - (cy << kCellYShift), kCellY - 1);
    if (x0 > x1 || y0 > y1) return 0u;
    const uint32_t row = ((2u << (x1 - x0)) - 1u) << x0;                    // the columns of one row
    const uint32_t rows = (0x01010101u >> (kCellX * (kCellY - 1 - (y1 - y0)))) << (kCellX * y0);
    return row * rows;
}

// The cells of the bounding box of four tile rectangles (not all empty).
__device__ __forceinline__ Rect cell_box(const Rect r[4]) {
    Rect box{1 << 30, 1 << 30, -1, -1};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const bool e = rect_empty(r[q]);
        box.x0 = e ? box.x0 : min(box.x0, r[q].x0);
        box.y0 = e ? box.y0 : min(box.y0, r[q].y0);
        box.x1 = e ? box.x1 : max(box.x1, r[q].x1);
        box.y1 = e ? box.y1 : max(box.y1, r[q].y1);
    }
    return cell_rect(box);
}

// The entries that a Gaussian of `tiles` tiles gets: one per cell of its
// cells' bounding box, an eighth or so of them without a tile, which the emit
// files apart.  The few whose bounding box has more cells than they have tiles
// (two or three tiles around a corner of four cells) get one per cell that
// holds a tile, so there are never more entries than tiles.
__device__ __forceinline__ uint32_t cell_entries(const Rect r[4], uint32_t tiles) {
    if (tiles == 0u) return 0u;
    const uint32_t cells = (uint32_t)rect_area(cell_box(r));
    if (cells <= tiles) return cells;
    Rect c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = cell_rect(r[q]);
    return union_count(c);
}

// A Gaussian's four sub-box rectangles in two uint4 (tile coordinates below
// 2^16), rectangle q in words 2q (x0 | y0 << 16) and 2q + 1 (x1 | y1 << 16).
__device__ __forceinline__ void pack_rects(const Rect r[4], uint4 out[2]) {
    uint32_t w[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        w[2 * q] = (uint32_t)r[q].x0 | ((uint32_t)r[q].y0 << 16);
        w[2 * q + 1] = (uint32_t)r[q].x1 | ((uint32_t)r[q].y1 << 16);
    }
    out[0] = make_uint4(w[0], w[1], w[2], w[3]);
    out[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

__device__ __forceinline__ Rect unpack_rect(uint32_t lo, uint32_t hi) {
    return Rect{(int)(lo & 0xffffu), (int)(lo >> 16), (int)(hi & 0xffffu), (int)(hi >> 16)};
}

// Naive traversal (QuadBox-dagger, Table 3): nested loops over each
// sub-box's rectangle, skipping tiles held by an earlier sub-box.
__device__ __forceinline__ bool in_rect(const Rect &r, int tx, int ty) {
    return !rect_empty(r) && tx >= r.x0 && tx <= r.x1 && ty >= r.y0 && ty <= r.y1;
}

__device__ __forceinline__ uint32_t naive_count(const Rect r[4]) {
    uint32_t c = 0;
    for (int q = 0; q < 4; ++q) {
        if (rect_empty(r[q])) continue;
        for (int ty = r[q].y0; ty <= r[q].y1; ++ty)
            for (int tx = r[q].x0; tx <= r[q].x1; ++tx) {
                bool seen = false;
                for (int p = 0; p < q; ++p) seen |= in_rect(r[p], tx, ty);
                c += seen ? 0u : 1u;
            }
    }
    return c;
}

}  // namespace qb
