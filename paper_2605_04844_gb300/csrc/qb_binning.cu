// qb_binning.cu -- K2, the exclusive scan of the per-Gaussian counts, and the
// full-key path's K3, DuplicateWithKeys with QPass traversal (Sec. 2, Sec.
// 3.2), and K5, the per-tile ranges of its sorted pairs.  The depth-first
// path bins through cells of tiles (qb_cells.cu).
//
// Pairs are emitted in an "emission order" of the Gaussians: index order for
// the full-key path, depth order for the depth-first path.  The scan runs in
// that order, so each Gaussian's pairs are one contiguous run and a warp's 32
// Gaussians own one contiguous output range.
#include "qb_scan.cuh"
#include "qb_sweep.cuh"

namespace qb {

constexpr int kScanBlock = 256;
constexpr int kScanItems = 8;
constexpr int kScanChunk = kScanBlock * kScanItems;

// K2 in one pass: block b (taken in launch order from a counter, so every
// earlier block is already running) scans its kScanChunk entries, publishes
// its sums, looks back over the earlier blocks' published words for its
// running totals (decoupled look-back) and writes its offsets.
//
// DUAL (depth-first): entry j is the pair cc[perm[j]] = (tiles, cells) of the
// j-th Gaussian in depth order; offsets gets the tiles' exclusive prefix,
// coff the cells'.  Otherwise entry j is counts[j] and offsets its prefix (coff
// is not used).  chunk_first[c] becomes the position whose outputs (cell entries
// or pairs) hold output c kEmitStride, so the emit's warps find their first
// Gaussian with one load instead of a search.  The last block writes P, and for
// DUAL the number of cell entries, 0 when P exceeds the capacity (then nothing
// downstream writes).
//
// Status of a block: two 64-bit words stored and loaded as one 128-bit word,
// flag (bit 63: sum of the block, bit 62: total through the block) and a
// 62-bit count; the first word's flag holds for both.
//
// The kernel is bound by latency (gathers, look-back): 8 entries per thread
// instead of 16 give twice the blocks, and all resident blocks reach their
// look-back at about the same time, so it reads 256 words at once instead of
// 32 (a chain of two or three loads where there were up to a dozen).
//
// A look-back that runs out leaves offsets that do not belong together: the
// number of cell entries is then 0, and the full-key emit is kept from using
// them by the failure word beside the block counter.
constexpr uint64_t kScanAgg = 1ull << 63, kScanIncl = 1ull << 62, kScanCount = kScanIncl - 1;

struct ScanWord {
    uint64_t a, b;
};

__device__ __forceinline__ ScanWord ld_status(const ScanWord *p) {
    ScanWord w;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(w.a), "=l"(w.b)
                 : "l"(p)
                 : "memory");
    return w;
}

__device__ __forceinline__ void st_status(ScanWord *p, ScanWord w) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(w.a), "l"(w.b)
                 : "memory");
}

struct ScanArgs {
    const uint32_t *counts;  // !DUAL: by index
    const uint2 *cc;         // DUAL: (tiles, cells) by record
    const uint32_t *perm;    // DUAL: record of each position
    int n;
    uint32_t *offsets, *coff, *chunk_first;
    uint32_t chunk_cap;
    ScanWord *status;  // one per block, zero
    uint32_t *counter;  // block counter, then the scan's failure word (zero): set when a look-back runs out
    const uint32_t *order_failed;  // DUAL, or null: the failure word of the sort that made perm
    uint64_t *n_pairs, *n_pairs_host, *n_cells;
    uint64_t capacity;
    uint32_t *err;
};

__device__ __forceinline__ void set_cells(const ScanArgs &A, uint64_t v) {
    atomicExch(reinterpret_cast<unsigned long long *>(A.n_cells), (unsigned long long)v);
}

// A block's look-back ran out.  DUAL: the number of cell entries ends as 0,
// whichever comes later, this or the last block's writing it: each writes its
// word, fences, and then the last block reads the failure word and this one
// writes the number, so that one of the two sees the other.
template <bool DUAL>
__device__ __forceinline__ void scan_gave_up(const ScanArgs &A) {
    atomicOr(A.err, kErrTimeout);
    atomicExch(A.counter + 1, 1u);
    if (DUAL) {
        __threadfence();
        set_cells(A, 0ull);
    }
}

template <bool DUAL>
__global__ void __launch_bounds__(kScanBlock, 4) scan_onepass_kernel(ScanArgs A) {
    __shared__ uint32_t s_block, s_ready[kScanBlock / 32], s_incl[kScanBlock / 32];
    __shared__ uint64_t s_sum[kScanBlock / 32], s_sumd[kScanBlock / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) s_block = atomicAdd(A.counter, 1u);
    __syncthreads();
    const uint32_t b = s_block;
    const int n = A.n;
    // (an order with gaps is not gathered through: every count reads as zero; the
    // order itself is read meanwhile, so that its loads do not wait for this one)
    const size_t n_in = DUAL && A.order_failed && *A.order_failed ? 0 : (size_t)n;
    const int nb = (n + kScanChunk - 1) / kScanChunk;
    const size_t base = (size_t)b * kScanChunk + (size_t)tid * kScanItems;
    const bool whole = base + kScanItems <= (size_t)n;
    uint32_t c[kScanItems], d[kScanItems];  // tiles (or counts), cells
    if constexpr (DUAL) {
        uint32_t g[kScanItems];
        // 16-byte loads where perm allows them (a batch camera's order starts at a
        // multiple of n records, which need not be one of four)
        if (whole && (reinterpret_cast<uintptr_t>(A.perm) & 15) == 0) {
#pragma unroll
            for (int q = 0; q < kScanItems / 4; ++q) {
                const uint4 v = reinterpret_cast<const uint4 *>(A.perm + base)[q];
                g[4 * q] = v.x, g[4 * q + 1] = v.y, g[4 * q + 2] = v.z, g[4 * q + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < kScanItems; ++k) g[k] = base + k < (size_t)n ? A.perm[base + k] : 0u;
        }
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const uint2 v = base + k < n_in ? A.cc[g[k]] : make_uint2(0u, 0u);
            c[k] = v.x;
            d[k] = v.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            c[k] = base + k < (size_t)n ? A.counts[base + k] : 0u;
            d[k] = 0u;
        }
    }
    uint64_t csum = 0, dsum = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) csum += c[k], dsum += d[k];
    uint64_t ctot, dtot = 0, cincl, dincl = 0;
    cincl = block_incl_scan<uint64_t>(csum, &ctot);
    if (DUAL) dincl = block_incl_scan<uint64_t>(dsum, &dtot);
    // Publish, then look back over 256 earlier blocks per step: thread k reads
    // the word of block t - k, and the sums of those before the first word not
    // yet published are added, up to and including the first inclusive word,
    // which ends the walk.  (Before block 0 reads as an inclusive zero.)
    if (tid == 0) st_status(A.status + b, ScanWord{(b == 0 ? kScanIncl : kScanAgg) | ctot, dtot});
    uint64_t acc = 0, accd = 0;
    int spins = 0;
    for (int64_t t = (int64_t)b - 1; t >= 0;) {
        const int64_t mine = t - tid;
        const ScanWord w = mine >= 0 ? ld_status(A.status + mine) : ScanWord{kScanIncl, 0};
        const uint32_t ready = __ballot_sync(0xffffffffu, (w.a & (kScanAgg | kScanIncl)) != 0);
        const uint32_t inclm = __ballot_sync(0xffffffffu, (w.a & kScanIncl) != 0);
        if (lane == 0) s_ready[wid] = ready, s_incl[wid] = inclm;
        __syncthreads();
        int first_unready = kScanBlock, first_incl = kScanBlock;
#pragma unroll
        for (int k = kScanBlock / 32 - 1; k >= 0; --k) {
            if (~s_ready[k]) first_unready = 32 * k + __ffs(~s_ready[k]) - 1;
            if (s_incl[k]) first_incl = 32 * k + __ffs(s_incl[k]) - 1;
        }
        const bool ends = first_incl < first_unready;
        const int used = ends ? first_incl + 1 : first_unready;
        uint64_t v = tid < used ? (w.a & kScanCount) : 0ull, u = tid < used ? w.b : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v += __shfl_xor_sync(0xffffffffu, v, o);
            if (DUAL) u += __shfl_xor_sync(0xffffffffu, u, o);
        }
        if (lane == 0) s_sum[wid] = v, s_sumd[wid] = u;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kScanBlock / 32; ++k) acc += s_sum[k], accd += s_sumd[k];
        if (ends) break;  // the same for the whole block
        t -= used;
        if (used == 0) {  // the nearest earlier block has not published yet
            if (++spins > kSpinLimit) {
                if (tid == 0) scan_gave_up<DUAL>(A);
                break;
            }
            __nanosleep(64);
        }
    }
    if (b == 1 && (ld_relaxed(A.err + 1) & kTestScan)) {  // test-only (stall_test)
        acc = accd = 0;
        if (tid == 0) scan_gave_up<DUAL>(A);
    }
    if (tid == 0) {
        if (b > 0) st_status(A.status + b, ScanWord{kScanIncl | ((acc + ctot) & kScanCount), accd + dtot});
        if ((int)b == nb - 1) {
            const uint64_t P = acc + ctot, E = accd + dtot;
            *A.n_pairs = P;
            if (A.n_pairs_host) *A.n_pairs_host = P;
            // (E <= P: cell_entries)
            if (DUAL) {
                set_cells(A, P <= A.capacity && E <= A.capacity ? E : 0ull);
                __threadfence();  // (scan_gave_up)
                if (ld_relaxed(A.counter + 1)) set_cells(A, 0ull);
            }
        }
    }
    uint64_t run = acc + cincl - csum;
    {
        uint64_t q = DUAL ? accd + dincl - dsum : run;  // outputs of the emit: cell entries or pairs
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const uint32_t e = DUAL ? d[k] : c[k];
            if (e > 0u) {
                // the run [q, q + e) of this Gaussian holds these chunk starts
                const uint64_t c0 = (q + kEmitStride - 1) / kEmitStride, c1 = (q + e - 1) / kEmitStride;
                for (uint64_t ch = c0; ch <= c1 && ch < A.chunk_cap; ++ch) A.chunk_first[ch] = (uint32_t)(base + k);
            }
            q += e;
        }
    }
    uint32_t r = (uint32_t)(accd + dincl - dsum);
    if (whole) {
        uint32_t o[kScanItems], p[kScanItems];
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            o[k] = (uint32_t)run;  // P <= 2^30 is checked before use
            run += c[k];
            p[k] = r;
            r += d[k];
        }
#pragma unroll
        for (int q = 0; q < kScanItems / 4; ++q) {
            reinterpret_cast<uint4 *>(A.offsets + base)[q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
            if (DUAL) reinterpret_cast<uint4 *>(A.coff + base)[q] = make_uint4(p[4 * q], p[4 * q + 1], p[4 * q + 2], p[4 * q + 3]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            if (base + k < (size_t)n) {
                A.offsets[base + k] = (uint32_t)run;
                if (DUAL) A.coff[base + k] = r;
            }
            run += c[k];
            r += d[k];
        }
    }
}

// 64-bit words of scratch: the blocks' status words, then the block counter and the failure word
size_t scan_partials_count(int n) { return 2 * (size_t)((n + kScanChunk - 1) / kScanChunk) + 2; }

const uint32_t *scan_failed(const uint64_t *partials, int n) {
    if (n == 0) return nullptr;
    return reinterpret_cast<const uint32_t *>(partials + 2 * ((n + kScanChunk - 1) / kScanChunk)) + 1;
}

static cudaError_t run_scan(ScanArgs A, uint64_t *partials, bool dual, cudaStream_t s) {
    if (A.n == 0) {
        cudaError_t e = cudaMemsetAsync(A.n_pairs, 0, sizeof(uint64_t), s);
        if (e == cudaSuccess && dual) e = cudaMemsetAsync(A.n_cells, 0, sizeof(uint64_t), s);
        return e;
    }
    const int nb = (A.n + kScanChunk - 1) / kScanChunk;
    cudaError_t e = cudaMemsetAsync(partials, 0, scan_partials_count(A.n) * sizeof(uint64_t), s);
    if (e != cudaSuccess) return e;
    A.status = reinterpret_cast<ScanWord *>(partials);
    A.counter = reinterpret_cast<uint32_t *>(partials + 2 * nb);
    note_launch("scan_onepass_kernel", s);
    if (dual) scan_onepass_kernel<true><<<nb, kScanBlock, 0, s>>>(A);
    else scan_onepass_kernel<false><<<nb, kScanBlock, 0, s>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_scan(const uint32_t *counts, int n, uint32_t *offsets, uint64_t *partials,
                        uint64_t *n_pairs, uint64_t *n_pairs_host, uint32_t *err, uint32_t *chunk_first,
                        uint32_t chunk_cap, cudaStream_t s) {
    ScanArgs A{};
    A.n_pairs_host = n_pairs_host;
    A.counts = counts;
    A.n = n;
    A.offsets = offsets;
    A.chunk_first = chunk_first;
    A.chunk_cap = chunk_cap;
    A.n_pairs = n_pairs;
    A.err = err;
    return run_scan(A, partials, false, s);
}

cudaError_t launch_scan_cells(const uint2 *cc, const uint32_t *perm, int n, uint32_t *offsets, uint32_t *coff,
                              uint64_t *partials, uint64_t *n_pairs, uint64_t *n_pairs_host, uint64_t *n_cells,
                              uint64_t capacity, uint32_t *err, const uint32_t *order_failed, uint32_t *chunk_first,
                              uint32_t chunk_cap, cudaStream_t s) {
    ScanArgs A{};
    A.order_failed = order_failed;
    A.n_pairs_host = n_pairs_host;
    A.chunk_first = chunk_first;
    A.chunk_cap = chunk_cap;
    A.cc = cc;
    A.perm = perm;
    A.n = n;
    A.offsets = offsets;
    A.coff = coff;
    A.n_pairs = n_pairs;
    A.n_cells = n_cells;
    A.capacity = capacity;
    A.err = err;
    return run_scan(A, partials, true, s);
}

__device__ __forceinline__ uint64_t make_key(uint32_t tile, uint32_t dbits) {
    return ((uint64_t)tile << kDepthBits) | dbits;
}

constexpr int kEmitWarps = 4;  // warps per block (8 measured 0.7 % slower on the forward)
constexpr int kSegPerWarp = 32 * 7;
constexpr uint32_t kEmitChunk = 1024;  // output positions per warp (512, 2048, 4096 measured slower)
static_assert(kEmitChunk % kEmitStride == 0, "a warp's range starts on the scan's chunk table");

// One warp's table of QPass segments for a batch of 32 Gaussians.
struct SegTable {
    int32_t start[kSegPerWarp];  // chunk position of the segment's first pair
    uint32_t geo[kSegPerWarp];   // first line | first cell << 16
    uint32_t len[kSegPerWarp];   // cells per line | owner lane << 16 | column flag << 24
    float inv[kSegPerWarp];      // 1 / cells per line
    uint32_t gid[32], dbits[32];
};

// K3 (QPass modes and the single-box modes) for the pair positions
// [C, C + L) of the emission order, run by one warp.  It takes the Gaussian
// whose run holds position C from the scan's table, then the following ones 32 at a time:
// each lane decomposes its Gaussian's QPass traversal into segments (runs of
// scan lines with one merged interval), and the warp produces the range 32
// consecutive positions at a time; lane q finds the segment holding its
// position from a ballot of the segment starts that fall in its group.
// sink(valid, p, tile, gid, depth bits) is called by all 32 lanes together
// once per group of 32 positions; valid lanes carry position C + p.
template <class Sink>
__device__ __forceinline__ void emit_range(const EmitArgs &a, uint64_t C, int32_t L, SegTable &S, Sink &&sink) {
    const int lane = threadIdx.x & 31;
    int64_t j0 = a.chunk_first[C / kEmitStride];  // C is a multiple of the stride
    const uint32_t le_mask = lanemask_le();
    int32_t done_to = 0;  // chunk positions [0, done_to) produced
    while (done_to < L && j0 < a.n) {
        const int64_t j = j0 + lane;
        const uint32_t gid = (uint32_t)j;
        uint32_t cnt = 0;
        int64_t rel = (int64_t)1 << 40;
        if (j < a.n) {
            cnt = a.counts[j];
            rel = (int64_t)a.offsets[j] - (int64_t)C;
        }
        const bool relevant = cnt > 0u && rel < L && rel + (int64_t)cnt > 0;
        QSeg seg[7];
#pragma unroll
        for (int q = 0; q < 7; ++q) seg[q] = QSeg{0, 0, 0, 0};
        bool columns = false;
        uint32_t dbits = 0;
        if (relevant) {
            dbits = __float_as_uint(a.rgbd[gid].w) & 0x7fffffffu;
            const uint4 w0 = a.rects[2 * (size_t)gid], w1 = a.rects[2 * (size_t)gid + 1];
            const Rect r[4] = {unpack_rect(w0.x, w0.y), unpack_rect(w0.z, w0.w), unpack_rect(w1.x, w1.y),
                               unpack_rect(w1.z, w1.w)};
            QPass qp;
            if (qpass_setup(r, qp)) {
                qpass_segments(qp, seg);
                columns = qp.columns;
            }
        }
        int ns = 0;
#pragma unroll
        for (int q = 0; q < 7; ++q) ns += seg_empty(seg[q]) ? 0 : 1;
        __syncwarp();
        S.gid[lane] = gid;
        S.dbits[lane] = dbits;
        const int sincl = warp_incl_scan(ns);
        const int nseg = __shfl_sync(0xffffffffu, sincl, 31);
        int32_t r0 = (int32_t)(rel > -((int64_t)1 << 30) ? rel : -((int64_t)1 << 30));
        int k = sincl - ns;  // this lane's first table entry
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            if (seg_empty(seg[q])) continue;
            S.start[k] = r0;
            S.geo[k] = (uint32_t)seg[q].s0 | ((uint32_t)seg[q].lo << 16);
            S.len[k] = (uint32_t)seg[q].len | ((uint32_t)lane << 16) | ((uint32_t)columns << 24);
            S.inv[k] = 1.0f / (float)seg[q].len;
            r0 += seg[q].nl * seg[q].len;
            ++k;
        }
        // end of this batch's pairs within the chunk
        const int64_t last_end = __shfl_sync(0xffffffffu, rel + (int64_t)cnt, 31);
        const int32_t batch_end = (int32_t)(last_end < (int64_t)L ? last_end : (int64_t)L);
        __syncwarp();
        // cur: last segment starting at or before done_to
        int cur = -1;
        for (int b = 0; b < nseg; b += 32) {
            const bool le = b + lane < nseg && S.start[b + lane] <= done_to;
            cur += __popc(__ballot_sync(0xffffffffu, le));
        }
        for (int32_t c0 = done_to; c0 < batch_end; c0 += 32) {
            const int cand = cur + 1 + lane;
            uint32_t bit = 0u;
            if (cand < nseg) {
                const int32_t st = S.start[cand];
                if (st < c0 + 32) bit = 1u << (st - c0);
            }
            const uint32_t M = __reduce_or_sync(0xffffffffu, bit);
            const int32_t p = c0 + lane;
            const bool valid = p < batch_end;
            uint32_t tile = 0u, gid_out = 0u, dbits_out = 0u;
            if (valid) {
                const int idx = cur + __popc(M & le_mask);
                const int32_t st = S.start[idx];
                const uint32_t geo = S.geo[idx], ln = S.len[idx];
                uint32_t q, r;
                seg_divide((uint32_t)(p - st), ln & 0xffffu, S.inv[idx], q, r);
                const uint32_t line = (geo & 0xffffu) + q, u = (geo >> 16) + r;
                const bool cols = (ln >> 24) & 1u;
                const uint32_t owner = (ln >> 16) & 0xffu;
                tile = (cols ? u : line) * a.tiles_x + (cols ? line : u);
                gid_out = S.gid[owner];
                dbits_out = S.dbits[owner];
            }
            sink(valid, p, tile, gid_out, dbits_out);  // all lanes, converged
            cur += __popc(M);
        }
        done_to = max(done_to, batch_end);
        j0 += 32;
    }
}

// K3 balanced over the output: warp w owns the pair positions
// [w C, (w+1) C), so stores are contiguous across the warp and every warp
// writes at most C pairs however large the Gaussians are.
__global__ void __launch_bounds__(kEmitWarps * 32) emit_warp_kernel(EmitArgs a, uint64_t *__restrict__ keys) {
    __shared__ SegTable s_seg[kEmitWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t P = *a.n_pairs;
    const uint64_t warp_id = (uint64_t)blockIdx.x * kEmitWarps + wid;
    if (*a.failed) return;
    if (P > a.capacity) {
        if (warp_id == 0 && lane == 0) atomicOr(a.err, kErrCapacity);
        return;
    }
    const uint64_t C = warp_id * kEmitChunk;
    if (C >= P || a.n == 0) return;
    const int32_t L = (int32_t)min((uint64_t)kEmitChunk, P - C);
    uint32_t *vals = a.vals;
    emit_range(a, C, L, s_seg[wid], [&](bool valid, int32_t p, uint32_t tile, uint32_t gid, uint32_t dbits) {
        if (valid) {
            keys[C + p] = make_key(tile, dbits);
            vals[C + p] = gid;
        }
    });
}

// K3 for QuadBox-dagger (QB_BIN_QUADBOX_NAIVE, the paper's ablation without
// QPass): one thread per Gaussian runs nested loops over each sub-box and
// skips tiles an earlier sub-box already holds.
__global__ void __launch_bounds__(256) emit_naive_kernel(EmitArgs a, uint64_t *__restrict__ keys) {
    const size_t j = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= (size_t)a.n || *a.failed) return;
    if (*a.n_pairs > a.capacity) {
        if (j == 0) atomicOr(a.err, kErrCapacity);
        return;
    }
    const uint32_t gid = (uint32_t)j;
    const uint32_t c = a.counts[gid];
    if (c == 0u) return;
    const uint32_t off = a.offsets[j];
    const uint32_t dbits = __float_as_uint(a.rgbd[gid].w) & 0x7fffffffu;
    const uint4 w0 = a.rects[2 * (size_t)gid], w1 = a.rects[2 * (size_t)gid + 1];
    const Rect r[4] = {unpack_rect(w0.x, w0.y), unpack_rect(w0.z, w0.w), unpack_rect(w1.x, w1.y),
                       unpack_rect(w1.z, w1.w)};
    uint32_t k = 0;
    for (int q = 0; q < 4; ++q) {
        if (rect_empty(r[q])) continue;
        for (int ty = r[q].y0; ty <= r[q].y1; ++ty)
            for (int tx = r[q].x0; tx <= r[q].x1; ++tx) {
                bool seen = false;
                for (int p = 0; p < q; ++p) seen |= in_rect(r[p], tx, ty);
                if (seen || k >= c) continue;
                keys[off + k] = make_key((uint32_t)ty * a.tiles_x + (uint32_t)tx, dbits);
                a.vals[off + k] = gid;
                ++k;
            }
    }
}

cudaError_t launch_emit(const EmitArgs &a, uint64_t *keys, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    if (a.mode == QB_BIN_QUADBOX_NAIVE) {
        note_launch("emit_naive_kernel", s), emit_naive_kernel<<<(a.n + 255) / 256, 256, 0, s>>>(a, keys);
    } else {
        const uint64_t pairs = a.n_pairs_host != UINT64_MAX ? a.n_pairs_host : a.capacity;
        const uint64_t warps = (pairs + kEmitChunk - 1) / kEmitChunk;
        uint64_t blocks = (warps + kEmitWarps - 1) / kEmitWarps;
        if (blocks == 0) blocks = 1;  // one block still flags an overflow
        note_launch("emit_warp_kernel", s), emit_warp_kernel<<<(unsigned)blocks, kEmitWarps * 32, 0, s>>>(a, keys);
    }
    return cudaGetLastError();
}

// K5: tile boundaries of the sorted keys; ranges must be zero on entry, and
// stay so when the scan or the sort before it failed.
__device__ __forceinline__ uint32_t tile_of(uint64_t k) { return (uint32_t)(k >> kDepthBits); }

__global__ void ranges_kernel(const uint64_t *keys, uint64_t n_max, const uint64_t *n_dev, uint2 *ranges,
                              uint32_t ntiles, const uint32_t *scan_fail, const uint32_t *sort_fail) {
    if ((scan_fail && *scan_fail) || *sort_fail) return;
    uint64_t n = n_dev ? (*n_dev > n_max ? 0 : *n_dev) : n_max;  // overflow (flagged by the emit): no pairs
    for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
         idx += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t tile = tile_of(keys[idx]);
        if (tile >= ntiles) continue;  // never for keys written by the emit kernels
        if (idx == 0 || tile_of(keys[idx - 1]) != tile) ranges[tile].x = (uint32_t)idx;
        if (idx == n - 1 || tile_of(keys[idx + 1]) != tile) ranges[tile].y = (uint32_t)(idx + 1);
    }
}

cudaError_t launch_ranges(const uint64_t *keys, uint64_t n_max, const uint64_t *n_dev, uint2 *ranges, int ntiles,
                          const uint32_t *scan_fail, void *sort_scratch, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(ranges, 0, sizeof(uint2) * (size_t)ntiles, s);
    if (e != cudaSuccess || n_max == 0) return e;
    uint64_t blocks = (n_max + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    note_launch("ranges_kernel", s), ranges_kernel<<<(unsigned)blocks, 256, 0, s>>>(keys, n_max, n_dev, ranges, (uint32_t)ntiles, scan_fail, sort_failed_at(sort_scratch));
    return cudaGetLastError();
}

// The tile id of every sorted pair position, from the ranges (one block per
// tile).
// Positions at or beyond n_out are not written.
__global__ void expand_ranges_kernel(const uint2 *ranges, uint32_t ntiles, uint32_t *out, uint64_t n_out) {
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const uint2 r = ranges[t];
        const uint64_t end = r.y < n_out ? r.y : n_out;
        for (uint64_t i = (uint64_t)r.x + threadIdx.x; i < end; i += blockDim.x) out[i] = t;
    }
}

cudaError_t launch_expand_ranges(const uint2 *ranges, int ntiles, uint32_t *out, uint64_t n_out, cudaStream_t s) {
    if (ntiles <= 0 || n_out == 0) return cudaSuccess;
    note_launch("expand_ranges_kernel", s), expand_ranges_kernel<<<ntiles < 65535 ? ntiles : 65535, 256, 0, s>>>(ranges, (uint32_t)ntiles, out, n_out);
    return cudaGetLastError();
}

}  // namespace qb
