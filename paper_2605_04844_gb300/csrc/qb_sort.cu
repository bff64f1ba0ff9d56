// qb_sort.cu -- K4: stable LSD radix sort of (key, u32 value) pairs with a
// onesweep schedule (one kernel per digit pass, decoupled look-back across
// tiles of 4096 keys), the SortPairs stage of the rasteriser (Sec. 2).  The
// pass body lives in qb_sweep.cuh.
//
// Per sort: one upfront pass reads all keys and builds the digit histograms
// of every pass, and a tiny kernel turns them into exclusive bucket offsets
// (the cell sort has them from its emit).  Each digit pass then reads and writes the
// pairs once.  Pass widths are balanced (pass_geo): 13 bits at digits of 8
// bits are sorted as 7 + 6, so no pass carries buckets that are always empty.
#include <algorithm>

#include "qb_sweep.cuh"

namespace qb {

size_t sort_scratch_bytes(uint64_t n, int end_bit, int digit_bits) {
    if (digit_bits < 8 || digit_bits > kMaxDigitBits || end_bit < 1 || end_bit > 64) return 0;
    const PassGeo g = pass_geo(end_bit, digit_bits);
    if (g.passes > kMaxPasses) return 0;
    return align256(kSortHeader + (size_t)g.passes * sort_tiles(n) * ((size_t)1 << digit_bits) * 4);
}

// Upfront histogram of every pass's digit (table stride kHistStride).  With
// done (a counter, zero at launch) the last block to finish turns the counts
// into exclusive bucket offsets.
template <typename KeyT>
__global__ void __launch_bounds__(256) sort_hist_kernel(const KeyT *__restrict__ keys, uint64_t n_max,
                                                        const uint64_t *n_dev, PassGeo g, uint32_t *hist,
                                                        uint32_t *done) {
    extern __shared__ uint32_t sh[];  // passes x 2^bits[p], packed
    __shared__ bool s_last;
    int off[kMaxPasses], total = 0;  // (indexed by unrolled loops only: registers)
#pragma unroll
    for (int p = 0; p < kMaxPasses; ++p) {
        off[p] = total;
        total += p < g.passes ? 1 << g.bits[p] : 0;
    }
    for (int j = threadIdx.x; j < total; j += blockDim.x) sh[j] = 0u;
    __syncthreads();
    const uint64_t n = device_count(n_dev, n_max);
    // J keys in flight per thread, consecutive lanes reading consecutive keys.
    // (Additions of one to the same word by several lanes of a warp are one
    // operation, so a thread's runs of equal digits are not collected first; that,
    // and the pass loops unrolled instead of indexing local arrays: 5M 64-bit keys
    // 39 -> 28 us, 1M 32-bit keys 17 -> 14.)
    constexpr int J = 8;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += J * stride) {
        KeyT k[J];
#pragma unroll
        for (int j = 0; j < J; ++j) k[j] = i0 + j * stride < n ? keys[i0 + j * stride] : KeyT(0);
#pragma unroll
        for (int j = 0; j < J; ++j) {
            if (i0 + j * stride >= n) break;
#pragma unroll
            for (int p = 0; p < kMaxPasses; ++p)
                if (p < g.passes) atomicAdd(&sh[off[p] + ((uint32_t)(k[j] >> g.shift[p]) & ((1u << g.bits[p]) - 1u))], 1u);
        }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < kMaxPasses; ++p) {
        if (p >= g.passes) break;
        for (int d = threadIdx.x; d < (1 << g.bits[p]); d += blockDim.x) {
            const uint32_t v = sh[off[p] + d];
            if (v) atomicAdd(&hist[p * kHistStride + d], v);
        }
    }
    if (!done) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int p = 0; p < g.passes; ++p) {
        const int R = 1 << g.bits[p];  // <= 256 (kScanInHist)
        uint32_t *h = hist + p * kHistStride;
        const uint32_t v = threadIdx.x < R ? __ldcg(h + threadIdx.x) : 0u;
        uint32_t total;
        const uint32_t run = block_excl_scan_u32(v, &total);
        if (threadIdx.x < R) h[threadIdx.x] = run;
    }
}

// Digits of at most this many bits are scanned by the histogram's last block
// (a launch less: 14 -> 12 us at 10k keys of 8 bits); wider ones take longer in
// one block than the launch of a block per pass.
constexpr int kScanInHist = 8;

// Counts -> exclusive bucket offsets, one block per pass.
__global__ void __launch_bounds__(1024) sort_hist_scan_kernel(uint32_t *hist, PassGeo g) {
    const int R = 1 << g.bits[blockIdx.x];
    const int per = (R + 1023) / 1024;
    uint32_t *h = hist + blockIdx.x * kHistStride;
    uint32_t v[2], s = 0;  // R <= 2048
    for (int k = 0; k < 2; ++k) {
        const int idx = threadIdx.x * per + k;
        v[k] = (k < per && idx < R) ? h[idx] : 0u;
        s += v[k];
    }
    uint32_t total;
    uint32_t run = block_excl_scan_u32(s, &total);
    for (int k = 0; k < 2; ++k) {
        const int idx = threadIdx.x * per + k;
        if (k < per && idx < R) h[idx] = run;
        run += v[k];
    }
}

// One digit pass of the pair sort, ITEMS keys per thread.
template <int RB, typename KeyT, int ITEMS>
__global__ void __launch_bounds__(kSortBlock, sizeof(KeyT) == 4 ? kSortBlocksPerSM : RB <= 9 ? kSortBlocksPerSM64 : 3) onesweep_kernel(const KeyT *__restrict__ kin,
                                                              const uint32_t *__restrict__ vin,
                                                              KeyT *__restrict__ kout, uint32_t *__restrict__ vout,
                                                              uint64_t n_max, const uint64_t *n_dev,
                                                              const uint32_t *__restrict__ bin_off,
                                                              uint32_t *lookback, uint32_t *counter, int shift,
                                                              uint32_t mask, uint32_t *err, uint32_t *failed) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_tile;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) s_tile = atomicAdd(counter, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint32_t n = (uint32_t)device_count(n_dev, n_max);  // <= 2^30
    const uint32_t tbase = tile * (uint32_t)(kSortBlock * ITEMS);
    if (tbase >= n) return;  // block-uniform

    // warp-striped load: item k of lane l at wbase + 32k + l; the values are
    // read only at the scatter, after the ranking
    const uint32_t wbase = tbase + (uint32_t)wid * (32 * ITEMS);
    KeyT key[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const uint32_t idx = wbase + 32 * k + lane;
        key[k] = idx < n ? __ldcs(kin + idx) : KeyT(0);
    }
    auto val = [&](int k) -> uint32_t { return __ldcs(vin + wbase + 32 * k + lane); };
    sweep_tile<RB, KeyT, uint32_t, true, ITEMS>(key, val, n, tbase, tile, bin_off, lookback, shift, mask, err, failed,
                                                kout, vout, smem);
}

template <int RB, typename KeyT, int ITEMS>
static cudaError_t launch_pass_t(const KeyT *kin, const uint32_t *vin, KeyT *kout, uint32_t *vout, uint64_t n_max,
                                 const uint64_t *n_dev, const uint32_t *bin_off, uint32_t *lookback,
                                 uint32_t *counter, int shift, uint32_t mask, uint32_t *err, uint32_t *failed,
                                 cudaStream_t s) {
    constexpr size_t smem = sweep_smem<RB, KeyT, uint32_t, ITEMS>();
    cudaError_t e = ensure_dyn_smem((const void *)onesweep_kernel<RB, KeyT, ITEMS>, smem);
    if (e != cudaSuccess) return e;
    note_launch("onesweep_kernel", s), onesweep_kernel<RB, KeyT, ITEMS><<<(unsigned)((n_max + kSortBlock * ITEMS - 1) / (kSortBlock * ITEMS)), kSortBlock, smem, s>>>(
        kin, vin, kout, vout, n_max, n_dev, bin_off, lookback, counter, shift, mask, err, failed);
    return cudaGetLastError();
}

// One pass on the digit bits [shift, shift + bits), bits <= 11.
template <typename KeyT>
static cudaError_t launch_pass(const KeyT *kin, const uint32_t *vin, KeyT *kout, uint32_t *vout, uint64_t n_max,
                               const uint64_t *n_dev, const uint32_t *bin_off, uint32_t *lookback,
                               uint32_t *counter, int shift, int bits, uint32_t *err, uint32_t *failed, int items,
                               cudaStream_t s) {
    const uint32_t mask = (1u << bits) - 1u;
#define QB_PASS_RUN(RB, ITEMS)                                                                                     \
    launch_pass_t<RB, KeyT, ITEMS>(kin, vin, kout, vout, n_max, n_dev, bin_off, lookback, counter, shift, mask, err,   \
                                   failed, s)
#define QB_PASS_CASE(RB)                                                                                           \
    case RB:                                                                                                       \
        if constexpr (sizeof(KeyT) == 4 && RB >= 7 && RB <= 8) {                                                   \
            if (items == 4) return QB_PASS_RUN(RB, 4);                                                             \
            if (items == 8) return QB_PASS_RUN(RB, 8);                                                             \
        }                                                                                                          \
        return QB_PASS_RUN(RB, kSortItems);
    switch (bits < 4 ? 4 : bits) {
        QB_PASS_CASE(4)
        QB_PASS_CASE(5)
        QB_PASS_CASE(6)
        QB_PASS_CASE(7)
        QB_PASS_CASE(8)
        QB_PASS_CASE(9)
        QB_PASS_CASE(10)
        QB_PASS_CASE(11)
    default: return cudaErrorInvalidValue;
    }
#undef QB_PASS_CASE
#undef QB_PASS_RUN
}

// Keys per thread of the depth order's passes (32-bit keys, digits of 7 and 8
// bits; its scratch is sized for it, depth_sort_scratch_bytes).  A pass over a
// short sort is bound by the latency of one block's chain (load, count, rank
// 16 rows in turn, look back, scatter) at a third of the warps an SM holds,
// so short sorts take fewer keys per thread and more blocks.  Four passes with 4,
// 8, 16 keys per thread: 10k keys 34, 38, 50 us; 200k 51, 48, 57; 1M 92, 79,
// 73 (there the look-back over twice the tiles costs more).
static int sort_items_u32(uint64_t n) { return n <= (1ull << 16) ? 4 : n <= 3ull << 18 ? 8 : kSortItems; }

size_t depth_sort_scratch_bytes(uint64_t n) {
    const uint64_t tile = (uint64_t)kSortBlock * sort_items_u32(n);
    const PassGeo g = pass_geo(kDepthBits, kDepthDigitBits);
    return align256(kSortHeader + (size_t)g.passes * ((n + tile - 1) / tile) * ((size_t)1 << kDepthDigitBits) * 4);
}

template <typename KeyT>
static cudaError_t sort_impl(KeyT *keys, uint32_t *vals, KeyT *keys_alt, uint32_t *vals_alt, uint64_t n_max,
                             const uint64_t *n_dev, int end_bit, int digit_bits, void *scratch, uint32_t *err,
                             cudaStream_t s, int *passes_out) {
    if (end_bit > (int)(8 * sizeof(KeyT)) || digit_bits < 8 || digit_bits > kMaxDigitBits) return cudaErrorInvalidValue;
    const PassGeo g = pass_geo(end_bit, digit_bits);
    if (g.passes > kMaxPasses) return cudaErrorInvalidValue;
    uint32_t *hist = sort_hist_at(scratch);
    *passes_out = g.passes;
    const int items = sizeof(KeyT) == 4 ? sort_items_u32(n_max) : kSortItems;
    const uint64_t tiles = (n_max + (uint64_t)kSortBlock * items - 1) / ((uint64_t)kSortBlock * items);
    const size_t pass_words = tiles * ((size_t)1 << digit_bits);
    // the table, the counters and the look-back words are adjacent
    cudaError_t e = cudaMemsetAsync(scratch, 0, kSortHeader + (size_t)g.passes * pass_words * 4, s);
    if (e != cudaSuccess || n_max == 0) return e;

    e = ensure_dyn_smem((const void *)sort_hist_kernel<KeyT>, (size_t)kMaxPasses * kHistStride * 4);
    if (e != cudaSuccess) return e;
    size_t smem = 0;
    for (int p = 0; p < g.passes; ++p) smem += (size_t)4 << g.bits[p];
    uint64_t hblocks = std::min<uint64_t>((n_max + 8 * 256 - 1) / (8 * 256), 152 * 4);
    const bool in_hist = g.bits[0] <= kScanInHist;  // (the first pass is the widest)
    note_launch("sort_hist_kernel", s), sort_hist_kernel<KeyT><<<(unsigned)hblocks, 256, smem, s>>>(
        keys, n_max, n_dev, g, hist, in_hist ? sort_counter_at(scratch, kMaxPasses) : nullptr);
    if (!in_hist) note_launch("sort_hist_scan_kernel", s), sort_hist_scan_kernel<<<g.passes, 1024, 0, s>>>(hist, g);
    KeyT *kin = keys, *kout = keys_alt;
    uint32_t *vin = vals, *vout = vals_alt;
    for (int p = 0; p < g.passes; ++p) {
        e = launch_pass<KeyT>(kin, vin, kout, vout, n_max, n_dev, hist + p * kHistStride,
                              sort_lookback_at(scratch, 0, digit_bits, 0) + p * pass_words,
                              sort_counter_at(scratch, p), g.shift[p], g.bits[p], err, sort_failed_at(scratch), items, s);
        if (e != cudaSuccess) return e;
        std::swap(kin, kout);
        std::swap(vin, vout);
    }
    return cudaSuccess;
}

cudaError_t sort_pairs(uint64_t *keys, uint32_t *vals, uint64_t *keys_alt, uint32_t *vals_alt, uint64_t n_max,
                       const uint64_t *n_dev, int end_bit, int digit_bits, void *scratch, uint32_t *err,
                       cudaStream_t s, int *passes_out) {
    return sort_impl(keys, vals, keys_alt, vals_alt, n_max, n_dev, end_bit, digit_bits, scratch, err, s, passes_out);
}

cudaError_t sort_pairs(uint32_t *keys, uint32_t *vals, uint32_t *keys_alt, uint32_t *vals_alt, uint64_t n_max,
                       const uint64_t *n_dev, int end_bit, int digit_bits, void *scratch, uint32_t *err,
                       cudaStream_t s, int *passes_out) {
    return sort_impl(keys, vals, keys_alt, vals_alt, n_max, n_dev, end_bit, digit_bits, scratch, err, s, passes_out);
}

// One digit pass of the cell sort: 32-bit cell ids with 64-bit values.  The
// number of entries is known on the device only and is a small part of the
// capacity, so resident blocks take tiles from the counter until none is
// left, instead of one block per tile of the capacity.
constexpr int kCellSortBlocksPerSM = 4;
template <int RB, bool WRITE_KEYS>
__global__ void __launch_bounds__(kSortBlock, RB <= 8 ? kCellSortBlocksPerSM : 2) cell_sort_kernel(
    const uint32_t *__restrict__ kin, const uint64_t *__restrict__ vin, uint32_t *__restrict__ kout,
    uint64_t *__restrict__ vout, const uint64_t *n_dev, const uint32_t *__restrict__ bin_off, uint32_t *lookback,
    uint32_t *counter, int shift, uint32_t mask, uint32_t *err, uint32_t *failed) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_tile;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t n = (uint32_t)*n_dev;  // <= 2^30
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        const uint64_t tbase64 = (uint64_t)tile * kSortTile;
        if (tbase64 >= n) return;  // block-uniform
        const uint32_t tbase = (uint32_t)tbase64;
        const uint32_t wbase = tbase + (uint32_t)wid * (32 * kSortItems);
        uint32_t key[kSortItems];
#pragma unroll
        for (int k = 0; k < kSortItems; ++k) {
            const uint32_t idx = wbase + 32 * k + lane;
            key[k] = idx < n ? __ldcs(kin + idx) : 0u;
        }
        auto val = [&](int k) -> uint64_t { return __ldcs(vin + wbase + 32 * k + lane); };
        sweep_tile<RB, uint32_t, uint64_t, WRITE_KEYS, kSortItems>(key, val, n, tbase, tile, bin_off, lookback, shift, mask, err,
                                                       failed, kout, vout, smem);
        __syncthreads();  // shared memory is taken again
    }
}

template <int RB, bool WRITE_KEYS>
static cudaError_t launch_cell_pass(const CellBin &b, int p, const uint32_t *kin, const uint64_t *vin, uint32_t *kout,
                                    uint64_t *vout, cudaStream_t s) {
    constexpr size_t smem = sweep_smem<RB, uint32_t, uint64_t, kSortItems>();
    cudaError_t e = ensure_dyn_smem((const void *)cell_sort_kernel<RB, WRITE_KEYS>, smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t resident = (uint64_t)sms * (RB <= 8 ? kCellSortBlocksPerSM : 2);
    const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>(sort_tiles(b.n_cells_max), resident));
    const int bits = b.geo.passes.bits[p];
    note_launch(WRITE_KEYS ? "cell_sort_pass" : "cell_sort_pass_values", s),
        cell_sort_kernel<RB, WRITE_KEYS><<<(unsigned)blocks, kSortBlock, smem, s>>>(
            kin, vin, kout, vout, b.n_cells, sort_hist_at(b.sort_scratch) + p * kHistStride,
            sort_lookback_at(b.sort_scratch, b.capacity, b.geo.digit_bits, p), sort_counter_at(b.sort_scratch, p),
            b.geo.passes.shift[p], (1u << bits) - 1u, b.err, sort_failed_at(b.sort_scratch));
    return cudaGetLastError();
}

cudaError_t cell_sort_passes(const CellBin &b, cudaStream_t s, bool *in_b) {
    const PassGeo &g = b.geo.passes;
    *in_b = g.passes & 1;
    uint32_t *kin = b.arr.keys_a, *kout = b.arr.keys_b;
    uint64_t *vin = b.arr.vals_a, *vout = b.arr.vals_b;
    for (int p = 0; p < g.passes; ++p) {
        const bool last = p + 1 == g.passes;
        cudaError_t e = cudaErrorInvalidValue;
#define QB_CELL_CASE(RB)                                                                   \
    case RB:                                                                               \
        e = last ? launch_cell_pass<RB, false>(b, p, kin, vin, kout, vout, s)              \
                 : launch_cell_pass<RB, true>(b, p, kin, vin, kout, vout, s);              \
        break;
        switch (g.bits[p] < 4 ? 4 : g.bits[p]) {
            QB_CELL_CASE(4)
            QB_CELL_CASE(5)
            QB_CELL_CASE(6)
            QB_CELL_CASE(7)
            QB_CELL_CASE(8)
            QB_CELL_CASE(9)
            QB_CELL_CASE(10)
            QB_CELL_CASE(11)
        default: break;
        }
#undef QB_CELL_CASE
        if (e != cudaSuccess) return e;
        std::swap(kin, kout);
        std::swap(vin, vout);
    }
    return cudaSuccess;
}

}  // namespace qb
