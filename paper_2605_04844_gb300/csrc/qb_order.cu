// qb_order.cu -- the emission order of the depth-first path: the Gaussians by
// (depth, index), and the exclusive scan of their tile and cell-entry counts
// in that order (K2).
//
// Up to kOrderSmall Gaussians one cluster of eight blocks does both in its
// shared memory.  Sorted pass by pass from memory, a few thousand keys cost
// the latency of eight launches (two memsets, the histogram, four passes, the
// scan): a call of 10k Gaussians at 256 x 256 took 187 us, with this kernel
// 168.  Beyond that the passes run from memory (sort_pairs,
// launch_scan_cells).
//
// The scattered stores to the other blocks bound the passes (about 0.8 us per
// key of a thread and pass) and the cluster barriers their number: a key and
// its value go in one 8-byte store, and the digit counts are pushed to all
// blocks before the barrier instead of read from them after it.  10k Gaussians
// 28.0 -> 23.9 us, 20k 38.4 -> 29.7 (with 3 keys per thread, 31.4 with 4).
#include <algorithm>

#include "qb_scan.cuh"
#include "qb_sweep.cuh"

namespace qb {

constexpr int kOrderCtas = 8;       // blocks per cluster (the portable limit)
constexpr int kOrderThreads = 1024;
constexpr int kOrderWarps = kOrderThreads / 32;
constexpr int kOrderItems = 4;      // keys per thread at most
constexpr int kOrderSmall = kOrderCtas * kOrderThreads * kOrderItems;
constexpr int kOrderDigits = 1 << kDepthDigitBits;

template <int ITEMS>
struct OrderShared {
    uint2 kv[2][kOrderThreads * ITEMS];         // (key, value)
    uint16_t whist[kOrderWarps][kOrderDigits];  // per warp: digit counts, then their prefix over the warps
    uint32_t count[kOrderCtas][kOrderDigits];   // every block's keys per digit (each block writes its own everywhere)
    uint32_t base[kOrderDigits];                // position of the block's first key of each digit
    uint64_t total[kOrderCtas][2];              // every block's tiles and cell entries
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}

// The address of p (this block's shared memory) in block `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}

__device__ __forceinline__ void st_cluster(uint32_t a, uint64_t v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

__device__ __forceinline__ void st_cluster(uint32_t a, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ void st_cluster(uint32_t a, uint32_t x, uint32_t y) {
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

// Block r of the cluster holds the positions [r share, (r + 1) share) of n,
// share a multiple of 32 and at most kOrderThreads ITEMS.  Per digit pass each
// warp ranks its contiguous keys in order (one ballot per digit bit), the
// blocks exchange their digit counts, and every key goes straight to its
// position in the shared memory of the block that holds it.
template <int ITEMS>
__global__ void __launch_bounds__(kOrderThreads) depth_order_small_kernel(OrderArgs a, int n, int share,
                                                                          uint32_t inv_share) {
    extern __shared__ __align__(16) uint8_t smem[];
    OrderShared<ITEMS> &S = *reinterpret_cast<OrderShared<ITEMS> *>(smem);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    cluster_arrive();  // (waited for before the first store to another block: it must have started)
    const uint32_t rank_cta = cluster_rank();
    const int first = (int)rank_cta * share, mine = max(0, min(share, n - first));
    const uint32_t lt = lanemask_lt();
    // item k of lane l of warp w: local position (w ITEMS + k) 32 + l
    uint32_t key[ITEMS], val[ITEMS];
    auto local = [&](int k) { return (wid * ITEMS + k) * 32 + lane; };
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = local(k);
        key[k] = i < mine ? a.keys[first + i] : 0u;
        val[k] = i < mine ? a.vals[first + i] : 0u;
    }
    const PassGeo g = pass_geo(kDepthBits, kDepthDigitBits);
    int buf = 0;
    for (int p = 0; p < g.passes; ++p) {
        const int shift = g.shift[p];
        const uint32_t mask = (1u << g.bits[p]) - 1u;
        for (int i = tid; i < kOrderWarps * kOrderDigits / 2; i += kOrderThreads)
            reinterpret_cast<uint32_t *>(S.whist)[i] = 0u;
        __syncthreads();
        uint16_t *wh = S.whist[wid];
        uint32_t rank[ITEMS];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const bool valid = local(k) < mine;
            const uint32_t d = valid ? (key[k] >> shift) & mask : (uint32_t)kOrderDigits;  // (a digit of its own)
            uint32_t peers = 0xffffffffu;
#pragma unroll
            for (int b = 0; b <= kDepthDigitBits; ++b) {
                const uint32_t bit = (d >> b) & 1u;
                const uint32_t bb = __ballot_sync(0xffffffffu, bit);
                peers &= ~(bb ^ (0u - bit));
            }
            const uint32_t pre = valid ? (uint32_t)wh[d] : 0u;
            const uint32_t lower = __popc(peers & lt);
            __syncwarp();
            if (valid && lower == 0) wh[d] = (uint16_t)(pre + __popc(peers));
            __syncwarp();
            rank[k] = pre + lower;
        }
        __syncthreads();
        {  // per digit the prefix over the warps, four threads a digit
            constexpr int kPer = kOrderWarps / 4;
            const int d = tid >> 2, q = tid & 3;
            uint32_t c[kPer], sum = 0;
#pragma unroll
            for (int w = 0; w < kPer; ++w) sum += c[w] = S.whist[q * kPer + w][d];
            uint32_t incl = sum;
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o, 4);
                if (q >= o) incl += u;
            }
            uint32_t run = incl - sum;
#pragma unroll
            for (int w = 0; w < kPer; ++w) {
                S.whist[q * kPer + w][d] = (uint16_t)run;
                run += c[w];
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 3, 4);
            if (p == 0) cluster_wait();
            for (uint32_t r = q; r < kOrderCtas; r += 4) st_cluster(cluster_addr(&S.count[rank_cta][d], r), total);
        }
        cluster_sync();
        uint32_t before = 0, all = 0;
        if (tid < kOrderDigits) {
#pragma unroll
            for (uint32_t r = 0; r < kOrderCtas; ++r) {
                const uint32_t v = S.count[r][tid];
                before += r < rank_cta ? v : 0u;
                all += v;
            }
        }
        uint32_t total;
        const uint32_t start = block_excl_scan_u32(all, &total);
        if (tid < kOrderDigits) S.base[tid] = start + before;
        __syncthreads();
        buf ^= 1;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            if (local(k) < mine) {
                const uint32_t d = (key[k] >> shift) & mask;
                const uint32_t pos = S.base[d] + S.whist[wid][d] + rank[k];
                const uint32_t r = __umulhi(pos, inv_share), i = pos - r * (uint32_t)share;
                st_cluster(cluster_addr(&S.kv[buf][i], r), key[k], val[k]);
            }
        }
        cluster_sync();
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = local(k);
            const uint2 kv = i < mine ? S.kv[buf][i] : make_uint2(0u, 0u);
            key[k] = kv.x;
            val[k] = kv.y;
        }
    }
    // the order, beside its input: keys and values stay as the preprocess wrote
    // them, so another emit of the same preprocess finds them again; from here
    // thread t takes ITEMS consecutive positions
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        if (local(k) < mine) a.vals_alt[first + local(k)] = val[k];
    const int i0 = tid * ITEMS;
    uint32_t c[ITEMS], e[ITEMS];
    uint64_t csum = 0, esum = 0;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const uint2 v = i0 + k < mine ? a.cc[S.kv[buf][i0 + k].y] : make_uint2(0u, 0u);
        c[k] = v.x;
        e[k] = v.y;
        csum += v.x;
        esum += v.y;
    }
    uint64_t ctot, etot;
    uint64_t crun = block_incl_scan<uint64_t>(csum, &ctot) - csum;
    uint64_t erun = block_incl_scan<uint64_t>(esum, &etot) - esum;
    if (tid < kOrderCtas) {
        st_cluster(cluster_addr(&S.total[rank_cta][0], (uint32_t)tid), ctot);
        st_cluster(cluster_addr(&S.total[rank_cta][1], (uint32_t)tid), etot);
    }
    cluster_sync();  // (the last access to another block's shared memory)
    uint64_t P = 0, E = 0;
#pragma unroll
    for (uint32_t r = 0; r < kOrderCtas; ++r) {
        const uint64_t x = S.total[r][0], y = S.total[r][1];
        if (r < rank_cta) crun += x, erun += y;
        P += x;
        E += y;
    }
    if (rank_cta == 0 && tid == 0) {
        *a.n_pairs = P;
        if (a.n_pairs_host) *a.n_pairs_host = P;
        *a.n_cells = P <= a.capacity && E <= a.capacity ? E : 0ull;  // (E <= P: cell_entries)
    }
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        if (i0 + k < mine) {
            const int j = first + i0 + k;
            a.offsets[j] = (uint32_t)crun;  // P <= 2^30 is checked before use
            a.coff[j] = (uint32_t)erun;
            if (e[k] > 0u) {
                const uint64_t c0 = (erun + kEmitStride - 1) / kEmitStride, c1 = (erun + e[k] - 1) / kEmitStride;
                for (uint64_t ch = c0; ch <= c1 && ch < a.chunk_cap; ++ch) a.chunk_first[ch] = (uint32_t)j;
            }
            crun += c[k];
            erun += e[k];
        }
    }
}

template <int ITEMS>
static cudaError_t launch_small(const OrderArgs &a, int n, int share, cudaStream_t s) {
    const void *f = (const void *)depth_order_small_kernel<ITEMS>;
    cudaError_t e = ensure_dyn_smem(f, sizeof(OrderShared<ITEMS>));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kOrderCtas);
    cfg.blockDim = dim3(kOrderThreads);
    cfg.dynamicSmemBytes = sizeof(OrderShared<ITEMS>);
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kOrderCtas;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    note_launch("depth_order_small_kernel", s);
    // floor(pos / share) = (pos inv) >> 32 for pos < kOrderSmall: the error is
    // below pos share / (share 2^32) < 2^-17, less than the 1 / share to the next whole number
    const uint32_t inv = (uint32_t)(((1ull << 32) + share - 1) / share);
    return cudaLaunchKernelEx(&cfg, depth_order_small_kernel<ITEMS>, a, n, share, inv);
}

cudaError_t launch_depth_order(const OrderArgs &a, int n, cudaStream_t s, bool *in_alt) {
    *in_alt = false;
    if (n > 0 && n <= kOrderSmall) {
        *in_alt = true;
        const int share = ((n + kOrderCtas - 1) / kOrderCtas + 31) & ~31;
        if (share <= kOrderThreads) return launch_small<1>(a, n, share, s);
        if (share <= 2 * kOrderThreads) return launch_small<2>(a, n, share, s);
        if (share <= 3 * kOrderThreads) return launch_small<3>(a, n, share, s);
        return launch_small<4>(a, n, share, s);
    }
    int passes = 0;
    if (n > 0) {
        cudaError_t e = sort_pairs(a.keys, a.vals, a.keys_alt, a.vals_alt, (uint64_t)n, nullptr, kDepthBits,
                                   kDepthDigitBits, a.sort_scratch, a.err, s, &passes);
        if (e != cudaSuccess) return e;
    }
    *in_alt = passes & 1;
    return launch_scan_cells(a.cc, *in_alt ? a.vals_alt : a.vals, n, a.offsets, a.coff, a.partials, a.n_pairs,
                             a.n_pairs_host, a.n_cells, a.capacity, a.err, n > 0 ? sort_failed_at(a.sort_scratch) : nullptr,
                             a.chunk_first, a.chunk_cap, s);
}

}  // namespace qb
