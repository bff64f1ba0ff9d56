// qb_render.cu -- K6: tile-parallel front-to-back compositing (Sec. 2
// "Render", Eq. 2), as one block per tile (single frame) or as a persistent
// kernel whose warps take half tiles of several cameras from a global work
// queue.
//
// A warp renders one half of a tile (rows 0-7 or 8-15) on its own; a thread
// owns four pixels of one column of the half, rows r, r + 2, r + 4 and r + 6,
// evaluated as two packed pairs (r, r + 2) and (r + 4, r + 6) that share the
// column's dx terms.  The warp walks the tile's depth-sorted Gaussian list 32
// entries at a time: each lane brings in one entry's record (asynchronous
// copies of the next 32 run during the walk of the current ones), tests its
// alpha ellipse against the half's 16 x 8 pixels (ellipse_meets_rect), and
// the entries that reach it are written, compacted, to the warp's staging
// memory.  An entry left out is one every pixel of the half would reject.
// Per entry and pixel (3DGS conventions):
//   power = -(a dx^2 + 2 b dx dy + c dy^2)/2, skip if it is so low that alpha
//   is certainly below 1/255 (power > 0 arises only as a float32 rounding of
//   0 and is kept);
//   alpha = min(0.99, o e^power), skip if alpha < 1/255;
//   T' = T (1 - alpha); stop before adding once T' < 1e-4;
//   C += alpha T c; T = T'.
// Each pair is evaluated with the packed FP32x2 instructions (fma/mul/add
// .f32x2); each packed lane rounds exactly like the scalar operation it
// replaces.  A warp ends as soon as all of its pixels have stopped.
//
// The kernel is bound by issue slots (and by the ALU pipe's compares and
// selects).  Against a two-warp block that staged 128 entries behind
// barriers and walked the set bits of a mask, a warp of its own needs no
// barrier, ends with its own pixels, and its compacted list has no bit scan:
// 1M Gaussians at 1080p 229 -> 181 us, 3M at 1440p seen from inside 1034 ->
// 911, 1M at 2160p 816 -> 653, 16 views of 1M (persistent) 3340 -> 2670; with
// the ellipse test of elongated Gaussians too (qb_internal.cuh; in index order)
// 174, 485, 578 and 2140.
// Measured slower: 64 registers (32 warps per SM, spills), two entries'
// exponents ahead of both blends, the next entry's operands loaded ahead
// (+21 %), T chosen by a select instead of multiplied by 1 - 0, a blend of the
// pair of rows that an entry reaches alone (where most reach both).
#include "qb_stage.cuh"

namespace qb {

constexpr int kRenderThreads = 64;  // a block of the single-frame kernel: the two halves of a tile
constexpr int kRenderPairs = 2;     // packed pixel pairs per thread

// The compositing state of one packed pair of pixels.  A pixel outside the
// image, or one that has stopped, carries a NaN row npy: its exponent and its
// alpha are then NaN and fail every test.
struct RenderPair {
    float2 T, cr, cg, cb, npy;
    int last0, last1;
    int n0, n1;  // the counted variant only
};

// Both pixels of a pair are composited in lock step.  An entry a pixel
// rejects (or a pixel that has stopped) takes weight 0, which leaves its
// colour and transmittance bit-for-bit unchanged, so the branch-free update
// composes exactly the entries the per-pixel rules of the header accept.
// (alpha >= 1/255 implies power >= skip, so the power test needs no second look.)
template <bool CAP, bool COUNT>
__device__ __forceinline__ void blend(RenderPair (&P)[kRenderPairs], const float2 (&pw)[kRenderPairs], float2 op,
                                      float2 cr, float2 cg, float2 cb, int nj) {
    float2 al[kRenderPairs], tT[kRenderPairs];
#pragma unroll
    for (int r = 0; r < kRenderPairs; ++r) {
        RenderPair &q = P[r];
        al[r] = __fmul2_rn(op, exp2_of(pw[r]));
        if (CAP) al[r] = f2(min_nan(kAlphaMax, al[r].x), min_nan(kAlphaMax, al[r].y));
        const bool ok0 = al[r].x >= kAlphaMin, ok1 = al[r].y >= kAlphaMin;
        // T (1 - alpha); fma(alpha, -1, 1) is 1 - alpha rounded once
        tT[r] = __fmul2_rn(q.T, __ffma2_rn(al[r], f2(-1.f, -1.f), f2(1.f, 1.f)));
        const bool ac0 = ok0 && tT[r].x >= kTStop, ac1 = ok1 && tT[r].y >= kTStop;
        // alpha of the accepted entries, 0 elsewhere: T (1 - 0) = T and
        // c + r * 0 = c exactly, so the updates need no select
        const float2 aa = f2(ac0 ? al[r].x : 0.f, ac1 ? al[r].y : 0.f);
        const float2 w = __fmul2_rn(aa, q.T);
        q.cr = __ffma2_rn(cr, w, q.cr);
        q.cg = __ffma2_rn(cg, w, q.cg);
        q.cb = __ffma2_rn(cb, w, q.cb);
        q.T = __fmul2_rn(q.T, __ffma2_rn(aa, f2(-1.f, -1.f), f2(1.f, 1.f)));
        q.last0 = ac0 ? nj : q.last0;
        q.last1 = ac1 ? nj : q.last1;
    }
    // Once in a pixel's life an accepted alpha takes T below the stop: its row
    // becomes NaN.  One minimum over the four pixels tells (a NaN loses against
    // any number in fminf); which of them stopped is looked at only then.
    if (fminf(fminf(tT[0].x, tT[0].y), fminf(tT[1].x, tT[1].y)) < kTStop) {
#pragma unroll
        for (int r = 0; r < kRenderPairs; ++r) {
            const bool st0 = al[r].x >= kAlphaMin && tT[r].x < kTStop, st1 = al[r].y >= kAlphaMin && tT[r].y < kTStop;
            if (st0) P[r].npy.x = kNaN;
            if (st1) P[r].npy.y = kNaN;
            if (COUNT && st0) P[r].n0 = nj;
            if (COUNT && st1) P[r].n1 = nj;
        }
    }
}

// One half (0: rows 0-7, 1: rows 8-15) of a tile by one warp; returns the
// largest last-contributor count of the lane's pixels.  COUNT (measurement
// only) also adds the half's (pixel, entry) evaluations and the evaluations
// whose power test passed to a.counts[0], a.counts[1].
template <bool COUNT = false>
__device__ __forceinline__ int render_half(const RenderArgs &a, uint32_t gtile, int half, const CamTile &C,
                                           RenderStage &S) {
    const uint32_t lt = gtile - C.tile_base;
    const int tx = (int)(lt % (uint32_t)C.tiles_x), ty = (int)(lt / (uint32_t)C.tiles_x);
    const int lane = threadIdx.x & 31;
    const int px = tx * kTile + (lane & (kTile - 1));
    const int pyb = ty * kTile + half * 8 + (lane >> kTileShift);
    const float2 npx = f2(-(float)px, -(float)px);
    // the half's pixels, for the ellipse test
    const float x0 = (float)(tx * kTile), y0 = (float)(ty * kTile + half * 8);
    RenderPair P[kRenderPairs];
#pragma unroll
    for (int r = 0; r < kRenderPairs; ++r) {
        const int ya = pyb + 4 * r, yb = ya + 2;
        P[r].npy = f2(px < C.W && ya < C.H ? -(float)ya : kNaN, px < C.W && yb < C.H ? -(float)yb : kNaN);
        P[r].T = f2(1.f, 1.f);
        P[r].cr = P[r].cg = P[r].cb = f2(0.f, 0.f);
        P[r].last0 = P[r].last1 = P[r].n0 = P[r].n1 = 0;
    }
    auto stopped = [](float npy) { return npy != npy; };
    auto all_done = [&]() {
        return stopped(P[0].npy.x) && stopped(P[0].npy.y) && stopped(P[1].npy.x) && stopped(P[1].npy.y);
    };

    const uint2 range = a.ranges[gtile];
    const int total = (int)(range.y - range.x);
    const uint32_t *vals = a.vals + C.vals_base + range.x;
    const StageSource src{a.xy, a.shape, a.conic_o, a.rgbd};
    uint32_t npass = 0;  // COUNT only
    if (lane < total) stage_copy(S, src, C.rec_base + vals[lane], lane);
    uint32_t vnext = 32 + lane < total ? vals[32 + lane] : 0u;

    for (int base = 0; base < total; base += 32) {
        copy_wait();
        const int cnt = stage_entries<false>(S, base + lane < total, base + lane + 1, x0, y0, lane);
        if (base + 32 + lane < total) {
            stage_copy(S, src, C.rec_base + vnext, lane);
            vnext = base + 64 + lane < total ? vals[base + 64 + lane] : 0u;
        }
        __syncwarp();
#pragma unroll 2
        for (int j = 0; j < cnt; ++j) {
            const float4 X = S.sx[j], Q = S.sq[j], K = S.sk[j];
            const uint32_t info = __float_as_uint(K.w);
            const float2 dx = __fadd2_rn(f2(X.x, X.y), npx);
            float2 pw[kRenderPairs];
            if (!(info & kLongEntry)) {
                // power = A + dy (B + cc dy), A = ca dx^2, B = cb dx; dx, A and
                // B are the column's, shared by the thread's four pixels
                const float2 A = __fmul2_rn(__fmul2_rn(f2(Q.x, Q.y), dx), dx);
                const float2 B = __fmul2_rn(f2(Q.z, Q.w), dx);
#pragma unroll
                for (int r = 0; r < kRenderPairs; ++r) {
                    const float2 dy = __fadd2_rn(f2(X.z, X.w), P[r].npy);
                    pw[r] = __ffma2_rn(dy, __ffma2_rn(f2(K.x, K.y), dy, B), A);
                }
            } else {
                // elongated (the same for the whole warp): power = ca u^2 +
                // ce dy^2, u = dx + rr dy
                const float4 E = S.se[j];
#pragma unroll
                for (int r = 0; r < kRenderPairs; ++r) {
                    const float2 dy = __fadd2_rn(f2(X.z, X.w), P[r].npy);
                    const float2 u = __ffma2_rn(f2(E.x, E.y), dy, dx);
                    pw[r] = __ffma2_rn(__fmul2_rn(f2(Q.x, Q.y), u), u, __fmul2_rn(__fmul2_rn(f2(E.z, E.w), dy), dy));
                }
            }
            // power >= skip for some pixel; the rule power <= 0 needs no test: a
            // positive exponent is a float32 rounding of 0 (the conic is
            // positive definite), where alpha = o e^power rounds like o.
            // (A NaN loses against any number in fmaxf.)
            const bool any = fmaxf(fmaxf(pw[0].x, pw[0].y), fmaxf(pw[1].x, pw[1].y)) >= K.z;
            if (COUNT)
                npass += (uint32_t)(pw[0].x >= K.z) + (uint32_t)(pw[0].y >= K.z) + (uint32_t)(pw[1].x >= K.z) +
                         (uint32_t)(pw[1].y >= K.z);
            if (!__any_sync(0xffffffffu, any)) continue;
            const float4 C1 = S.s1[j], C2 = S.s2[j];
            // o G can reach the 0.99 cap only for o near it (G <= 1 up to the
            // exponential's rounding); the same for the whole warp
            if (!(info & kSlowEntry))
                blend<false, COUNT>(P, pw, f2(C1.x, C1.y), f2(C1.z, C1.w), f2(C2.x, C2.y), f2(C2.z, C2.w), (int)info);
            else
                blend<true, COUNT>(P, pw, f2(C1.x, C1.y), f2(C1.z, C1.w), f2(C2.x, C2.y), f2(C2.z, C2.w),
                                   (int)(info & ~(kSlowEntry | kLongEntry)));
        }
        if (__all_sync(0xffffffffu, all_done())) break;
    }
    copy_wait();  // the staging memory is the warp's next tile's
    const size_t plane = (size_t)C.W * C.H;
    float *img = a.img + 3 * C.pix_base;
    unsigned long long ev = 0;
#pragma unroll
    for (int r = 0; r < kRenderPairs; ++r) {
        RenderPair &q = P[r];
        // a pixel that never stopped evaluated the whole list
        if (COUNT && !stopped(q.npy.x)) q.n0 = total;
        if (COUNT && !stopped(q.npy.y)) q.n1 = total;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int py = pyb + 4 * r + 2 * h;
            if (px >= C.W || py >= C.H) continue;
            const size_t pix = (size_t)py * C.W + px;
            const float T = h ? q.T.y : q.T.x;
            img[pix] = fmaf(T, a.bg[0], h ? q.cr.y : q.cr.x);
            img[plane + pix] = fmaf(T, a.bg[1], h ? q.cg.y : q.cg.x);
            img[2 * plane + pix] = fmaf(T, a.bg[2], h ? q.cb.y : q.cb.x);
            a.tfinal[C.pix_base + pix] = T;
            a.ncontrib[C.pix_base + pix] = h ? q.last1 : q.last0;
            if (COUNT) {
                a.neval[C.pix_base + pix] = h ? q.n1 : q.n0;
                ev += (unsigned long long)(h ? q.n1 : q.n0);
            }
        }
    }
    if (COUNT) {
        unsigned long long ps = npass;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ev += __shfl_xor_sync(0xffffffffu, ev, o);
            ps += __shfl_xor_sync(0xffffffffu, ps, o);
        }
        if (lane == 0) {
            atomicAdd(a.counts, ev);
            atomicAdd(a.counts + 1, ps);
        }
    }
    return max(max(P[0].last0, P[0].last1), max(P[1].last0, P[1].last1));
}

// One block per tile of a single camera, a warp per half (72 registers, 14
// blocks per SM; unbounded the compiler takes 77, 12 blocks); with an order, the
// blocks (which start roughly in index order) take the heaviest tiles first,
// so that the last blocks to start are short ones.
template <bool COUNT>
__global__ void __launch_bounds__(kRenderThreads, COUNT ? 1 : 14) render_kernel(RenderArgs a) {
    __shared__ RenderStage s_stage[2];
    __shared__ int s_last[2];
    const int wid = threadIdx.x >> 5;
    const uint32_t t = a.order.cnt ? order_pick(a.order, a.ts.total_tiles, blockIdx.x) : (uint32_t)blockIdx.x;
    const int last = render_half<COUNT>(a, t, wid, a.ts.cam[0], s_stage[wid]);
    if (a.order_out.cnt) {
        // the tile's largest last-contributor count (the backward walks that
        // many entries) files it for the backward
        const int m = __reduce_max_sync(0xffffffffu, last);
        if ((threadIdx.x & 31) == 0) s_last[wid] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            const uint32_t walked = (uint32_t)max(s_last[0], s_last[1]);
            order_file(a.order_out, a.ts.total_tiles, t, walked);
            if (a.order_known.cnt) order_file(a.order_known, a.ts.total_tiles, t, walked);
        }
    }
}

// A warp per tile walks the tile's list 32 entries at a time for two sample
// pixels (offsets (3, 4) and (12, 11); four measured the same render and a
// third more here): each lane takes one entry's
// 1 - alpha at each pixel (the render's accept rules on the plain conic
// form), a product scan over the lanes gives the transmittance after every
// entry, and the first entry that takes a pixel below the stop ends that
// pixel.  The estimate is the largest stop position, or the list length when
// a pixel has not stopped within kWorkChunks chunks.  The next chunk's
// records and the one after's indices are loaded while a chunk is scanned.
constexpr int kWorkPix = 2;  // sample pixels per tile, at these offsets in the tile
__device__ constexpr int kWorkX[kWorkPix] = {3, 12};
__device__ constexpr int kWorkY[kWorkPix] = {4, 11};
constexpr uint32_t kWorkChunks = 32;  // beyond 1024 entries every tile files into the top bucket
__global__ void __launch_bounds__(256) tile_work_kernel(RenderArgs a) {
    const int lane = threadIdx.x & 31;
    const uint32_t t = blockIdx.x * 8u + (threadIdx.x >> 5);
    if (t >= a.ts.total_tiles) return;  // warp-uniform
    const CamTile &C = a.ts.cam[0];
    const int tx = (int)(t % (uint32_t)C.tiles_x), ty = (int)(t / (uint32_t)C.tiles_x);
    float sx[kWorkPix], sy[kWorkPix], T[kWorkPix];
    bool done[kWorkPix];
#pragma unroll
    for (int k = 0; k < kWorkPix; ++k) {
        const int x = tx * kTile + kWorkX[k], y = ty * kTile + kWorkY[k];
        sx[k] = (float)x;
        sy[k] = (float)y;
        T[k] = 1.f;
        done[k] = x >= C.W || y >= C.H;
    }
    const uint2 range = a.ranges[t];
    const uint32_t total = range.y - range.x;
    const uint32_t *vals = a.vals + range.x;
    // records of chunk 0, indices of chunk 1
    float2 m = make_float2(0.f, 0.f);
    float4 co = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lane < total) {
        const uint32_t g = vals[lane];
        m = a.xy[g];
        co = a.conic_o[g];
    }
    uint32_t gn = 32 + lane < total ? vals[32 + lane] : 0u;
    uint32_t work = 0;
    bool open = true;
    for (uint32_t c = 0; c < kWorkChunks && 32 * c < total; ++c) {
        const uint32_t base = 32 * c;
        const bool have = base + lane < total;
        const float2 mc = m;
        const float4 cc = co;
        if (base + 32 + lane < total) {  // prefetch: records of chunk c + 1, indices of chunk c + 2
            m = a.xy[gn];
            co = a.conic_o[gn];
            gn = base + 64 + lane < total ? vals[base + 64 + lane] : 0u;
        }
        float om[kWorkPix];
#pragma unroll
        for (int k = 0; k < kWorkPix; ++k) om[k] = 1.f;
        if (have) {
            const float skip = skip_threshold(cc.w);
#pragma unroll
            for (int k = 0; k < kWorkPix; ++k) {
                const float dx = mc.x - sx[k], dy = mc.y - sy[k];
                const float pw = -0.5f * (cc.x * dx * dx + cc.z * dy * dy) - cc.y * dx * dy;
                if (pw >= skip) {
                    const float al = fminf(kAlphaMax, cc.w * __expf(pw));
                    if (al >= kAlphaMin) om[k] = 1.f - al;
                }
            }
        }
        bool all = true;
#pragma unroll
        for (int k = 0; k < kWorkPix; ++k) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float v = __shfl_up_sync(0xffffffffu, om[k], o);
                if (lane >= o) om[k] *= v;
            }
            const float Tl = T[k] * om[k];
            const uint32_t stop = __ballot_sync(0xffffffffu, Tl < kTStop);
            if (!done[k] && stop) {
                done[k] = true;
                work = max(work, base + (uint32_t)__ffs(stop));
            }
            T[k] = __shfl_sync(0xffffffffu, Tl, 31);
            all = all && done[k];
        }
        if (all) {
            open = false;
            break;
        }
    }
    if (open) {
        bool any_open = false;
#pragma unroll
        for (int k = 0; k < kWorkPix; ++k) any_open = any_open || !done[k];
        if (any_open) work = total;
    }
    if (lane == 0) order_file(a.order, a.ts.total_tiles, t, work);
}

cudaError_t launch_tile_work(const RenderArgs &a, cudaStream_t s) {
    if (a.ts.total_tiles == 0) return cudaSuccess;
    note_launch("tile_work_kernel", s), tile_work_kernel<<<(a.ts.total_tiles + 7) / 8, 256, 0, s>>>(a);
    return cudaGetLastError();
}

// Persistent warps take the halves of tiles_per_fetch consecutive tiles at a
// time from a global counter over the tiles of all cameras in the set.
__global__ void __launch_bounds__(kRenderThreads) render_persistent_kernel(RenderArgs a) {
    __shared__ RenderStage s_stage[2];
    RenderStage &S = s_stage[threadIdx.x >> 5];
    const uint32_t halves = 2u * a.ts.total_tiles, take = 2u * (uint32_t)a.tiles_per_fetch;
    for (;;) {
        uint32_t h0 = 0;
        if ((threadIdx.x & 31) == 0) h0 = atomicAdd(a.queue, take);
        h0 = __shfl_sync(0xffffffffu, h0, 0);
        if (h0 >= halves) break;
        const uint32_t h1 = min(h0 + take, halves);
        for (uint32_t h = h0; h < h1; ++h) {
            const uint32_t t = h >> 1;
            const CamTile C = a.cam_table[camera_in_table(a.cam_table, a.ts.n_cams, t)];
            render_half(a, t, (int)(h & 1u), C, S);
        }
    }
}

cudaError_t launch_render(const RenderArgs &a, cudaStream_t s) {
    if (a.ts.total_tiles == 0) return cudaSuccess;
    if (a.queue) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, render_persistent_kernel, kRenderThreads, 0);
        if (a.blocks_per_sm > 0 && a.blocks_per_sm < per_sm) per_sm = a.blocks_per_sm;
        note_launch("render_persistent_kernel", s), render_persistent_kernel<<<sms * (per_sm > 0 ? per_sm : 1), kRenderThreads, 0, s>>>(a);
    } else if (a.counts) {
        note_launch("render_kernel_counted", s), render_kernel<true><<<a.ts.total_tiles, kRenderThreads, 0, s>>>(a);
    } else {
        note_launch("render_kernel", s), render_kernel<false><<<a.ts.total_tiles, kRenderThreads, 0, s>>>(a);
    }
    return cudaGetLastError();
}

}  // namespace qb
