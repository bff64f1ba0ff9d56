// qb_render.cu -- K6: tile-parallel front-to-back compositing (Sec. 2
// "Render", Eq. 2), as one block per tile (single frame) or as a persistent
// kernel whose warps take half tiles of several cameras from a global work
// queue.
//
// A warp renders one half of a tile (rows 0-7 or 8-15) on its own; a thread
// owns four pixels of one column of the half, rows r, r + 2, r + 4 and r + 6,
// evaluated as two packed pairs (r, r + 2) and (r + 4, r + 6) that share the
// column's dx terms.  (In a frame of few tiles a warp renders a quarter, a
// thread one pair.)  The warp walks the tile's depth-sorted Gaussian list 32
// entries at a time: each lane brings in one entry's record (asynchronous
// copies of the next 32 run during the walk of the current ones), tests its
// alpha ellipse against the part's pixels (ellipse_meets_rect), and
// the entries that reach it are written, compacted, to the warp's staging
// memory.  An entry left out is one every pixel of the part would reject.
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

constexpr int kRenderThreads = 64;             // the two halves of a tile
constexpr uint32_t kQuarterBlocksPerSM = 8;    // blocks of four quarters, by registers

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
template <bool CAP, bool COUNT, int PAIRS>
__device__ __forceinline__ void blend(RenderPair (&P)[PAIRS], const float2 (&pw)[PAIRS], float2 op, float2 cr,
                                      float2 cg, float2 cb, int nj) {
    float2 al[PAIRS], tT[PAIRS];
#pragma unroll
    for (int r = 0; r < PAIRS; ++r) {
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
    // becomes NaN.  One minimum over the thread's pixels tells (a NaN loses
    // against any number in fminf); which of them stopped is looked at only then.
    float low = fminf(tT[0].x, tT[0].y);
#pragma unroll
    for (int r = 1; r < PAIRS; ++r) low = fminf(low, fminf(tT[r].x, tT[r].y));
    if (low < kTStop) {
#pragma unroll
        for (int r = 0; r < PAIRS; ++r) {
            const bool st0 = al[r].x >= kAlphaMin && tT[r].x < kTStop, st1 = al[r].y >= kAlphaMin && tT[r].y < kTStop;
            if (st0) P[r].npy.x = kNaN;
            if (st1) P[r].npy.y = kNaN;
            if (COUNT && st0) P[r].n0 = nj;
            if (COUNT && st1) P[r].n1 = nj;
        }
    }
}

// One part of a tile (16 x 4 PAIRS pixels: a half of two pairs per thread, or
// a quarter of one) by one warp; returns the largest last-contributor count of
// the lane's pixels.  COUNT (measurement only) also adds the part's (pixel,
// entry) evaluations and the evaluations whose power test passed to
// a.counts[0], a.counts[1].
template <int PAIRS, bool COUNT = false>
__device__ __forceinline__ int render_part(const RenderArgs &a, uint32_t gtile, int part, const CamTile &C,
                                           RenderStage &S) {
    constexpr int kRows = 4 * PAIRS;
    const uint32_t lt = gtile - C.tile_base;
    const int tx = (int)(lt % (uint32_t)C.tiles_x), ty = (int)(lt / (uint32_t)C.tiles_x);
    const int lane = threadIdx.x & 31;
    const int px = tx * kTile + (lane & (kTile - 1));
    const int pyb = ty * kTile + part * kRows + (lane >> kTileShift);
    const float2 npx = f2(-(float)px, -(float)px);
    // the part's pixels, for the ellipse test
    const float x0 = (float)(tx * kTile), y0 = (float)(ty * kTile + part * kRows);
    RenderPair P[PAIRS];
#pragma unroll
    for (int r = 0; r < PAIRS; ++r) {
        const int ya = pyb + 4 * r, yb = ya + 2;
        P[r].npy = f2(px < C.W && ya < C.H ? -(float)ya : kNaN, px < C.W && yb < C.H ? -(float)yb : kNaN);
        P[r].T = f2(1.f, 1.f);
        P[r].cr = P[r].cg = P[r].cb = f2(0.f, 0.f);
        P[r].last0 = P[r].last1 = P[r].n0 = P[r].n1 = 0;
    }
    auto stopped = [](float npy) { return npy != npy; };
    auto all_done = [&]() {
        bool d = true;
#pragma unroll
        for (int r = 0; r < PAIRS; ++r) d = d && stopped(P[r].npy.x) && stopped(P[r].npy.y);
        return d;
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
        const int cnt = stage_entries<false, kRows, COUNT>(S, base + lane < total, base + lane + 1, x0, y0, lane);
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
            float2 pw[PAIRS];
            if (!(info & kLongEntry)) {
                // power = A + dy (B + cc dy), A = ca dx^2, B = cb dx; dx, A and
                // B are the column's, shared by the thread's pixels
                const float2 A = __fmul2_rn(__fmul2_rn(f2(Q.x, Q.y), dx), dx);
                const float2 B = __fmul2_rn(f2(Q.z, Q.w), dx);
#pragma unroll
                for (int r = 0; r < PAIRS; ++r) {
                    const float2 dy = __fadd2_rn(f2(X.z, X.w), P[r].npy);
                    pw[r] = __ffma2_rn(dy, __ffma2_rn(f2(K.x, K.y), dy, B), A);
                }
            } else {
                // elongated (the same for the whole warp): power = ca u^2 +
                // ce dy^2, u = dx + rr dy
                const float4 E = S.se[j];
#pragma unroll
                for (int r = 0; r < PAIRS; ++r) {
                    const float2 dy = __fadd2_rn(f2(X.z, X.w), P[r].npy);
                    const float2 u = __ffma2_rn(f2(E.x, E.y), dy, dx);
                    pw[r] = __ffma2_rn(__fmul2_rn(f2(Q.x, Q.y), u), u, __fmul2_rn(__fmul2_rn(f2(E.z, E.w), dy), dy));
                }
            }
            // power >= skip for some pixel; the rule power <= 0 needs no test: a
            // positive exponent is a float32 rounding of 0 (the conic is
            // positive definite), where alpha = o e^power rounds like o.
            // (A NaN loses against any number in fmaxf.)
            float high = fmaxf(pw[0].x, pw[0].y);
#pragma unroll
            for (int r = 1; r < PAIRS; ++r) high = fmaxf(high, fmaxf(pw[r].x, pw[r].y));
            if (COUNT) {
#pragma unroll
                for (int r = 0; r < PAIRS; ++r) npass += (uint32_t)(pw[r].x >= K.z) + (uint32_t)(pw[r].y >= K.z);
            }
            if (!__any_sync(0xffffffffu, high >= K.z)) continue;
            const float4 C1 = S.s1[j], C2 = S.s2[j];
            // o G can reach the 0.99 cap only for o near it (G <= 1 up to the
            // exponential's rounding); the same for the whole warp
            if (!(info & kSlowEntry))
                blend<false, COUNT, PAIRS>(P, pw, f2(C1.x, C1.y), f2(C1.z, C1.w), f2(C2.x, C2.y), f2(C2.z, C2.w), (int)info);
            else
                blend<true, COUNT, PAIRS>(P, pw, f2(C1.x, C1.y), f2(C1.z, C1.w), f2(C2.x, C2.y), f2(C2.z, C2.w),
                                   (int)(info & ~(kSlowEntry | kLongEntry)));
        }
        if (__all_sync(0xffffffffu, all_done())) break;
    }
    copy_wait();  // the staging memory is the warp's next tile's
    const size_t plane = (size_t)C.W * C.H;
    float *img = a.img + 3 * C.pix_base;
    unsigned long long ev = 0;
#pragma unroll
    for (int r = 0; r < PAIRS; ++r) {
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
    int last = 0;
#pragma unroll
    for (int r = 0; r < PAIRS; ++r) last = max(last, max(P[r].last0, P[r].last1));
    return last;
}

// One block per tile of a single camera.  PAIRS 2: a warp per half, 72
// registers, 14 blocks per SM (unbounded the compiler takes 77, 12 blocks).
// PAIRS 1: a warp per quarter, 64 registers, 8 blocks of four warps per SM.
//
// Quarters are for frames whose blocks are all resident at once (at most
// kQuarterBlocksPerSM tiles per SM): such a frame lasts as long as its longest
// warp, and a quarter's walk is shorter, by the entries that miss it and by
// half the work per entry.  Halves against quarters, Gaussians: 10k at 256^2
// (256 tiles) 28 : 23 us, 20k at 333 x 217 (294) 52 : 42, 50k at 400^2 (625)
// 73 : 55, at 512^2 (1024) 64 : 56, 100k at 640 x 480 (1200) 69 : 65; beyond,
// the doubled staging costs more: 100k at 800 x 600 (1900 tiles) 78 : 83, 200k
// at 1001 x 701 (2772) 99 : 110, 500k at 1264 x 832 (4108) 101 : 126.
// Tiles run in index order.  Heaviest first by an estimate of the work was no
// faster on any frame, estimate included (100k at 800 x 600 83 : 78 us, 200k
// 96 : 99, 500k 103 : 101, 1M at 1080p 201 : 196).  order_out files the tiles
// by the work there was, for the backward.
template <int PAIRS, bool COUNT>
__global__ void __launch_bounds__(2 * kRenderThreads / PAIRS, COUNT ? 1 : PAIRS == 1 ? (int)kQuarterBlocksPerSM : 14) render_kernel(RenderArgs a) {
    constexpr int kParts = 4 / PAIRS;
    __shared__ RenderStage s_stage[kParts];
    __shared__ int s_last[kParts];
    const int wid = threadIdx.x >> 5;
    const uint32_t t = blockIdx.x;
    const int last = render_part<PAIRS, COUNT>(a, t, wid, a.ts.cam[0], s_stage[wid]);
    if (a.order_out[0].cnt) {
        // the tile's largest last-contributor count (the backward walks that
        // many entries) files it for the backward
        const int m = __reduce_max_sync(0xffffffffu, last);
        if ((threadIdx.x & 31) == 0) s_last[wid] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t walked = 0;
#pragma unroll
            for (int k = 0; k < kParts; ++k) walked = max(walked, (uint32_t)s_last[k]);
            order_file(a.order_out[0], a.ts.total_tiles, t, walked);
            order_file(a.order_out[1], a.ts.total_tiles, t, walked);
        }
    }
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
            render_part<2>(a, t, (int)(h & 1u), C, S);
        }
    }
}

cudaError_t launch_render(const RenderArgs &a, cudaStream_t s) {
    if (a.ts.total_tiles == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (a.queue) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, render_persistent_kernel, kRenderThreads, 0);
        if (a.blocks_per_sm > 0 && a.blocks_per_sm < per_sm) per_sm = a.blocks_per_sm;
        note_launch("render_persistent_kernel", s), render_persistent_kernel<<<sms * (per_sm > 0 ? per_sm : 1), kRenderThreads, 0, s>>>(a);
    } else if (a.counts) {
        note_launch("render_kernel_counted", s), render_kernel<2, true><<<a.ts.total_tiles, kRenderThreads, 0, s>>>(a);
    } else if (a.ts.total_tiles <= kQuarterBlocksPerSM * (uint32_t)sms) {
        note_launch("render_kernel", s), render_kernel<1, false><<<a.ts.total_tiles, 2 * kRenderThreads, 0, s>>>(a);
    } else {
        note_launch("render_kernel", s), render_kernel<2, false><<<a.ts.total_tiles, kRenderThreads, 0, s>>>(a);
    }
    return cudaGetLastError();
}

}  // namespace qb
