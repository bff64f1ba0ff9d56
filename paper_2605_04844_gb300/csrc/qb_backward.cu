// qb_backward.cu -- K7 render backward and K8 preprocess backward of the
// differentiable rasteriser (Sec. 4.1 states the rasteriser is differentiable;
// the gradients below differentiate Eq. 2 and the Sec. 2 projection).
//
// K7: a warp per half tile (16 x 8 pixels, four pixels of a column per lane,
// rows r, r+2, r+4, r+6 of the half, evaluated as two pairs with the packed
// FP32x2 instructions) walks the tile list in reverse, from the largest
// last-contributor position of its own pixels down to 0, staging the entries
// that reach its pixels like the forward (qb_stage.cuh); the blocks take the
// tiles by decreasing walk length, the order the forward render filed.  Each
// pixel recomputes alpha exactly as the forward did and the transmittance by
// division,
// T_k = T_{k+1} / (1 - alpha_k); with B_k = sum_{i>k} T_i alpha_i c_i + T_final bg
// the colour behind entry k,
//   dC/dc_k     = T_k alpha_k
//   dC/dalpha_k = T_k c_k - B_k / (1 - alpha_k)
// and B enters dL/dalpha only through S2 = sum_c dL/dC_c B_c, which is carried
// per pixel instead of B.  alpha = min(0.99, o G), G = exp(power): zero
// derivative where the cap binds.
// The 9 per-Gaussian sums (mu_x, mu_y, Sigma11, Sigma12, Sigma22, o, r, g, b;
// the covariance entries are the well-conditioned parametrisation, with
// dL/dLambda = -Sigma dL/dSigma Sigma) are summed over the warp three entries
// at a time: every lane puts its 9 values in a row of shared memory each, and
// 27 lanes then sum a row of 32 with eight 16-byte loads and add it to its
// float64 accumulator: 19 instructions per entry where a 12-shuffle transpose
// reduction with its selects took about 70.  (The chain to the scale and
// rotation of a thin Gaussian amplifies the rounding of these sums, so they
// keep the order of the butterfly.)  The same routine serves one block per tile
// and a persistent kernel over several cameras.
//
// The kernel is bound by latency between dependent packed operations at 20
// warps per SM (96 registers; issue 65 %, FMA pipe 52 %).  1M Gaussians at
// 1080p 461 -> 357 us, 5 views of 200k (persistent) 2023 -> 1710 (with the
// ellipse test of elongated Gaussians 326 and 1530); 80 or 88
// registers (12 or 11 blocks per SM) measured 3 to 6 % slower.
//
// K8: one thread per Gaussian with any nonzero sum chains the (mu^2D, Sigma2D, o, colour)
// gradients of every camera of the set to means, (log-)scales, quaternions,
// opacity (logits) and SH, summing over cameras in registers.
#include "qb_project.cuh"
#include "qb_stage.cuh"

namespace qb {

constexpr int kBwdThreads = 64;  // a block of the single-frame kernel: the two halves of a tile

// float -> double by rebuilding the IEEE-754 bit pattern with integer
// operations (exponent rebias 127 -> 1023, mantissa 23 -> 52 bits), so the
// float64 atomics below need no float64 arithmetic in the SM; float32
// subnormals (|v| < 1.2e-38) become zero.
__device__ __forceinline__ double widen(float v) {
    const uint32_t u = __float_as_uint(v);
    const uint32_t e = (u >> 23) & 0xffu;
    if (e == 0u) return 0.0;
    const uint64_t bits = ((uint64_t)(u & 0x80000000u) << 32) | ((uint64_t)(e + 896u) << 52) |
                          ((uint64_t)(u & 0x7fffffu) << 29);
    return __longlong_as_double((long long)bits);
}

// 1 / x for x in [0.01, 1].
__device__ __forceinline__ float reciprocal(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The warp sums of up to kRedEntries entries: row 9 e + i holds, per lane, value
// i of the e-th waiting entry.  Rows of 36 floats put the 16-byte loads of
// eight neighbouring lanes (each summing a row of its own) on distinct banks.
constexpr int kRedEntries = 3, kRedStride = 36;
struct BwdStage {
    RenderStage in;
    float red[9 * kRedEntries * kRedStride];
    uint32_t ids[32];             // record of each staged entry
    uint32_t red_id[kRedEntries];  // record of each waiting entry
};

// Adds the waiting entries' sums to the accumulators (all lanes; the rows and
// ids are written by then up to a warp synchronisation, done here).  The
// staged values carry the sign and factor that are applied to the sums here:
// -1 for 0..4 and 6..8, and 1/2 for the squares 2 and 4.
__device__ __forceinline__ void bwd_flush(const BwdStage &S, int waiting, double *g_screen, int lane) {
    __syncwarp();
    if (lane < 9 * waiting) {
        const float4 *row = reinterpret_cast<const float4 *>(S.red + lane * kRedStride);
        // lanes l and l + 16, then l and l + 8, + 4, + 2, + 1: the tree of a
        // butterfly over the warp
        float2 v[16];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float4 q = row[k];
            v[2 * k] = f2(q.x, q.y);
            v[2 * k + 1] = f2(q.z, q.w);
        }
#pragma unroll
        for (int d = 8; d > 0; d >>= 1)
#pragma unroll
            for (int k = 0; k < d; ++k) v[k] = __fadd2_rn(v[k], v[k + d]);
        const float2 s = v[0];
        const int e = lane / 9, i = lane - 9 * e;
        const float z = (s.x + s.y) * (i == 5 ? 1.f : i == 2 || i == 4 ? -0.5f : -1.f);
        if (z != 0.f) atomicAdd(g_screen + (size_t)S.red_id[e] * 9 + i, widen(z));
    }
    __syncwarp();
}

// The per-pixel state of a pair of pixels (one packed lane each): the
// transmittance in front of the current entry, T; -S2 with
// S2 = sum_c dL/dC_c B_c (the colour behind the entry, B_c, only enters the
// gradient through this sum, which is updated as S2 += w S1 when an entry of
// weight w = alpha T is passed); and dL/dC per channel.  npy is kFar until the
// walk reaches the 32 entries that hold the pixel's last contributor: at that
// distance the exponent is hugely negative and every term finite.
constexpr float kFar = 1e15f;
struct BwdPair {
    float2 T, nS2, g0, g1, g2, npy;
    int last0, last1;
};

// Operands of an entry that all pixels of a column share.
struct BwdEntry {
    float2 dx, cadx2, B, cb;       // dx; 2 ca dx, cb dx, cb
    float2 no, cr, cg, cbl;        // -opacity, colour
};

// One entry for the thread's four pixels: updates their state and returns
// their summed contributions (each pair's two pixels packed) in X.  An entry a
// pixel does not composite takes alpha = 0 (T, S2 unchanged, no contribution),
// so the pairs run in lock step without branches.  CAP: the entry may meet
// the 0.99 cap; LONG: vx, vy come from the exact form.
//   T <- T / (1 - alpha)                       (T in front of the entry)
//   dL/dc_k     += alpha T dL/dC
//   dL/dalpha    = T S1 - S2 / (1 - alpha),    S1 = sum_c dL/dC_c c_k,c
//   S2          += alpha T S1
// and, where the opacity cap does not bind (o G < 0.99), with
// v = -dpower/dmu = (2 ca dx + cb dy, cb dx + 2 cc dy):
//   dL/do += G dL/dalpha, dpower = o G dL/dalpha,
//   dL/dmu += dpower v, dL/dSigma += dpower (vx^2/2, vx vy, vy^2/2).
// X0..X4 and X6..X8 come with the opposite sign, X2 and X4 without the 1/2
// (bwd_flush).
template <bool CAP>
__device__ __forceinline__ bool bwd_entry(BwdPair (&P)[2], const float2 (&pw)[2], const float2 (&vx)[2],
                                          const float2 (&vy)[2], const BwdEntry &E, int nj, float2 (&X)[9]) {
    bool contrib = false;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        BwdPair &q = P[r];
        const float2 G = exp2_of(pw[r]);
        const float2 noG = __fmul2_rn(E.no, G);  // -o G
        bool c0, c1;
        float2 na, Gm;
        if constexpr (CAP) {
            const float a0 = min_nan(kAlphaMax, -noG.x), a1 = min_nan(kAlphaMax, -noG.y);
            c0 = nj <= q.last0 && a0 >= kAlphaMin;
            c1 = nj <= q.last1 && a1 >= kAlphaMin;
            na = f2(c0 ? -a0 : 0.f, c1 ? -a1 : 0.f);
            // derivative through o G where the cap does not bind
            Gm = f2(c0 && -noG.x < kAlphaMax ? G.x : 0.f, c1 && -noG.y < kAlphaMax ? G.y : 0.f);
        } else {
            c0 = nj <= q.last0 && noG.x <= -kAlphaMin;
            c1 = nj <= q.last1 && noG.y <= -kAlphaMin;
            Gm = f2(c0 ? G.x : 0.f, c1 ? G.y : 0.f);
            na = __fmul2_rn(E.no, Gm);  // -alpha of the composited, 0 elsewhere
        }
        contrib = contrib || c0 || c1;
        const float2 om = __fadd2_rn(f2(1.f, 1.f), na);  // 1 - alpha (1 where not composited)
        const float2 inv = f2(reciprocal(om.x), reciprocal(om.y));  // exactly 1 where om is
        q.T = __fmul2_rn(q.T, inv);
        const float2 nw = __fmul2_rn(na, q.T);  // -alpha T
        const float2 S1 = __ffma2_rn(q.g0, E.cr, __ffma2_rn(q.g1, E.cg, __fmul2_rn(q.g2, E.cbl)));
        const float2 dal = __ffma2_rn(inv, q.nS2, __fmul2_rn(q.T, S1));
        q.nS2 = __ffma2_rn(nw, S1, q.nS2);
        // -dpower; o Gm is alpha where the cap does not bind
        const float2 ndp = __fmul2_rn(dal, CAP ? __fmul2_rn(E.no, Gm) : na);
        const float2 dpvx = __fmul2_rn(ndp, vx[r]), dpvy = __fmul2_rn(ndp, vy[r]);
        if (r == 0) {
            X[0] = dpvx;
            X[1] = dpvy;
            X[2] = __fmul2_rn(dpvx, vx[r]);
            X[3] = __fmul2_rn(dpvx, vy[r]);
            X[4] = __fmul2_rn(dpvy, vy[r]);
            X[5] = __fmul2_rn(Gm, dal);
            X[6] = __fmul2_rn(nw, q.g0);
            X[7] = __fmul2_rn(nw, q.g1);
            X[8] = __fmul2_rn(nw, q.g2);
        } else {
            X[0] = __fadd2_rn(X[0], dpvx);
            X[1] = __fadd2_rn(X[1], dpvy);
            X[2] = __ffma2_rn(dpvx, vx[r], X[2]);
            X[3] = __ffma2_rn(dpvx, vy[r], X[3]);
            X[4] = __ffma2_rn(dpvy, vy[r], X[4]);
            X[5] = __ffma2_rn(Gm, dal, X[5]);
            X[6] = __ffma2_rn(nw, q.g0, X[6]);
            X[7] = __ffma2_rn(nw, q.g1, X[7]);
            X[8] = __ffma2_rn(nw, q.g2, X[8]);
        }
    }
    return contrib;
}

// One half (0: rows 0-7, 1: rows 8-15) of a tile by one warp.
__device__ __forceinline__ void render_bwd_half(const BwdArgs &a, uint32_t gtile, int half, const CamTile &C,
                                                BwdStage &S) {
    const uint32_t lt = gtile - C.tile_base;
    const int tx = (int)(lt % (uint32_t)C.tiles_x), ty = (int)(lt / (uint32_t)C.tiles_x);
    const int lane = threadIdx.x & 31;
    const int px = tx * kTile + (lane & (kTile - 1));
    const int py_first = ty * kTile + half * 8 + (lane >> kTileShift);
    const float2 npx = f2(-(float)px, -(float)px);
    const float x0 = (float)(tx * kTile), y0 = (float)(ty * kTile + half * 8);
    const size_t plane = (size_t)C.W * C.H;
    const float *dl = a.dL_dimg + 3 * C.pix_base;

    BwdPair P[2];
    int mylast = 0;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int py = py_first + 2 * h;
        float T = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f;
        int last = 0;
        if (px < C.W && py < C.H) {
            const size_t pix = (size_t)py * C.W + px;
            T = a.tfinal[C.pix_base + pix];
            last = a.ncontrib[C.pix_base + pix];
            g0 = dl[pix];
            g1 = dl[plane + pix];
            g2 = dl[2 * plane + pix];
        }
        // the colour behind the last entry is the background seen through T
        const float nS2 = -(g0 * (T * a.bg[0]) + g1 * (T * a.bg[1]) + g2 * (T * a.bg[2]));
        BwdPair &q = P[h >> 1];
        if (h & 1) {
            q.T.y = T, q.nS2.y = nS2, q.g0.y = g0, q.g1.y = g1, q.g2.y = g2, q.last1 = last;
        } else {
            q.T.x = T, q.nS2.x = nS2, q.g0.x = g0, q.g1.x = g1, q.g2.x = g2, q.last0 = last;
        }
        mylast = max(mylast, last);
    }
    const int maxlast = __reduce_max_sync(0xffffffffu, mylast);
    if (maxlast == 0) return;
    const uint32_t *vals = a.vals + C.vals_base + a.ranges[gtile].x;
    const StageSource src{a.xy, a.shape, a.conic_o, a.rgbd};
    // lane l takes position end - 1 - l of the 32 entries before `end`, so the
    // staged entries run from the back to the front
    uint32_t rec = 0u, vnext = 0u;
    if (lane < maxlast) {
        rec = C.rec_base + vals[maxlast - 1 - lane];
        stage_copy(S.in, src, rec, lane);
    }
    if (lane + 32 < maxlast) vnext = vals[maxlast - 33 - lane];
    int waiting = 0;  // entries in S.red

    for (int end = maxlast; end > 0; end -= 32) {
        copy_wait();
        const int cnt = stage_entries<true>(S.in, lane < end, end - lane, x0, y0, lane, rec, S.ids);
        if (lane + 32 < end) {
            rec = C.rec_base + vnext;
            stage_copy(S.in, src, rec, lane);
            if (lane + 64 < end) vnext = vals[end - 65 - lane];
        }
        // pixels whose last contributor lies before these entries stay out
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int py = py_first + 4 * r;
            P[r].npy = f2(P[r].last0 > end - 32 ? -(float)py : kFar, P[r].last1 > end - 32 ? -(float)(py + 2) : kFar);
        }
        __syncwarp();
        for (int j = 0; j < cnt; ++j) {
            const float4 X4 = S.in.sx[j], Q = S.in.sq[j], K = S.in.sk[j];
            const uint32_t info = __float_as_uint(K.w);
            BwdEntry E;
            E.dx = __fadd2_rn(f2(X4.x, X4.y), npx);
            const float2 ca = f2(Q.x, Q.y), cc = f2(K.x, K.y);
            float2 dy[2], pw[2], vx[2], vy[2];
            if (!(info & kLongEntry)) {
                const float2 cadx = __fmul2_rn(ca, E.dx);
                const float2 A = __fmul2_rn(cadx, E.dx);
                E.cb = f2(Q.z, Q.w);
                E.B = __fmul2_rn(E.cb, E.dx);
                E.cadx2 = __fadd2_rn(cadx, cadx);
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    dy[r] = __fadd2_rn(f2(X4.z, X4.w), P[r].npy);
                    pw[r] = __ffma2_rn(dy[r], __ffma2_rn(cc, dy[r], E.B), A);
                }
            } else {
                // the forward's exact power form (the same operations)
                const float4 L = S.in.se[j];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    dy[r] = __fadd2_rn(f2(X4.z, X4.w), P[r].npy);
                    const float2 u = __ffma2_rn(f2(L.x, L.y), dy[r], E.dx);
                    vx[r] = __fmul2_rn(ca, u);
                    pw[r] = __ffma2_rn(vx[r], u, __fmul2_rn(__fmul2_rn(f2(L.z, L.w), dy[r]), dy[r]));
                }
            }
            // the forward's power test
            const bool any = fmaxf(fmaxf(pw[0].x, pw[0].y), fmaxf(pw[1].x, pw[1].y)) >= K.z;
            if (!__any_sync(0xffffffffu, any)) continue;
            // v = -dpower/dmu: (2 ca dx + cb dy, cb dx + 2 cc dy), or in the
            // exact form (2 ca u, 2 ca u rr + 2 ce dy), which does not cancel
            if (!(info & kLongEntry)) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    vx[r] = __ffma2_rn(E.cb, dy[r], E.cadx2);
                    vy[r] = __ffma2_rn(f2(2.f, 2.f), __fmul2_rn(cc, dy[r]), E.B);
                }
            } else {
                const float4 L = S.in.se[j];
                const float2 ce2 = f2(L.z + L.z, L.w + L.w);
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    vx[r] = __fadd2_rn(vx[r], vx[r]);
                    vy[r] = __ffma2_rn(vx[r], f2(L.x, L.y), __fmul2_rn(ce2, dy[r]));
                }
            }
            const float4 C1 = S.in.s1[j], C2 = S.in.s2[j];
            E.no = f2(C1.x, C1.y), E.cr = f2(C1.z, C1.w), E.cg = f2(C2.x, C2.y), E.cbl = f2(C2.z, C2.w);
            float2 X[9];
            bool contrib;
            if (!(info & kSlowEntry)) contrib = bwd_entry<false>(P, pw, vx, vy, E, (int)info, X);
            else contrib = bwd_entry<true>(P, pw, vx, vy, E, (int)(info & ~(kSlowEntry | kLongEntry)), X);
            if (__any_sync(0xffffffffu, contrib)) {
                float *row = S.red + 9 * waiting * kRedStride + lane;
#pragma unroll
                for (int i = 0; i < 9; ++i) row[i * kRedStride] = X[i].x + X[i].y;
                if (lane == 0) S.red_id[waiting] = S.ids[j];
                if (++waiting == kRedEntries) {
                    bwd_flush(S, waiting, a.g_screen, lane);
                    waiting = 0;
                }
            }
        }
    }
    if (waiting > 0) bwd_flush(S, waiting, a.g_screen, lane);
    copy_wait();
    __syncwarp();
}

// One block per tile; with an order, the heaviest tiles first.
__global__ void __launch_bounds__(kBwdThreads) render_bwd_kernel(BwdArgs a) {
    __shared__ __align__(16) BwdStage s_stage[2];
    const int wid = threadIdx.x >> 5;
    const uint32_t t = a.order.cnt ? order_pick(a.order, a.ts.total_tiles, blockIdx.x) : (uint32_t)blockIdx.x;
    render_bwd_half(a, t, wid, a.ts.cam[0], s_stage[wid]);
}

// Persistent warps take the halves of tiles_per_fetch consecutive tiles at a
// time from a global counter over the tiles of all cameras in the set.  (At
// most 104 registers: unbounded the compiler takes 112, nine blocks per SM
// instead of ten, 4 % slower.)
__global__ void __maxnreg__(104) render_bwd_persistent_kernel(BwdArgs a) {
    __shared__ __align__(16) BwdStage s_stage[2];
    BwdStage &S = s_stage[threadIdx.x >> 5];
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
            render_bwd_half(a, t, (int)(h & 1u), C, S);
        }
    }
}

cudaError_t launch_render_bwd(const BwdArgs &a, cudaStream_t s) {
    if (a.ts.total_tiles == 0) return cudaSuccess;
    if (a.queue) {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, render_bwd_persistent_kernel, kBwdThreads, 0);
        if (a.blocks_per_sm > 0 && a.blocks_per_sm < per_sm) per_sm = a.blocks_per_sm;
        note_launch("render_bwd_persistent_kernel", s), render_bwd_persistent_kernel<<<sms * (per_sm > 0 ? per_sm : 1), kBwdThreads, 0, s>>>(a);
    } else {
        note_launch("render_bwd_kernel", s), render_bwd_kernel<<<a.ts.total_tiles, kBwdThreads, 0, s>>>(a);
    }
    return cudaGetLastError();
}

// SH rows of 3 K floats, as float4 when K is even and the row pointer 16-byte
// aligned (all rows then are).
template <int K>
__device__ __forceinline__ void load_row(const float *p, bool vec, float (&out)[K * 3]) {
    if constexpr ((K * 3) % 4 == 0) {
        if (vec) {
#pragma unroll
            for (int q = 0; q < (K * 3) / 4; ++q) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(p) + q);
                out[4 * q] = v.x;
                out[4 * q + 1] = v.y;
                out[4 * q + 2] = v.z;
                out[4 * q + 3] = v.w;
            }
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < K * 3; ++k) out[k] = __ldg(p + k);
}

// grad += Y[k] * gcol[c] at row position 3 k + c.
template <int K>
__device__ __forceinline__ void add_row(float *p, bool vec, const float (&Y)[16], const float (&gcol)[3]) {
    if constexpr ((K * 3) % 4 == 0) {
        if (vec) {
#pragma unroll
            for (int q = 0; q < (K * 3) / 4; ++q) {
                float4 v = reinterpret_cast<float4 *>(p)[q];
                v.x += Y[(4 * q) / 3] * gcol[(4 * q) % 3];
                v.y += Y[(4 * q + 1) / 3] * gcol[(4 * q + 1) % 3];
                v.z += Y[(4 * q + 2) / 3] * gcol[(4 * q + 2) % 3];
                v.w += Y[(4 * q + 3) / 3] * gcol[(4 * q + 3) % 3];
                reinterpret_cast<float4 *>(p)[q] = v;
            }
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < K * 3; ++k) p[k] += Y[k / 3] * gcol[k % 3];
}

// The screen-space sums of most Gaussians of a frame are exactly zero (no pixel
// composited them), and then so is everything they add to the gradients, which
// is nine tenths of the bytes preprocess_bwd would move for them.  So for one
// camera's view the Gaussians with any sum that is not zero are listed first.
// (A colour that is not finite makes the direction's gradient NaN even from
// zero sums, so such a Gaussian is listed too: kMetaNonFinite.)  A kernel of
// its own, because it is a stream of 76 bytes per Gaussian that wants many
// loads in flight, and the chain a few dependent loads and 90 registers per
// listed Gaussian that want full warps: the two in one kernel, each block
// listing 512 Gaussians for itself, kept a warp or two per block busy.
// 1M Gaussians at 1080p, a sixth of them listed: 188 us a thread per Gaussian,
// 70 in one kernel, now 16 + 17 (500k at 1264 x 832: 102, 43, 10 + 18).  The
// list with 8-byte loads 27, with 256 Gaussians and 128 threads per block 18.
// Of several cameras' views nearly every Gaussian is in some, where a list
// measured slower than a thread per Gaussian (220 against 166 us, five views of
// 200k).
constexpr int kListSpan = 512, kListThreads = 256;
__global__ void __launch_bounds__(kListThreads) bwd_list_kernel(PreBwdArgs a) {
    __shared__ uint8_t s_any[kListSpan];
    __shared__ uint32_t s_count, s_at;
    __shared__ uint16_t s_item[kListSpan];
    const int tid = threadIdx.x, span = min(kListSpan, a.n - (int)blockIdx.x * kListSpan);
    const size_t first = (size_t)blockIdx.x * kListSpan;
    if (tid == 0) s_count = 0u;
    for (int i = tid; i < kListSpan; i += kListThreads) s_any[i] = 0;
    __syncthreads();
    const double *g = a.g_screen + first * 9;
    const int words = 9 * span;
    if (span == kListSpan && reinterpret_cast<uintptr_t>(g) % 16 == 0) {
        constexpr int U = 9 * kListSpan / 2 / kListThreads;
        ulonglong2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = __ldcs(reinterpret_cast<const ulonglong2 *>(g) + tid + u * kListThreads);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = 2 * (tid + u * kListThreads);
            if (v[u].x << 1) s_any[i / 9] = 1;  // not +-0
            if (v[u].y << 1) s_any[(i + 1) / 9] = 1;
        }
    } else {
        for (int i = tid; i < words; i += kListThreads)
            if (g[i] != 0.0) s_any[i / 9] = 1;
    }
    for (int i = tid; i < span; i += kListThreads)
        if (a.meta[first + i] & kMetaNonFinite) s_any[i] = 1;
    __syncthreads();
    for (int i = tid; i < kListSpan; i += kListThreads) {  // whole warps pass
        const bool on = s_any[i];
        const uint32_t m = __ballot_sync(0xffffffffu, on);
        uint32_t at = 0;
        if ((tid & 31) == 0 && m) at = atomicAdd(&s_count, (uint32_t)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (on) s_item[at + __popc(m & ((1u << (tid & 31)) - 1u))] = (uint16_t)i;
    }
    __syncthreads();
    const uint32_t count = s_count;
    if (tid == 0 && count) s_at = atomicAdd(a.list_count, count);
    __syncthreads();
    for (uint32_t k = tid; k < count; k += kListThreads) a.list[s_at + k] = (uint32_t)first + s_item[k];
}

constexpr int kChainThreads = 128;
// SINGLE: one camera (a frame); the SH gradient Y gcol^T is then written
// directly instead of being summed over cameras in registers.
template <int DEG, bool SINGLE>
__device__ __forceinline__ void preprocess_bwd_one(const PreBwdArgs &a, int i) {
    constexpr int K = (DEG + 1) * (DEG + 1);
    constexpr int KS = SINGLE ? 1 : K;  // sizes of the multi-camera accumulator
    const float m0 = a.means[3 * i], m1 = a.means[3 * i + 1], m2 = a.means[3 * i + 2];
    const float sc0 = a.scales[3 * i], sc1 = a.scales[3 * i + 1], sc2 = a.scales[3 * i + 2];
    const float qw = a.quats[4 * i], qx = a.quats[4 * i + 1], qy = a.quats[4 * i + 2], qz = a.quats[4 * i + 3];
    const float *sh = a.sh + (size_t)i * K * 3;
    const bool vec = a.sh_vec4;
    float gmean[3] = {0.f, 0.f, 0.f}, gsc[3] = {0.f, 0.f, 0.f}, gq[4] = {0.f, 0.f, 0.f, 0.f}, gop = 0.f;
    float gsh[KS * 3];
#pragma unroll
    for (int k = 0; k < KS * 3; ++k) gsh[k] = 0.f;
    float Y1[16], gcol1[3] = {0.f, 0.f, 0.f};  // SINGLE: the one camera's basis and colour gradient
    bool any = false;
    for (int cam = 0; cam < (SINGLE ? 1 : a.cams.n_cams); ++cam) {
        const size_t rec = (size_t)cam * a.n + i;
        const int meta = a.meta[rec];
        if (!(meta & kMetaVisible)) continue;
        const CamDev &cd = a.cams.cam[cam];
        Proj p;
        if (!project_gaussian(cd, m0, m1, m2, sc0, sc1, sc2, qw, qx, qy, qz, a.raw, p)) continue;
        any = true;
        const double *gsd = a.g_screen + rec * 9;
        const float gmx = (float)gsd[0], gmy = (float)gsd[1];
        gop += (float)gsd[5];
        const float grgb[3] = {(float)gsd[6], (float)gsd[7], (float)gsd[8]};
        // gradient w.r.t. Sigma2D = [s11 s12; s12 s22] (s12 one parameter) as the
        // full-matrix gradient H with dL = tr(H^T dSigma)
        const float H00 = (float)gsd[2], H01 = 0.5f * (float)gsd[3], H11 = (float)gsd[4];
        // Sigma2D = A A^T + 0.3 I  ->  dL/dA = 2 H A
        float gA[6];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            gA[k] = 2.f * (H00 * p.A[k] + H01 * p.A[3 + k]);
            gA[3 + k] = 2.f * (H01 * p.A[k] + H11 * p.A[3 + k]);
        }
        // A = M (R S), M = J W
        const float *V = cd.V;
        float M0[3], M1[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            M0[j] = fmaf(p.J00, V[j], p.J02 * V[8 + j]);
            M1[j] = fmaf(p.J11, V[4 + j], p.J12 * V[8 + j]);
        }
        float gM0[3], gM1[3], gR[9];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            gM0[j] = 0.f;
            gM1[j] = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float rs = p.R[3 * j + k] * p.s[k];
                gM0[j] += gA[k] * rs;
                gM1[j] += gA[3 + k] * rs;
                const float grs = M0[j] * gA[k] + M1[j] * gA[3 + k];
                gR[3 * j + k] = grs * p.s[k];
                gsc[k] += (a.raw ? p.s[k] : 1.f) * grs * p.R[3 * j + k];
            }
        }
        float gJ00 = 0.f, gJ02 = 0.f, gJ11 = 0.f, gJ12 = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            gJ00 += gM0[j] * V[j];
            gJ02 += gM0[j] * V[8 + j];
            gJ11 += gM1[j] * V[4 + j];
            gJ12 += gM1[j] * V[8 + j];
        }
        // J(t) and mu^2D(t) -> t
        const float tz = p.tz, tzi = 1.f / tz, tzi2 = tzi * tzi;
        float gtx = gmx * cd.fx * tzi, gty = gmy * cd.fy * tzi;
        float gtz = -(gmx * cd.fx * p.tx + gmy * cd.fy * p.ty) * tzi2;
        gtz += -(gJ00 * cd.fx + gJ11 * cd.fy) * tzi2;
        if (p.clx) {
            gtz += -gJ02 * p.J02 * tzi;  // J02 = -fx L / tz
        } else {
            gtx += -gJ02 * cd.fx * tzi2;
            gtz += gJ02 * 2.f * cd.fx * p.tx * tzi2 * tzi;
        }
        if (p.cly) {
            gtz += -gJ12 * p.J12 * tzi;
        } else {
            gty += -gJ12 * cd.fy * tzi2;
            gtz += gJ12 * 2.f * cd.fy * p.ty * tzi2 * tzi;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) gmean[j] += V[j] * gtx + V[4 + j] * gty + V[8 + j] * gtz;

        // rotation of the normalised quaternion -> quaternion
        const float w = p.qn[0], x = p.qn[1], y = p.qn[2], z = p.qn[3];
        const float gw = gR[1] * (-2.f * z) + gR[2] * (2.f * y) + gR[3] * (2.f * z) + gR[5] * (-2.f * x) +
                         gR[6] * (-2.f * y) + gR[7] * (2.f * x);
        const float gx = gR[1] * (2.f * y) + gR[2] * (2.f * z) + gR[3] * (2.f * y) + gR[4] * (-4.f * x) +
                         gR[5] * (-2.f * w) + gR[6] * (2.f * z) + gR[7] * (2.f * w) + gR[8] * (-4.f * x);
        const float gy = gR[0] * (-4.f * y) + gR[1] * (2.f * x) + gR[2] * (2.f * w) + gR[3] * (2.f * x) +
                         gR[5] * (2.f * z) + gR[6] * (-2.f * w) + gR[7] * (2.f * z) + gR[8] * (-4.f * y);
        const float gz = gR[0] * (-4.f * z) + gR[1] * (-2.f * w) + gR[2] * (2.f * x) + gR[3] * (2.f * w) +
                         gR[4] * (-4.f * z) + gR[5] * (2.f * y) + gR[6] * (2.f * x) + gR[7] * (2.f * y);
        const float dot = gw * w + gx * x + gy * y + gz * z;
        const float iq = 1.f / p.qnorm;
        gq[0] += (gw - w * dot) * iq;
        gq[1] += (gx - x * dot) * iq;
        gq[2] += (gy - y * dot) * iq;
        gq[3] += (gz - z * dot) * iq;

        // colour from SH
        const float vx = m0 - cd.campos[0], vy = m1 - cd.campos[1], vz = m2 - cd.campos[2];
        const float vn = sqrtf(vx * vx + vy * vy + vz * vz), ivn = 1.f / vn;
        const float dx = vx * ivn, dy = vy * ivn, dz = vz * ivn;
        float Y[16];
        sh_eval<DEG>(dx, dy, dz, Y);
        float gcol[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) gcol[ch] = (meta >> (kMetaClampShift + ch)) & 1 ? 0.f : grgb[ch];
        if constexpr (SINGLE) {
#pragma unroll
            for (int k = 0; k < 16; ++k) Y1[k] = k < K ? Y[k] : 0.f;
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) gcol1[ch] = gcol[ch];
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                gsh[3 * k] += Y[k] * gcol[0];
                gsh[3 * k + 1] += Y[k] * gcol[1];
                gsh[3 * k + 2] += Y[k] * gcol[2];
            }
        }
        if (DEG > 0) {
            float c[K * 3], wsh[16];
            load_row<K>(sh, vec, c);
#pragma unroll
            for (int k = 0; k < K; ++k) wsh[k] = c[3 * k] * gcol[0] + c[3 * k + 1] * gcol[1] + c[3 * k + 2] * gcol[2];
            float ddx, ddy, ddz;
            sh_grad<DEG>(dx, dy, dz, wsh, ddx, ddy, ddz);
            const float r = ddx * dx + ddy * dy + ddz * dz;
            gmean[0] += (ddx - r * dx) * ivn;
            gmean[1] += (ddy - r * dy) * ivn;
            gmean[2] += (ddz - r * dz) * ivn;
        }
    }
    if (!any) return;
    // opacity: o = sigmoid(logit) when raw
    const float ov = a.opac[i];
    const float o = a.raw ? 1.f / (1.f + expf(-ov)) : ov;
    a.go[i] += a.raw ? gop * o * (1.f - o) : gop;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        a.gm[3 * i + j] += gmean[j];
        a.gs[3 * i + j] += gsc[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) a.gq[4 * i + j] += gq[j];
    float *gshp = a.gsh + (size_t)i * K * 3;
    if constexpr (SINGLE) {
        add_row<K>(gshp, a.gsh_vec4, Y1, gcol1);
    } else {
#pragma unroll
        for (int k = 0; k < K * 3; ++k) gshp[k] += gsh[k];
    }
}

template <int DEG, bool SINGLE>
__global__ void __launch_bounds__(SINGLE ? kChainThreads : 256) preprocess_bwd_kernel(PreBwdArgs a) {
    if constexpr (SINGLE) {
        const uint32_t count = *a.list_count;
        for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x)
            preprocess_bwd_one<DEG, SINGLE>(a, (int)a.list[k]);
    } else {
        const int i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i < a.n) preprocess_bwd_one<DEG, SINGLE>(a, i);
    }
}

template <bool SINGLE>
static void run_preprocess_bwd(const PreBwdArgs &a, int deg, cudaStream_t s) {
    const unsigned block = SINGLE ? kChainThreads : 256;
    unsigned grid = ((unsigned)a.n + block - 1) / block;
    if constexpr (SINGLE) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        grid = std::min(grid, (unsigned)sms * 5u);  // the resident blocks; they stride over the list
        note_launch("bwd_list_kernel", s);
        bwd_list_kernel<<<((unsigned)a.n + kListSpan - 1) / kListSpan, kListThreads, 0, s>>>(a);
    }
    note_launch("preprocess_bwd_kernel", s);
    switch (deg) {
    case 0: preprocess_bwd_kernel<0, SINGLE><<<grid, block, 0, s>>>(a); break;
    case 1: preprocess_bwd_kernel<1, SINGLE><<<grid, block, 0, s>>>(a); break;
    case 2: preprocess_bwd_kernel<2, SINGLE><<<grid, block, 0, s>>>(a); break;
    default: preprocess_bwd_kernel<3, SINGLE><<<grid, block, 0, s>>>(a); break;
    }
}

cudaError_t launch_preprocess_bwd(const PreBwdArgs &a, int deg, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    if (a.cams.n_cams == 1) run_preprocess_bwd<true>(a, deg, s);
    else run_preprocess_bwd<false>(a, deg, s);
    return cudaGetLastError();
}

}  // namespace qb
