// qb_stage.cuh -- how a warp brings the entries of a tile's list to its shared
// memory, for the render (K6) and its backward (K7).
#pragma once

#include "qb_kernels.cuh"

namespace qb {

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

#define kNaN __int_as_float(0x7fc00000)
constexpr float kCapTest = 0.98f;  // opacities above this may meet the 0.99 cap

// A warp's shared memory.  raw: one entry's record per lane, the target of
// the asynchronous copies, read back by the same lane.  The others hold the
// compacted entries laid out for the packed FP32x2 arithmetic of sm_100+:
// every operand the two pixels of a pair share is stored twice, so a pair
// register loads it without a move.
//   sx = (mu_x, mu_x, mu_y, mu_y), sq = (ca, ca, cb, cb),
//   sk = (cc, cc, skip threshold, info), s1 = (o, o, r, r), s2 = (g, g, b, b),
//   se = (rr, rr, ce, ce) (elongated entries only).
// info is the entry's position in the list + 1, with kSlowEntry set where the
// entry may meet the 0.99 cap or is elongated (qb_internal.cuh), kLongEntry
// for the latter: then its exponent is ca u^2 + ce dy^2 with
// u = dx + rr dy, rr = b / a, ce = -1 / (2 Sigma22), which does not cancel.
constexpr uint32_t kSlowEntry = 0x80000000u, kLongEntry = 0x40000000u;  // positions are below 2^30
struct RenderStage {
    float4 raw_co[32], raw_rgb[32];
    float2 raw_xy[32], raw_sh[32];
    float4 sx[32], sq[32], sk[32], s1[32], s2[32], se[32];
};

__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

__device__ __forceinline__ void copy_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// min(a, b), NaN where either is
__device__ __forceinline__ float min_nan(float a, float b) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

struct StageSource {
    const float2 *xy, *shape;
    const float4 *conic_o, *rgbd;
};

// Starts the copies of the lane's record g.
__device__ __forceinline__ void stage_copy(RenderStage &S, const StageSource &src, uint32_t g, int lane) {
    copy_async16(&S.raw_co[lane], src.conic_o + g);
    copy_async16(&S.raw_rgb[lane], src.rgbd + g);
    copy_async8(&S.raw_xy[lane], src.xy + g);
    copy_async8(&S.raw_sh[lane], src.shape + g);
}

// Stages the warp's entries (lane's record copied; `have`: the lane has one,
// at list position pos - 1) that reach the 16 x ROWS pixels from (x0, y0), in
// lane order; returns how many.  BACKWARD stores -o instead of o, and the
// record's index rec in ids.  COUNT: for the counted render.  All lanes pass
// through the ballot, so the walk of the last entries is over.  The caller
// synchronises the warp before it reads them.
template <bool BACKWARD, int ROWS = 8, bool COUNT = false>
__device__ __forceinline__ int stage_entries(RenderStage &S, bool have, int pos, float x0, float y0, int lane,
                                             uint32_t rec = 0u, uint32_t *ids = nullptr) {
    bool hit = false;
    float2 m = f2(0.f, 0.f), sh = f2(0.f, 0.f);
    float4 co = make_float4(0.f, 0.f, 0.f, 0.f), rgb = co;
    float skip = 0.f;
    if (have) {
        m = S.raw_xy[lane];
        sh = S.raw_sh[lane];
        co = S.raw_co[lane];
        rgb = S.raw_rgb[lane];
        skip = skip_threshold<COUNT>(co.w);
        hit = ellipse_meets_rect(m.x, m.y, co.x, co.y, co.z, skip, sh, x0, y0, x0 + 15.f, y0 + (float)(ROWS - 1));
    }
    const uint32_t hits = __ballot_sync(0xffffffffu, hit);
    if (hit) {
        const int k = __popc(hits & ((1u << lane) - 1u));
        const float ca = -0.5f * co.x, cbv = -co.y, cc = -0.5f * co.z;
        const float o = BACKWARD ? -co.w : co.w;
        uint32_t info = (uint32_t)pos;
        if (co.w > kCapTest) info |= kSlowEntry;
        if (sh.y != 0.f) info |= kSlowEntry | kLongEntry;
        S.sx[k] = make_float4(m.x, m.x, m.y, m.y);
        S.sq[k] = make_float4(ca, ca, cbv, cbv);
        S.sk[k] = make_float4(cc, cc, skip, __uint_as_float(info));
        S.s1[k] = make_float4(o, o, rgb.x, rgb.x);
        S.s2[k] = make_float4(rgb.y, rgb.y, rgb.z, rgb.z);
        if (sh.y != 0.f) S.se[k] = make_float4(sh.x, sh.x, sh.y, sh.y);
        if (BACKWARD) ids[k] = rec;
    }
    return __popc(hits);
}

}  // namespace qb
