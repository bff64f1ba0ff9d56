// qb_preprocess.cu -- K1: Gaussian-parallel preprocess (Sec. 2 "Preprocess",
// Sec. 3.1 QuadBox construction, Sec. 3.2 QPass count).
//
// One thread per Gaussian.  Reads the raw parameters (44 B + 12 (deg+1)^2 B),
// writes mu^2D, conic+opacity, colour+depth, the box record, the 3-sigma
// radius, a meta word, the tile and cell counts, the sub-boxes' tile
// rectangles and the depth-sort pair.  Culled Gaussians write only their
// counts and meta word and skip the SH read.
#include "qb_kernels.cuh"
#include "qb_project.cuh"

namespace qb {

template <int DEG>
__global__ void __launch_bounds__(256, 3) preprocess_kernel(PreArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    const int ci = blockIdx.y;  // camera of this grid row
    const CamDev &cam = a.cams.cam[ci];
    const size_t o = (size_t)ci * a.n + i;  // output record
    const float m0 = a.means[3 * i], m1 = a.means[3 * i + 1], m2 = a.means[3 * i + 2];
    Proj p;
    float4 q4;
    if (a.quat_vec4) {
        q4 = __ldg(reinterpret_cast<const float4 *>(a.quats) + i);
    } else {
        q4 = make_float4(a.quats[4 * i], a.quats[4 * i + 1], a.quats[4 * i + 2], a.quats[4 * i + 3]);
    }
    bool ok = project_gaussian(cam, m0, m1, m2, a.scales[3 * i], a.scales[3 * i + 1], a.scales[3 * i + 2], q4.x,
                               q4.y, q4.z, q4.w, a.raw, p);
    if (ok) {
        float ov = a.opac[i];
        p.o = a.raw ? 1.0f / (1.0f + expf(-ov)) : ov;
        ok = p.o >= kAlphaMin;  // no pixel of this Gaussian reaches alpha_min
    }
    if (!ok) {
        a.counts[o] = 0u;
        a.cc[o] = make_uint2(0u, 0u);
        a.meta[o] = 0;
        a.shape[o] = make_float2(0.f, 0.f);
        if (a.depth_keys) {  // no tiles: sorts after every Gaussian that has some
            a.depth_keys[o] = 0x7fffffffu;
            a.depth_vals[o] = (uint32_t)o;
        }
        return;
    }
    BoxTerms bt = box_terms(p);

    // view-dependent colour
    constexpr int K = (DEG + 1) * (DEG + 1);
    float dx = m0 - cam.campos[0], dy = m1 - cam.campos[1], dz = m2 - cam.campos[2];
    float inv = 1.0f / sqrtf(dx * dx + dy * dy + dz * dz);
    float Y[16];
    sh_eval<DEG>(dx * inv, dy * inv, dz * inv, Y);
    const float *sh = a.sh + (size_t)i * (K * 3);
    float rgb[3] = {0.5f, 0.5f, 0.5f};
    if ((K * 3) % 4 == 0 && a.sh_vec4) {
        // 16-byte loads of the coefficient row (3K floats, K even)
        float c[K * 3];
        const float4 *sh4 = reinterpret_cast<const float4 *>(sh);
#pragma unroll
        for (int q = 0; q < (K * 3) / 4; ++q) {
            const float4 v = __ldg(sh4 + q);
            c[4 * q] = v.x;
            c[4 * q + 1] = v.y;
            c[4 * q + 2] = v.z;
            c[4 * q + 3] = v.w;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            rgb[0] = fmaf(Y[k], c[3 * k], rgb[0]);
            rgb[1] = fmaf(Y[k], c[3 * k + 1], rgb[1]);
            rgb[2] = fmaf(Y[k], c[3 * k + 2], rgb[2]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            rgb[0] = fmaf(Y[k], __ldg(sh + 3 * k), rgb[0]);
            rgb[1] = fmaf(Y[k], __ldg(sh + 3 * k + 1), rgb[1]);
            rgb[2] = fmaf(Y[k], __ldg(sh + 3 * k + 2), rgb[2]);
        }
    }
    int meta = kMetaVisible | (bt.orient ? kMetaOrient : 0);
    if (!isfinite(rgb[0]) || !isfinite(rgb[1]) || !isfinite(rgb[2])) meta |= kMetaNonFinite;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        if (rgb[ch] < 0.f) {
            meta |= 1 << (kMetaClampShift + ch);
            rgb[ch] = 0.f;
        }
    }

    Rect rects[4];
    box_rects(p.mx, p.my, bt.box, bt.r3, bt.orient, a.mode, a.clamp3s, cam.W, cam.H, rects);
    // tiles of the QPass traversal, and the entries it gets among the cells of
    // 8 x 4 tiles: the cells of the bounding box of its tiles (cell_entries)
    uint32_t cnt, ccnt;
    if (a.mode == QB_BIN_QUADBOX_NAIVE) {  // the same set, counted the naive way
        Rect crects[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) crects[q] = cell_rect(rects[q]);
        cnt = naive_count(rects);
        ccnt = naive_count(crects);
    } else {
        // (a mode of a single box has the others empty)
        cnt = a.mode == QB_BIN_AABB3S || a.mode == QB_BIN_ADR ? (uint32_t)rect_area(rects[0]) : union_count(rects);
        ccnt = cell_entries(rects, cnt);
    }
    if (cnt > 0u) {
        uint4 pk[2];
        pack_rects(rects, pk);
        a.rects[2 * o] = pk[0];
        a.rects[2 * o + 1] = pk[1];
    }

    a.xy[o] = make_float2(p.mx, p.my);
    // the exact power form's terms (qb_internal.cuh), for elongated Gaussians only
    float2 shape = make_float2(0.f, 0.f);
    if (p.det < kElongatedF2 * (p.s11 * p.s22)) {
        const float inv22 = 1.0f / p.s22;
        shape = make_float2(-p.s12 * inv22, -0.5f * inv22);
    }
    a.shape[o] = shape;
    a.conic_o[o] = make_float4(p.a, p.b, p.c, p.o);
    a.rgbd[o] = make_float4(rgb[0], rgb[1], rgb[2], p.tz);
    a.box[o] = bt.box;
    a.r3[o] = bt.r3;
    a.meta[o] = meta;
    a.counts[o] = cnt;
    a.cc[o] = make_uint2(cnt, ccnt);
    if (a.depth_keys) {
        // the depth-order sort's input: positive float depths order like their
        // bits; Gaussians without tiles sort last
        a.depth_keys[o] = cnt ? (__float_as_uint(p.tz) & 0x7fffffffu) : 0x7fffffffu;
        a.depth_vals[o] = (uint32_t)o;
    }
}

cudaError_t launch_preprocess(const PreArgs &a, int deg, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    dim3 grid((a.n + 255) / 256, a.cams.n_cams), block(256);
    switch (deg) {
    case 0: note_launch("preprocess_kernel", s), preprocess_kernel<0><<<grid, block, 0, s>>>(a); break;
    case 1: note_launch("preprocess_kernel", s), preprocess_kernel<1><<<grid, block, 0, s>>>(a); break;
    case 2: note_launch("preprocess_kernel", s), preprocess_kernel<2><<<grid, block, 0, s>>>(a); break;
    default: note_launch("preprocess_kernel", s), preprocess_kernel<3><<<grid, block, 0, s>>>(a); break;
    }
    return cudaGetLastError();
}

}  // namespace qb
