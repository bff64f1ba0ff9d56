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

// The SH rows of a warp's Gaussians are brought to shared memory by
// asynchronous copies, consecutive lanes taking consecutive pieces, while the
// projection is computed: read by their own lanes, 16 bytes at a stride of a
// row, half of every 32-byte sector came twice (497 MB from L2 for 236 MB of
// scene) and the loads were waited for at a third of the SM's warps.  Only the
// rows of Gaussians past the near plane and the opacity test are copied.
// Pieces of 16 bytes at degrees 1 and 3 (a row of degree 3 is padded to 52
// floats, so that eight lanes' 16-byte reads fall on distinct banks), of 4
// bytes at degree 2 (rows of 27 floats); degree 0 reads its 3 floats directly.
// 1M Gaussians of degree 3 86 -> 70 us (326 MB, 4.7 TB/s; 80 registers, three
// blocks per SM), 3M seen from inside 210 -> 177; 16 views of 1M, whose cameras
// now share a Gaussian's reads, 1084 -> 766.
constexpr int kPreThreads = 256;

template <int DEG>
struct ShRows {
    static constexpr int kFloats = 3 * (DEG + 1) * (DEG + 1);
    static constexpr int kPiece = DEG == 2 ? 1 : 4;          // floats per copy
    static constexpr int kStride = DEG == 3 ? 52 : kFloats;  // floats between rows
    static constexpr int kCopies = kFloats / kPiece;         // per row, and per lane for 32 rows
    static constexpr int kBytes = DEG == 0 ? 0 : 4 * kStride * kPreThreads;
};

template <int DEG>
__device__ __forceinline__ void copy_sh_rows(float *rows, const float *sh, uint32_t wanted, int lane) {
    using R = ShRows<DEG>;
#pragma unroll
    for (int c = 0; c < R::kCopies; ++c) {
        const int e = 32 * c + lane, row = e / R::kCopies, q = e - row * R::kCopies;
        if ((wanted >> row) & 1u) {
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(rows + row * R::kStride + q * R::kPiece);
            const float *src = sh + (size_t)row * R::kFloats + q * R::kPiece;
            if constexpr (R::kPiece == 4)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
            else
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
        }
    }
}

// Block b takes Gaussians kPreThreads (b / cameras) ... of camera b mod
// cameras, so that the cameras of a group read a Gaussian's parameters while
// they are in L2.
template <int DEG>
__global__ void __launch_bounds__(kPreThreads, 3) preprocess_kernel(PreArgs a) {
    extern __shared__ __align__(16) float s_rows[];
    const int lane = threadIdx.x & 31;
    const int ci = (int)(blockIdx.x % (uint32_t)a.cams.n_cams);
    const int i = (int)(blockIdx.x / (uint32_t)a.cams.n_cams) * kPreThreads + threadIdx.x;
    const bool in = i < a.n;
    const CamDev &cam = a.cams.cam[ci];
    const size_t o = (size_t)ci * a.n + i;  // output record
    float m0 = 0.f, m1 = 0.f, m2 = 0.f, sc0 = 0.f, sc1 = 0.f, sc2 = 0.f;
    float4 q4 = make_float4(1.f, 0.f, 0.f, 0.f);
    Proj p;
    bool ok = in;
    if (in) {
        m0 = a.means[3 * i], m1 = a.means[3 * i + 1], m2 = a.means[3 * i + 2];
        const float ov = a.opac[i];
        if (a.quat_vec4) {
            q4 = __ldg(reinterpret_cast<const float4 *>(a.quats) + i);
        } else {
            q4 = make_float4(a.quats[4 * i], a.quats[4 * i + 1], a.quats[4 * i + 2], a.quats[4 * i + 3]);
        }
        sc0 = a.scales[3 * i], sc1 = a.scales[3 * i + 1], sc2 = a.scales[3 * i + 2];
        p.o = a.raw ? 1.0f / (1.0f + expf(-ov)) : ov;
        ok = p.o >= kAlphaMin;  // else no pixel of this Gaussian reaches alpha_min
        // (project_gaussian's own test of the near plane)
        ok = ok && fmaf(cam.V[8], m0, fmaf(cam.V[9], m1, fmaf(cam.V[10], m2, cam.V[11]))) > cam.znear;
    }
    float *rows = s_rows + (threadIdx.x >> 5) * 32 * ShRows<DEG>::kStride;
    const bool staged = DEG == 2 || (DEG != 0 && a.sh_vec4);
    if constexpr (DEG != 0) {
        const uint32_t wanted = __ballot_sync(0xffffffffu, ok);
        if (staged) copy_sh_rows<DEG>(rows, a.sh + (size_t)(i - lane) * ShRows<DEG>::kFloats, wanted, lane);
    }
    if (ok) ok = project_gaussian(cam, m0, m1, m2, sc0, sc1, sc2, q4.x, q4.y, q4.z, q4.w, a.raw, p);
    if (staged) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
    }
    if (!in) return;
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
    if (staged) {
        float c[K * 3];
        const float *row = rows + lane * ShRows<DEG>::kStride;
        if constexpr (ShRows<DEG>::kPiece == 4) {
#pragma unroll
            for (int q = 0; q < (K * 3) / 4; ++q) {
                const float4 v = reinterpret_cast<const float4 *>(row)[q];
                c[4 * q] = v.x;
                c[4 * q + 1] = v.y;
                c[4 * q + 2] = v.z;
                c[4 * q + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < K * 3; ++q) c[q] = row[q];
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

template <int DEG>
static cudaError_t run_preprocess(const PreArgs &a, cudaStream_t s) {
    constexpr size_t smem = ShRows<DEG>::kBytes;
    if (smem > 48 * 1024) {
        const cudaError_t e = ensure_dyn_smem((const void *)preprocess_kernel<DEG>, smem);
        if (e != cudaSuccess) return e;
    }
    const unsigned blocks = ((unsigned)a.n + kPreThreads - 1) / kPreThreads * (unsigned)a.cams.n_cams;
    note_launch("preprocess_kernel", s), preprocess_kernel<DEG><<<blocks, kPreThreads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_preprocess(const PreArgs &a, int deg, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    switch (deg) {
    case 0: return run_preprocess<0>(a, s);
    case 1: return run_preprocess<1>(a, s);
    case 2: return run_preprocess<2>(a, s);
    default: return run_preprocess<3>(a, s);
    }
}

}  // namespace qb
