// qb_train.cu -- one optimisation step around the differentiable rasteriser:
// the L1 image loss and its gradient, and a fused Adam update of the raw
// scene parameters (Kingma & Ba's bias-corrected rule).  Both are plain
// elementwise HBM-bound kernels; the loss is summed per block in FP64.
#include "qb_kernels.cuh"

namespace qb {

// dL[i] = sign(img[i] - target[i]) * scale (0 where equal); *loss += scale *
// sum |img - target| when loss is non-null.
__global__ void __launch_bounds__(256) l1_grad_kernel(const float *__restrict__ img, const float *__restrict__ target,
                                                      float *__restrict__ dL, uint64_t n, float scale, double *loss) {
    double acc = 0.0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const float d = img[i] - target[i];
        dL[i] = d > 0.f ? scale : (d < 0.f ? -scale : 0.f);
        acc += fabs((double)d);
    }
    if (!loss) return;
    __shared__ double s[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s[w];
        atomicAdd(loss, t * (double)scale);
    }
}

// Adam, step t (1-based): m = b1 m + (1 - b1) g; v = b2 v + (1 - b2) g^2;
// p -= lr * (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps).
// One pass over seven arrays' worth of traffic, bound by memory: with VEC
// (16-byte aligned arrays) a thread has four 16-byte loads of two groups of four
// parameters in flight, instead of four 4-byte ones.  500k Gaussians of SH
// degree 3 (five launches, 826 MB): 195 -> 160 us with the launches' gaps.
__device__ __forceinline__ void adam_one(float &p, float g, float &m, float &v, float lr, float b1, float b2, float eps,
                                         float c1, float c2) {
    const float mi = fmaf(b1, m, (1.f - b1) * g);
    const float vi = fmaf(b2, v, (1.f - b2) * g * g);
    m = mi;
    v = vi;
    p -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

template <bool VEC>
__global__ void __launch_bounds__(256) adam_kernel(float *__restrict__ p, const float *__restrict__ g,
                                                   float *__restrict__ m, float *__restrict__ v, uint64_t n, float lr,
                                                   float b1, float b2, float eps, float c1, float c2) {
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, threads = (uint64_t)gridDim.x * blockDim.x;
    uint64_t i0 = 0;
    if constexpr (VEC) {
        const uint64_t n4 = n / 4;
        constexpr int U = 2;
        for (uint64_t j = t; j < n4; j += U * threads) {
            float4 P[U], G[U], M[U], V[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t k = j + u * threads;
                if (k < n4) {
                    P[u] = reinterpret_cast<const float4 *>(p)[k];
                    G[u] = reinterpret_cast<const float4 *>(g)[k];
                    M[u] = reinterpret_cast<const float4 *>(m)[k];
                    V[u] = reinterpret_cast<const float4 *>(v)[k];
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t k = j + u * threads;
                if (k < n4) {
                    adam_one(P[u].x, G[u].x, M[u].x, V[u].x, lr, b1, b2, eps, c1, c2);
                    adam_one(P[u].y, G[u].y, M[u].y, V[u].y, lr, b1, b2, eps, c1, c2);
                    adam_one(P[u].z, G[u].z, M[u].z, V[u].z, lr, b1, b2, eps, c1, c2);
                    adam_one(P[u].w, G[u].w, M[u].w, V[u].w, lr, b1, b2, eps, c1, c2);
                    reinterpret_cast<float4 *>(p)[k] = P[u];
                    reinterpret_cast<float4 *>(m)[k] = M[u];
                    reinterpret_cast<float4 *>(v)[k] = V[u];
                }
            }
        }
        i0 = 4 * n4;  // at most three are left
    }
    for (uint64_t i = i0 + t; i < n; i += threads) {
        float pi = p[i], mi = m[i], vi = v[i];
        adam_one(pi, g[i], mi, vi, lr, b1, b2, eps, c1, c2);
        p[i] = pi;
        m[i] = mi;
        v[i] = vi;
    }
}

// Zeroes five arrays in one launch (the gradients of a scene, before the
// backward adds to them).
struct Zero5 {
    float *p[5];
    uint64_t n[5];
};
__global__ void __launch_bounds__(256) zero5_kernel(Zero5 z) {
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, threads = (uint64_t)gridDim.x * blockDim.x;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        uint64_t i0 = 0;
        if ((reinterpret_cast<uintptr_t>(z.p[k]) & 15) == 0) {
            const uint64_t n4 = z.n[k] / 4;
            for (uint64_t i = t; i < n4; i += threads) reinterpret_cast<float4 *>(z.p[k])[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            i0 = 4 * n4;
        }
        for (uint64_t i = i0 + t; i < z.n[k]; i += threads) z.p[k][i] = 0.f;
    }
}

static unsigned grid_for(uint64_t n) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t want = (n + 255) / 256, cap = (uint64_t)(sms > 0 ? sms : 1) * 8;
    return (unsigned)(want < cap ? (want > 0 ? want : 1) : cap);
}

cudaError_t launch_l1_grad(const float *img, const float *target, float *dL, uint64_t n, float scale, double *loss,
                           cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    note_launch("l1_grad_kernel", s), l1_grad_kernel<<<grid_for(n), 256, 0, s>>>(img, target, dL, n, scale, loss);
    return cudaGetLastError();
}

cudaError_t launch_zero5(float *const p[5], const uint64_t n[5], cudaStream_t s) {
    Zero5 z;
    uint64_t most = 0;
    for (int k = 0; k < 5; ++k) {
        z.p[k] = p[k];
        z.n[k] = n[k];
        most = n[k] > most ? n[k] : most;
    }
    if (most == 0) return cudaSuccess;
    note_launch("zero5_kernel", s), zero5_kernel<<<grid_for((most + 3) / 4), 256, 0, s>>>(z);
    return cudaGetLastError();
}

cudaError_t launch_adam(float *p, const float *g, float *m, float *v, uint64_t n, float lr, float b1, float b2,
                        float eps, int t, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    const bool vec = ((reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(g) | reinterpret_cast<uintptr_t>(m) |
                       reinterpret_cast<uintptr_t>(v)) & 15) == 0;
    note_launch("adam_kernel", s);
    if (vec) adam_kernel<true><<<grid_for((n + 7) / 8), 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
    else adam_kernel<false><<<grid_for(n), 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

}  // namespace qb
