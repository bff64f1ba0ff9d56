// qb_scan.cuh -- warp and block scans, and the division by a small segment
// length, shared by the binning kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace qb {

__device__ __forceinline__ uint32_t lanemask_le() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_le;" : "=r"(m));
    return m;
}

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Inclusive block scan (blockDim.x a multiple of 32, <= 1024); *total gets
// the block sum.
template <typename T>
__device__ __forceinline__ T block_incl_scan(T v, T *total) {
    __shared__ T warp_sums[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T incl = warp_incl_scan(v);
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        T s = lane < nw ? warp_sums[lane] : T(0);
        s = warp_incl_scan(s);
        warp_sums[lane] = s;
    }
    __syncthreads();
    T before = wid > 0 ? warp_sums[wid - 1] : T(0);
    *total = warp_sums[nw - 1];
    __syncthreads();
    return incl + before;
}

// k / len and k % len through the reciprocal inv = 1 / len: for k < 2^24 the
// estimate is off by at most one, which one exact correction mends.
__device__ __forceinline__ void seg_divide(uint32_t k, uint32_t len, float inv, uint32_t &q, uint32_t &r) {
    int32_t a = (int32_t)((float)k * inv);
    int32_t b = (int32_t)k - a * (int32_t)len;
    if (b < 0) { --a; b += (int32_t)len; }
    if (b >= (int32_t)len) { ++a; b -= (int32_t)len; }
    q = (uint32_t)a;
    r = (uint32_t)b;
}

}  // namespace qb
