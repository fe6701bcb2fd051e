// Block sums of several FP64 values and their combination over the blocks of a grid, in
// a fixed order (kernels of kRedThreads threads).
#pragma once

#include "omm_internal.cuh"

namespace omm {

constexpr int kRedThreads = 256;

// Sums of NV (at most 16) values over the block, value t in lane t of warp 0.  The
// lanes of a warp halve the values between them (16 additions for 16 values where a
// tree per value takes 80: an FP64 instruction occupies this part's FP64 unit for ~18
// cycles, and eight warps of such trees took 5 us); the partners are the tree's, so the sums
// are too.  Then a lane per value adds the warps' sums in order.
template <int NV>
__device__ __forceinline__ double block_totals(const double (&v)[NV], double *red /* smem 8 P, P = 4 or 16 */) {
    constexpr int P = NV <= 4 ? 4 : 16;
    static_assert(NV <= 16, "one lane per value");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double w[P];
#pragma unroll
    for (int q = 0; q < P; ++q) w[q] = q < NV ? v[q < NV ? q : 0] : 0.0;
    // after the step with partner lane ^ off a lane holds half as many values
#pragma unroll
    for (int n = P / 2, off = 16; n > 0; n >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const double give = up ? w[i] : w[i + n], keep = up ? w[i + n] : w[i];
            w[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    }
#pragma unroll
    for (int off = 16 / P; off > 0; off >>= 1) w[0] += __shfl_xor_sync(0xffffffffu, w[0], off);
    if (lane % (32 / P) == 0) red[warp * P + lane / (32 / P)] = w[0];
    __syncthreads();
    double s = 0.0;
    if (warp == 0 && lane < NV)
#pragma unroll
        for (int q = 0; q < kRedThreads / 32; ++q) s += red[q * P + lane];
    __syncthreads();
    return s;
}

// Publish this block's NV partials (value t in lane t of warp 0); returns true in the
// last block to finish, whose threads then all hold the totals in `tot`.  The last
// block sums the partials in a fixed order (warp per value, lane-strided blocks, shuffle
// tree), so the result does not depend on which block finished last.  Blocks from `parts`
// on hold no partials and only count.
template <int NV>
__device__ __forceinline__ bool publish_totals(double v, double *partials, unsigned int *counter, double (&tot)[NV],
                                               double *red, unsigned parts) {
    __shared__ bool is_last;
    if (threadIdx.x < 32) {
        if (threadIdx.x < NV && blockIdx.x < parts) partials[blockIdx.x * NV + threadIdx.x] = v;
        __threadfence();
        __syncwarp();
        if (threadIdx.x == 0) is_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
    }
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
    // warp w sums values w, w + NT/32, ...: its lanes take blocks lane, lane + 32,
    // ... in order, then a fixed shuffle tree (one dependent chain per value on
    // the long-latency FP64 unit, instead of a block-wide tree per value)
    for (int q = threadIdx.x >> 5; q < NV; q += kRedThreads / 32) {
        double s = 0.0;
        // the lane's blocks in order, eight loads in flight at a time
        unsigned b = threadIdx.x & 31;
        for (; b + 224 < parts; b += 256) {
            double p[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) p[k] = __ldcg(&partials[(b + 32 * k) * NV + q]);
#pragma unroll
            for (int k = 0; k < 8; ++k) s += p[k];
        }
        for (; b < parts; b += 32) s += __ldcg(&partials[b * NV + q]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if ((threadIdx.x & 31) == 0) red[q] = s;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) tot[q] = red[q];
    if (threadIdx.x == 0) *counter = 0u;
    __syncthreads();   // red is free again for the caller
    return true;
}

}  // namespace omm
