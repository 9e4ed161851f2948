// Device helpers shared by the reductions over the state.
#pragma once

namespace svk {

constexpr int RED_THREADS = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sum; result valid in thread 0.
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double ws[RED_THREADS / 32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) ws[w] = v;
    __syncthreads();
    double r = 0.0;
    if (w == 0) {
        r = lane < RED_THREADS / 32 ? ws[lane] : 0.0;
        r = warp_sum(r);
    }
    __syncthreads();
    return r;
}

// |alpha|^2 in the state's precision: fl(fl(x*x) + fl(y*y)) with round-to-nearest and
// no contraction, one fixed formula shared by probs, norm and top-k (so that a host
// computing the same IEEE operations takes the same top-k decisions).
__device__ __forceinline__ float prob_of(float x, float y) {
    return __fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y));
}
__device__ __forceinline__ double prob_of(double x, double y) {
    return __dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y));
}

}  // namespace svk
