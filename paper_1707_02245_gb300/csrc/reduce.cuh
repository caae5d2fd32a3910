// Block-wide FP64 sums used by the duality-gap kernels (deterministic order for a
// fixed launch shape: warp shuffles, then one warp over the per-warp sums).
#pragma once
#include <cuda_runtime.h>

namespace pat {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sums NV doubles per thread over the block; the result is valid in the thread with
// linear index 0.  The block size must be a multiple of 32 and at most 1024.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV]) {
    __shared__ double sh[NV][32];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    const int nw = (blockDim.x * blockDim.y) >> 5;
#pragma unroll
    for (int c = 0; c < NV; ++c) v[c] = warp_sum(v[c]);
    __syncthreads();  // sh may still be read by a previous call
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < NV; ++c) sh[c][wid] = v[c];
    }
    __syncthreads();
    if (wid == 0) {
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            double x = lane < nw ? sh[c][lane] : 0.0;
            v[c] = warp_sum(x);
        }
    }
}

// s + e = a + b exactly (Knuth's TwoSum); the intrinsics keep the compiler from
// contracting or reordering the roundings
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// (hi, lo) += (h2, l2) for unevaluated pairs of FP32 numbers
__device__ __forceinline__ void pair_add(float& hi, float& lo, float h2, float l2) {
    float s, e;
    two_sum(hi, h2, s, e);
    two_sum(s, __fadd_rn(__fadd_rn(lo, l2), e), hi, lo);
}

// Warp sums of NV <= 16 FP32 values per lane.  They are carried as unevaluated pairs hi + lo
// of FP32 numbers, so a sum keeps about 48 significant bits without FP64 arithmetic (GB300's
// FP64 pipe runs at 1/64 of FP32).  The lanes of a pair exchange halves of their values at
// every step, so the values take 16 pair additions in all instead of 5 each (the gap's 11
// sums in every warp of K cost 4 us per evaluation at 64^2 with a tree for each).  Lanes 2c
// and 2c + 1 return the sum of value c; its order is fixed.
template <int NV>
__device__ __forceinline__ double warp_sums_pair(const float (&t)[NV]) {
    static_assert(NV <= 16, "two lanes to a value");
    const int lane = threadIdx.x & 31;
    float hi[16], lo[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        hi[c] = c < NV ? t[c < NV ? c : 0] : 0.f;
        lo[c] = 0.f;
    }
#pragma unroll
    for (int h = 8, o = 16; h > 0; h >>= 1, o >>= 1) {
        // lanes with bit o keep the upper half of their 2h values, the others the lower half
        const bool up = lane & o;
#pragma unroll
        for (int c = 0; c < h; ++c) {
            const float sh = up ? hi[c] : hi[c + h], sl = up ? lo[c] : lo[c + h];
            hi[c] = up ? hi[c + h] : hi[c];
            lo[c] = up ? lo[c + h] : lo[c];
            const float rh = __shfl_xor_sync(0xffffffffu, sh, o), rl = __shfl_xor_sync(0xffffffffu, sl, o);
            pair_add(hi[c], lo[c], rh, rl);
        }
    }
    const float rh = __shfl_xor_sync(0xffffffffu, hi[0], 1), rl = __shfl_xor_sync(0xffffffffu, lo[0], 1);
    pair_add(hi[0], lo[0], rh, rl);
    return (double)hi[0] + (double)lo[0];
}

// Block sums of NV <= 16 FP32 values per thread: warps reduce with warp_sums_pair, then one
// warp adds the per-warp sums in FP64, two lanes to a value, so all values share each FP64
// instruction (a warp's FP64 addition holds the SM's FP64 pipe for 16 clocks whatever its
// lanes do).  Lanes 2c of warp 0 return the sum of value c; the order is fixed for a fixed
// launch shape.  The block size must be a multiple of 32 and at most 1024.  sh is the
// caller's scratch in shared memory (which nothing else may use meanwhile).
template <int NV>
__device__ __forceinline__ double block_sums_pair(const float (&t)[NV], double (*sh)[32]) {
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    const int nw = (blockDim.x * blockDim.y) >> 5;
    const double w = warp_sums_pair<NV>(t);
    if ((lane & 1) == 0 && lane / 2 < NV) sh[lane / 2][wid] = w;
    __syncthreads();
    double x = 0.0;
    if (wid == 0) {
        if (lane / 2 < NV)
            for (int k = lane & 1; k < nw; k += 2) x += sh[lane / 2][k];
        x += __shfl_down_sync(0xffffffffu, x, 1);
    }
    return x;
}

}  // namespace pat
