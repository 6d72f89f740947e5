// Deterministic block reductions: a fixed warp-shuffle tree, then the same over
// the warps' values in the first warp.  Per-block results go to a partials array that a
// single-block kernel later sums in a fixed order, so a reduction over a
// given launch shape always rounds the same way.
#pragma once
#include "dw.cuh"

namespace jqcd {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ dwacc warp_sum_dw(dwacc v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float s2 = __shfl_down_sync(kFull, v.s, o);
    float c2 = __shfl_down_sync(kFull, v.c, o);
    float s, e;
    two_sum(v.s, s2, s, e);
    v.s = s;
    v.c = __fadd_rn(__fadd_rn(v.c, c2), e);
  }
  return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
  return v;
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
  return v;
}

// Block sum of one double per warp (given by lane 0); result in thread 0.
// blockDim.x must be a multiple of 32 and <= 1024.  A shuffle tree: a warp's
// FP64 add lasts about 67 cycles, so eight warps' values added one after the
// other took 0.28 us.
__device__ __forceinline__ double block_sum_warp_values(double warp_value) {
  __shared__ double sh[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) sh[warp] = warp_value;
  __syncthreads();
  double r = 0.0;
  if (warp == 0) {
    r = lane < nw ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1)
      if (o < nw) r += __shfl_down_sync(kFull, r, o);
  }
  __syncthreads();
  return r;
}

__device__ __forceinline__ double block_sum_dw(dwacc v) {
  v = warp_sum_dw(v);
  return block_sum_warp_values((double)v.s + (double)v.c);
}

__device__ __forceinline__ double block_sum_f(float v) {
  v = warp_sum_f(v);
  return block_sum_warp_values((double)v);
}

__device__ __forceinline__ double block_sum_d(double v) {
  v = warp_sum_d(v);
  return block_sum_warp_values(v);
}

// This thread's share of sum(partials[0..n)), i = tid, tid + blockDim.x, ...:
// sixteen loads are in flight before the first add.  Rows past n are left out,
// not added as zeros: each FP64 add of a warp holds its unit for about 67
// cycles, and with two warps a unit the fourteen or fifteen rows that a small
// grid's partials do not fill took most of a scalar step: with them left out,
// one warp a unit (reduce_threads) and the scalars read beside the partials, a
// hop with its norm takes 4.97 -> 4.25 us at 8^4 and 106.95 -> 106.15 us at
// 24^3x48 (2592 partials); mixed FP16 solve 16^4 2.84 -> 2.73 ms, 24^3x48 13.46
// -> 13.33 ms; staggered solve 24^3x48 36.2 -> 35.3 ms.  L2: loads from
// L2 (ld.global.cg), for partials written by other blocks of the same launch.
template <bool L2 = false>
__device__ __forceinline__ double thread_sum_partials(const double *partials, int n) {
  double v = 0.0;
  constexpr int kU = 16;
  const int bd = (int)blockDim.x;
  for (int row = 0; row < n; row += kU * bd) {  // uniform over the block
    double t[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = row + u * bd + (int)threadIdx.x;
      t[u] = i < n ? (L2 ? __ldcg(partials + i) : partials[i]) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (row + u * bd >= n) break;
      v += t[u];
    }
  }
  return v;
}

// sum of partials[0..n) by the whole block in a fixed order (valid in thread 0)
template <bool L2 = false>
__device__ __forceinline__ double block_sum_partials(const double *partials, int n) {
  return block_sum_d(thread_sum_partials<L2>(partials, n));
}

}  // namespace jqcd
