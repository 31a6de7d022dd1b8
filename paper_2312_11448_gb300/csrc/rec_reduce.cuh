// Fixed-order block reductions for the streaming passes.  Each block writes
// its partials; the last block to finish (atomic ticket) combines all
// partials in block order.  Given the grid size, the result is bit-identical
// from run to run (no floating-point atomics).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "rec_df.cuh"

namespace rec {

// Sums of K values over the lanes of a warp by the tree lane l + lane l ^ 16, 8, ..., 1.
// Only half of the lanes' additions matter after the first step, a quarter
// after the second, and so on, so each step adds two values at once, one in the lanes
// whose step bit is clear and one in the others: with K = 5, 8 additions instead
// of 25 (and the same sums), which counts where an addition occupies the binary64
// pipe for 16 cycles.  The sum of value k ends in lane sum_lane(k).
__device__ __forceinline__ constexpr int sum_lane(int k) {
  return ((k & 1) << 4) | ((k & 2) << 2) | (k & 4) | ((k & 8) >> 2) | ((k & 16) >> 4);
}
__device__ __forceinline__ double sum_shfl(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
__device__ __forceinline__ dfloat sum_shfl(dfloat v, int off) {
  return dfloat{__shfl_xor_sync(0xffffffffu, v.hi, off), __shfl_xor_sync(0xffffffffu, v.lo, off)};
}
__device__ __forceinline__ double sum_add(double a, double b) { return a + b; }
__device__ __forceinline__ dfloat sum_add(dfloat a, dfloat b) { return df_add(a, b); }

template <int K, class V>
__device__ __forceinline__ V warp_sums(V (&v)[K]) {
  static_assert(K <= 32, "one value per lane");
  const int lane = threadIdx.x & 31;
  int n = K;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int p = 0; p < (K + 1) / 2; ++p) {
      if (2 * p + 1 < n) {
        const V keep = up ? v[2 * p + 1] : v[2 * p];
        const V send = up ? v[2 * p] : v[2 * p + 1];
        v[p] = sum_add(keep, sum_shfl(send, off));
      } else if (2 * p < n) {
        v[p] = sum_add(v[2 * p], sum_shfl(v[2 * p], off));
      }
    }
    n = (n + 1) / 2;
  }
  return v[0];
}

// Sum K values over the block (fixed shuffle tree, then warps in order).
// Result valid in thread 0.
template <int K, int NT>
__device__ __forceinline__ void block_sum(double (&v)[K]) {
  __shared__ double sm[NT / 32][K], out[K];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double t = warp_sums<K>(v);
  __syncthreads();  // sm may still be read by a previous call
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (lane == sum_lane(k)) sm[warp][k] = t;
  __syncthreads();
  if (threadIdx.x < 32) {
    if (threadIdx.x < K) {  // one thread per value
      double s = sm[0][threadIdx.x];
      for (int w = 1; w < NT / 32; ++w) s += sm[w][threadIdx.x];
      out[threadIdx.x] = s;
    }
    __syncwarp();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] = out[k];
    }
  }
}

// The first K entries of a longer array.
template <int K, int NT, int N>
__device__ __forceinline__ void block_sum_first(double (&v)[N]) {
  static_assert(K <= N, "block_sum_first: K exceeds the array");
  block_sum<K, NT>(*reinterpret_cast<double(*)[K]>(&v[0]));
}

template <int NT>
__device__ __forceinline__ double block_max(double v) {
  __shared__ double sm[NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, off));
  __syncthreads();
  if (lane == 0) sm[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < NT / 32; ++w) v = fmax(v, sm[w]);
    v = fmax(v, sm[0]);
  }
  return v;
}

// True in every thread of the last block of the grid (or of nblk blocks
// sharing the counter) to arrive.  The caller
// has written its partials before calling; the fence makes them visible.
__device__ __forceinline__ bool last_block_done(uint32_t* counter, uint32_t nblk) {
  __shared__ bool am_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) am_last = (atomicAdd(counter, 1u) == nblk - 1);
  __syncthreads();
  return am_last;
}
__device__ __forceinline__ bool last_block_done(uint32_t* counter) { return last_block_done(counter, gridDim.x); }

// In the last block: combine K partial sums of nblk blocks (layout
// part[b*stride + k]) in a fixed order.  Result valid in thread 0.
template <int K, int NT>
__device__ __forceinline__ void combine_partials(const double* part, int nblk, int stride, double (&out)[K]);
// Combined into the first K entries of a longer array (the rest set to zero).
template <int K, int NT, int N>
__device__ __forceinline__ void combine_partials_first(const double* part, int nblk, int stride, double (&out)[N]) {
  static_assert(K <= N, "combine_partials_first: K exceeds the array");
#pragma unroll
  for (int k = K; k < N; ++k) out[k] = 0.0;
  combine_partials<K, NT>(part, nblk, stride, *reinterpret_cast<double(*)[K]>(&out[0]));
}

template <int K, int NT>
__device__ __forceinline__ void combine_partials(const double* part, int nblk, int stride, double (&out)[K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = 0.0;
  for (int b = threadIdx.x; b < nblk; b += NT) {
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] += __ldcg(part + (size_t)b * stride + k);
  }
  block_sum<K, NT>(out);
}

template <int NT>
__device__ __forceinline__ double combine_max(const double* part, int nblk, int stride, int slot) {
  double m = 0.0;
  for (int b = threadIdx.x; b < nblk; b += NT) m = fmax(m, __ldcg(part + (size_t)b * stride + slot));
  return block_max<NT>(m);
}

// Compensated (two-sum) accumulation in binary32: the running error term
// keeps per-thread partial sums accurate to about 1e-14 relative.
struct Kahan32 {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float v) {
    float y = v - c;
    float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// Block sum of K compensated binary32 accumulators into binary64 (result in
// thread 0).  The warp tree adds the (s, -c) pairs in double-float arithmetic
// (binary32 operations only); the first warp widens all warps' pairs, one per lane,
// and adds the warps in order in binary64, one lane per value.  On GB300 the binary64
// pipe is slow (16 cycles per warp instruction, however few lanes take part), so
// this keeps the reduction off it.
template <int K, int NT, int N>
__device__ __forceinline__ void block_sum_kahan(const Kahan32 (&acc)[K], double (&out)[N]) {
  static_assert(K <= N, "block_sum_kahan: K exceeds the output");
  constexpr int W = NT / 32;
  __shared__ dfloat pair[W * K];
  __shared__ double wide[W * K], sum[K];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  dfloat v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = df_fast_two_sum(acc[k].s, -acc[k].c);
  const dfloat t = warp_sums<K>(v);
  __syncthreads();  // pair may still be read by a previous call
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (lane == sum_lane(k)) pair[warp * K + k] = t;
  __syncthreads();
  if (threadIdx.x < 32) {
    for (int i = lane; i < W * K; i += 32) wide[i] = (double)pair[i].hi + (double)pair[i].lo;
    __syncwarp();
    if (lane < K) {
      double s = wide[lane];
      for (int w = 1; w < W; ++w) s += wide[w * K + lane];
      sum[lane] = s;
    }
    __syncwarp();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int k = 0; k < K; ++k) out[k] = sum[k];
    }
  }
}

}  // namespace rec
