// Dot products and norms of short vectors as one launch without scratch
// (Section 3, Tables 5-7): one cluster of eight blocks whose partial sums meet
// in the first block's shared memory.
//
// The general path is two kernels over a scratch buffer: blocks of 256 threads
// leave partial sums, one block adds them.  At a few thousand elements that is
// two launches and an allocation for a microsecond's work.  Here every group of
// 256 threads stands for a block of that path and adds the same elements in the
// same order, and the partials are added as there: the same bits.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"
#include "spmv.cuh"

namespace helm {

// Blocks of the general path that a cluster can stand for: one element per
// thread and one partial per thread of the final sum.
constexpr int kShortThreads = 1024, kShortCluster = 8, kShortBlocks = 256;
constexpr int64_t kShortMax = static_cast<int64_t>(kShortBlocks) * 256;

// conj(x) y, x y and |x|^2 of one element, as the general kernels form them.
struct ElemDotc {
  static constexpr int K = 2;
  template <class V> __device__ static void eval(const V* x, const V* y, int64_t i, double (&v)[2]) {
    V a = ld_stream(x + i);
    a.y = -a.y;
    const V p = mac(a, ld_stream(y + i), vzero<V>());
    v[0] = static_cast<double>(p.x), v[1] = static_cast<double>(p.y);
  }
};
struct ElemDotu {
  static constexpr int K = 2;
  template <class V> __device__ static void eval(const V* x, const V* y, int64_t i, double (&v)[2]) {
    const V p = mac(ld_stream(x + i), ld_stream(y + i), vzero<V>());
    v[0] = static_cast<double>(p.x), v[1] = static_cast<double>(p.y);
  }
};
struct ElemNorm {
  static constexpr int K = 1;
  template <class V> __device__ static void eval(const V* x, const V*, int64_t i, double (&v)[1]) {
    using S = decltype(V().x);
    const V a = ld_stream(x + i);
    v[0] = static_cast<double>(fma(a.y, a.y, fma(a.x, a.x, S(0))));
  }
};

template <class V, class E>
__global__ void __cluster_dims__(kShortCluster, 1, 1) __launch_bounds__(kShortThreads)
    k_short_sum(int64_t n, const V* __restrict__ x, const V* __restrict__ y, double* out) {
  namespace cg = cooperative_groups;
  constexpr int K = E::K;
  __shared__ double part[kShortBlocks * K];  // the first block's holds the partials
  __shared__ double red[32 * K];
  cg::cluster_group cl = cg::this_cluster();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = static_cast<int>((n + 255) / 256);
  double* first = cl.map_shared_rank(part, 0);
  cl.sync();  // the first block has started: its shared memory can be written
#pragma unroll 1
  for (int b0 = 4 * static_cast<int>(blockIdx.x); b0 < nb; b0 += 4 * kShortCluster) {
    const int64_t i = static_cast<int64_t>(b0) * 256 + threadIdx.x;
    double v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = 0.0;
    if (i < n) E::template eval<V>(x, y, i, v);
    const double ws = warp_sum_t<K>(v);
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (lane == warp_sum_lane<K>(k)) red[warp * K + k] = ws;
    __syncthreads();
    // warp q < 4: the sums of group q's eight warps in order, lane k component k
    if (warp < 4 && lane < K && b0 + warp < nb) {
      double s = 0.0;
#pragma unroll 1
      for (int w = 0; w < 8; ++w) s += red[(8 * warp + w) * K + lane];
      first[(b0 + warp) * K + lane] = s;
    }
    __syncthreads();
  }
  cl.sync();
  if (blockIdx.x != 0) return;
  // the final kernel: thread t takes partial t, then the tree of a 256-thread block
  if (warp < 8) {
    double v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = static_cast<int>(threadIdx.x) < nb ? part[threadIdx.x * K + k] : 0.0;
    const double ws = warp_sum_t<K>(v);
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (lane == warp_sum_lane<K>(k)) red[warp * K + k] = ws;
  }
  __syncthreads();
  if (threadIdx.x < K) {
    double s = 0.0;
#pragma unroll 1
    for (int w = 0; w < 8; ++w) s += red[w * K + threadIdx.x];
    out[threadIdx.x] = K == 1 ? sqrt(s) : s;
  }
}

// (x, y) of n <= kShortMax elements.
template <class V>
inline void launch_short_dot(int64_t n, const V* x, const V* y, bool conj, double* out, cudaStream_t s) {
  if (conj) k_short_sum<V, ElemDotc><<<kShortCluster, kShortThreads, 0, s>>>(n, x, y, out);
  else k_short_sum<V, ElemDotu><<<kShortCluster, kShortThreads, 0, s>>>(n, x, y, out);
}
template <class V>
inline void launch_short_norm(int64_t n, const V* x, double* out, cudaStream_t s) {
  k_short_sum<V, ElemNorm><<<kShortCluster, kShortThreads, 0, s>>>(n, x, x, out);
}

}  // namespace helm
