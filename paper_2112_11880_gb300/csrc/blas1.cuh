// Dot products and norms of short vectors as one launch without scratch
// (Section 3, Tables 5-7): one cluster of eight blocks whose sums meet in the
// first block's shared memory.
//
// The general path is two kernels over a scratch buffer.  At a few thousand
// elements that is two launches and an allocation for a microsecond's work.
// What bounds the cluster is the FP64 pipe of its eight SMs (a warp instruction
// takes 20 clocks, so a thread adds its own elements up rather than sum every 256
// over the warps) and, below, the chain from the loads to the result.  The line is
// where that pipe takes as long as the general path's second launch.
//
// Measured, n = 9,261 complex128: a dot product 6.1 us back to back, the launch
// included (every 256 elements summed over the warps as in the general path: 10.7);
// copy, axpy, scal, dot and norm of a first pass after a synchronisation, which
// gives the general path's scratch back to the driver, 297 -> 94 us.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"
#include "spmv.cuh"

namespace helm {

constexpr int kShortThreads = 256, kShortCluster = 8;
constexpr int64_t kShortMax = 32768;

// conj(x) y, x y and |x|^2 of one element added to v; complex64 products are FP32,
// their sums FP64.
struct ElemDotc {
  static constexpr int K = 2;
  __device__ static void add(double2 a, double2 b, double (&v)[2]) {
    a.y = -a.y;
    const double2 p = cfma(a, b, make_double2(v[0], v[1]));
    v[0] = p.x, v[1] = p.y;
  }
  __device__ static void add(float2 a, float2 b, double (&v)[2]) {
    a.y = -a.y;
    const float2 p = cfma32(a, b, make_float2(0.f, 0.f));
    v[0] += static_cast<double>(p.x), v[1] += static_cast<double>(p.y);
  }
};
struct ElemDotu {
  static constexpr int K = 2;
  __device__ static void add(double2 a, double2 b, double (&v)[2]) {
    const double2 p = cfma(a, b, make_double2(v[0], v[1]));
    v[0] = p.x, v[1] = p.y;
  }
  __device__ static void add(float2 a, float2 b, double (&v)[2]) {
    const float2 p = cfma32(a, b, make_float2(0.f, 0.f));
    v[0] += static_cast<double>(p.x), v[1] += static_cast<double>(p.y);
  }
};
struct ElemNorm {
  static constexpr int K = 1;
  __device__ static void add(double2 a, double2, double (&v)[1]) { v[0] = cabs2_acc(a, v[0]); }
  __device__ static void add(float2 a, float2, double (&v)[1]) {
    v[0] += static_cast<double>(fmaf(a.y, a.y, a.x * a.x));
  }
};

// Sum over the eight values of component k that lanes 8 k .. 8 k + 7 hold.
__device__ __forceinline__ double sum_of_8(double v) {
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

template <class V, class E>
__global__ void __cluster_dims__(kShortCluster, 1, 1) __launch_bounds__(kShortThreads)
    k_short_sum(int64_t n, const V* __restrict__ x, const V* __restrict__ y, double* out) {
  namespace cg = cooperative_groups;
  static_assert(kShortThreads == 8 * 32 && kShortCluster == 8, "sum_of_8 over warps, then blocks");
  constexpr int K = E::K, U = 4, T = kShortThreads * kShortCluster;
  __shared__ double part[8 * K];  // the first block's holds the blocks' sums
  __shared__ double red[8 * K];
  cg::cluster_group cl = cg::this_cluster();
  cl.barrier_arrive();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, m = static_cast<int>(n);
  double v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = 0.0;
#pragma unroll 1
  for (int i = static_cast<int>(blockIdx.x) * kShortThreads + static_cast<int>(threadIdx.x); i < m; i += U * T) {
    V a[U], b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      a[u] = b[u] = vzero<V>();
      if (i + u * T < m) {
        a[u] = ld_stream(x + i + u * T);
        if (K > 1) b[u] = ld_stream(y + i + u * T);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i + u * T < m) E::add(a[u], b[u], v);
  }
  const double ws = warp_sum_t<K>(v);
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (lane == warp_sum_lane<K>(k)) red[k * 8 + warp] = ws;
  __syncthreads();
  cl.barrier_wait();  // the first block has started: its shared memory can be written
  if (warp == 0) {
    const double s = sum_of_8(lane < 8 * K ? red[lane] : 0.0);
    if (lane < 8 * K && (lane & 7) == 0) cl.map_shared_rank(part, 0)[lane + blockIdx.x] = s;
  }
  cl.sync();
  if (blockIdx.x != 0 || warp != 0) return;
  const double s = sum_of_8(lane < 8 * K ? part[lane] : 0.0);
  if (lane < 8 * K && (lane & 7) == 0) out[lane >> 3] = K == 1 ? sqrt(s) : s;
}

// (x, y) and ||x|| of n <= kShortMax elements.
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
