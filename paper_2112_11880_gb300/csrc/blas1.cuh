// Dot products and norms of short vectors as one launch without scratch
// (Section 3, Tables 5-7): one cluster of blocks whose sums meet in the first
// block's shared memory.
//
// The general path is two kernels over a scratch buffer.  At a few thousand
// elements that is two launches and an allocation for a microsecond's work.
// What bounds the cluster is the FP64 pipe of its SMs (a warp instruction takes 20
// clocks, so a thread adds its own elements up rather than sum every 256 over the
// warps) and, below, the chain from the loads to the result.  Eight blocks are what
// every device takes; above 8,192 elements (four of a thread) sixteen, eight where
// they are refused.
//
// Measured, complex128, us a dot product in a graph, two kernels / 8 blocks / 16: 9,261
// elements 4.9 / 4.9 / 3.6, 16,384 5.0 / 5.0 / 3.8, 24,000 5.0 / 6.2 / 5.2, 32,768 5.0
// / 7.2 / 5.1; called from Python at 32,768 25 / 9.9 / 7.8 (the general path
// allocates).  Copy, axpy, scal, dot and norm of 9,261 elements, a first pass after a
// synchronisation, which gives the general path's scratch back to the driver: 297 ->
// 94 us.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"
#include "spmv.cuh"

namespace helm {

constexpr int kShortThreads = 256, kShortCluster = 8, kShortWide = 16;
constexpr int64_t kShortMax = 32768, kShortNarrow = 8192;

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

// Sum over the C values of component k that lanes C k .. C k + C - 1 hold.
template <int C>
__device__ __forceinline__ double sum_of(double v) {
#pragma unroll
  for (int off = C / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// The sums by one cluster of C blocks.
template <class V, class E, int C>
__device__ __forceinline__ void short_sum(int64_t n, const V* __restrict__ x, const V* __restrict__ y, double* out) {
  namespace cg = cooperative_groups;
  constexpr int K = E::K, U = 4, T = kShortThreads * C;
  static_assert(kShortThreads == 8 * 32 && C * K <= 32, "sums over eight warps, then over C blocks in one warp");
  __shared__ double part[C * K];  // the first block's holds the blocks' sums
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
    const double s = sum_of<8>(lane < 8 * K ? red[lane] : 0.0);
    if (lane < 8 * K && (lane & 7) == 0) cl.map_shared_rank(part, 0)[(lane >> 3) * C + blockIdx.x] = s;
  }
  cl.sync();
  if (blockIdx.x != 0 || warp != 0) return;
  const double s = sum_of<C>(lane < C * K ? part[lane] : 0.0);
  if (lane < C * K && lane % C == 0) out[lane / C] = K == 1 ? sqrt(s) : s;
}
template <class V, class E>
__global__ void __cluster_dims__(kShortCluster, 1, 1) __launch_bounds__(kShortThreads)
    k_short_sum(int64_t n, const V* __restrict__ x, const V* __restrict__ y, double* out) {
  short_sum<V, E, kShortCluster>(n, x, y, out);
}
template <class V, class E>  // launched as one cluster of kShortWide
__global__ void __launch_bounds__(kShortThreads)
    k_short_sum_wide(int64_t n, const V* __restrict__ x, const V* __restrict__ y, double* out) {
  short_sum<V, E, kShortWide>(n, x, y, out);
}

template <class V, class E>
inline void launch_short_sum(int64_t n, const V* x, const V* y, double* out, cudaStream_t s) {
  if (n > kShortNarrow) {
    void (*fn)(int64_t, const V*, const V*, double*) = k_short_sum_wide<V, E>;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kShortWide;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kShortWide);
    cfg.blockDim = dim3(kShortThreads);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(reinterpret_cast<const void*>(fn), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
            cudaSuccess &&
        cudaLaunchKernelEx(&cfg, fn, n, x, y, out) == cudaSuccess)
      return;
    (void)cudaGetLastError();  // more than eight blocks are not every device's
  }
  k_short_sum<V, E><<<kShortCluster, kShortThreads, 0, s>>>(n, x, y, out);
}
// (x, y) and ||x|| of n <= kShortMax elements.
template <class V>
inline void launch_short_dot(int64_t n, const V* x, const V* y, bool conj, double* out, cudaStream_t s) {
  if (conj) launch_short_sum<V, ElemDotc>(n, x, y, out, s);
  else launch_short_sum<V, ElemDotu>(n, x, y, out, s);
}
template <class V>
inline void launch_short_norm(int64_t n, const V* x, double* out, cudaStream_t s) {
  launch_short_sum<V, ElemNorm>(n, x, x, out, s);
}

}  // namespace helm
