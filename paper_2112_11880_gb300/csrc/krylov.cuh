// BiCGStab kernels with device-resident scalars, generic over the vector
// precision (complex128 for the FP64 solver, complex64 for the inner solve of
// mixed precision).  Section 4 of the paper: P-BiCGSTAB with residual
// tolerance, zero initial guess and an iteration cap; identity preconditioner
// (right Jacobi runs the same kernels on A D^-1); the recurrence of van der
// Vorst 1992 / Saad 2003 Algorithm 7.7 with conjugated inner products.
//
// One iteration is five phases; each dot product the recurrence needs is
// fused into the phase that produces its operands, and the scalar it feeds
// is formed in FP64 on the device:
//   P1  p = r + beta (p - omega v)
//   P2  v = A p          + (r^, v)        -> alpha = rho / (r^, v)
//   P3  s = r - alpha v  + ||s||^2        -> stop at s if ||s|| / ||b|| <= tol
//   P4  t = A s          + (t, s), ||t||^2 -> omega = (t, s) / (t, t)
//   P5  x += alpha p + omega s, r = s - omega t + (r^, r), ||r||^2
//                                         -> stop test, rho, beta
// For complex64 the products are FP32; each thread's partial sums, block and grid
// sums and every scalar of the recurrence are FP64.
//
// Three ways to run the loop, with the same arithmetic bit for bit:
//   * persistent (the default but for long rows, and for complex64 on the smallest
//     and the large meshes): one cooperative kernel for the whole solve; a grid
//     barrier ends every phase, after which every block adds the block partials
//     itself (same order, so the same scalars in every block) -- no kernel
//     launches, no last-block step;
//   * graph: one kernel per phase; the last block to finish a phase (ticket
//     counter) adds the block partials and forms the scalars; the loop is a
//     CUDA graph with a conditional WHILE node (four iterations per pass);
//   * host: the graph's kernels launched from the host (for profilers).
// All give each row to the same thread in every phase (SliceRows of the
// SpMV engine) on the same grid, and add the same partials in the same order.
#pragma once

#include <algorithm>
#include <type_traits>
#include <cstring>
#include <initializer_list>
#include <utility>
#include <vector>

#include "common.cuh"
#include "internal.hpp"
#include "persist.cuh"
#include "spmv.cuh"

namespace helm {

// The complex128 matrix a solve runs on: A, or A D^-1 under right Jacobi.
inline CsrDev<double2> csr_for(helm_csr A, const helm_opts& o) {
  if (o.precond == HELM_PRECOND_JACOBI) return csr_dev<double2>(A, A->jac_vals, A->svjac);
  return csr_dev<double2>(A, static_cast<const double2*>(A->vals), A->sv);
}

// SolverState::method of the Krylov loop: plain, or the inner loop of the
// mixed-precision solve (aux[0] = (||r|| when the process began, in its
// scale; iteration it began), aux[1].x = refinement step due, aux[2].x =
// scale of the inner residual, aux[3] = (steps in a row without a 2x gain,
// inner_tol)).
constexpr int32_t kModePlain = 0;
constexpr int32_t kModeRefine = 1;
constexpr int kInnerMax = 50000;  // inner iterations per refinement step at most

// Per-thread partial sums of dot products and norms accumulate in FP64: for complex128 operands the FP64 product (4 or 2 FMA),
// for complex64 operands the product formed in FP32 and added in FP64.
// Measured alternatives for complex64: an uncompensated FP32 running sum
// over the ~10 rows a thread takes on the 200x100x80 cavity slowed the inner
// solves of mixed precision visibly; a compensated (Kahan) FP32 sum made an
// inner iteration 2-6 % faster on the 120x60x50 and 200x100x80 cavities, but
// the 200x100x80 solve to 1e-10 then stalled (289,524 inner iterations, not
// converged, against 188,207 to convergence with FP64 sums).
// A device scalar in the precision of the vectors.
template <class V> struct Prec;
template <> struct Prec<double2> {
  __device__ static __forceinline__ double2 cvt(double2 z) { return z; }
};
template <> struct Prec<float2> {
  __device__ static __forceinline__ float2 cvt(double2 z) {
    return make_float2(static_cast<float>(z.x), static_cast<float>(z.y));
  }
};

// acc + conj(a) b and acc + |a|^2 in the precision rules above
__device__ __forceinline__ double2 dot_acc(double2 acc, double2 a, double2 b) { return cfma_conj(a, b, acc); }
__device__ __forceinline__ double2 dot_acc(double2 acc, float2 a, float2 b) {
  const float re = fmaf(a.x, b.x, a.y * b.y);
  const float im = fmaf(a.x, b.y, -a.y * b.x);
  return make_double2(acc.x + static_cast<double>(re), acc.y + static_cast<double>(im));
}
__device__ __forceinline__ double nrm_acc(double acc, double2 a) { return cabs2_acc(a, acc); }
__device__ __forceinline__ double nrm_acc(double acc, float2 a) {
  return acc + static_cast<double>(fmaf(a.x, a.x, a.y * a.y));
}

// Solver shapes, by the slices of the mesh per SM (krylov_shapes).  The shape
// fixes which thread owns which row, in how many parts a row is summed, and so
// the rounding of every reduction: every form of a solve takes the same one, and
// it depends on nothing but the size, so that a solve gives the same bits on
// every run.
//   small: one block per SM; a row is summed in kParts parts, which the
//          persistent kernel gives to three warps;
//   mid:   one block per SM of at most 768 threads (80 registers a thread);
//   large: two blocks per SM of at most 512 threads (64 registers).
// complex64 (the inner solves of mixed precision): mid or large (us per inner
// iteration, persistent / graph / before: 20^3 29.7 / 33.9 / 44.5, 60x30x25 29.4 /
// 34.5 / 37.1, 80x40x32 37.6 / 44.9 / 47; large: 120x60x50 71.5 / 67.8 / 77.9,
// 200x100x80 191 / 171 / 205: there the default is the graph).
// Measured (BiCGStab, us per iteration: persistent / graph kernels; before, on
// one shape with graph kernels):
//   20^3 box      (2 slices per SM)  small 25.8 / 35.4                       (49.4)
//   60x30x25      (10)               mid   36.2 / 39.6, large 50.1 / 47.6    (46.5)
//   80x40x32      (23)               mid   53.9 / 58.9, large 60.0 / 67.0    (66.3)
//   120x60x50     (77)               mid  121.6 / 133.1, large 135.4 / 140.2 (139.1)
//   200x100x80    (338)              mid  504 (512 threads), large 474 / 472 (488)
// (mid of 640 threads: 37.3, 55.1, 121.5; 704: 40.5, 61.0, 124.1; more spill.  The
// figures of a shape a mesh does not take are of a graph without loads ahead.)
enum : int { SHAPE_SMALL = 0, SHAPE_MID = 1, SHAPE_LARGE = 2 };
constexpr int kMidSlices = 150;    // slices per SM from which the shape is large
// for complex64 sooner: whether its inner solves converge on an indefinite system
// of that size hangs on the order of their sums (kOrderedSums; 120x60x50 at 10
// points per wavelength, inner_tol 0.01: converges on the large shape, not on mid).
// Up to 50 slices either order converges: 30x15x12 to 104x52x42 (49.2 slices) at 8, 10
// and 14 points per wavelength, to 1e-8 and 1e-10, inner_tol 0.5 to 1e-4, 336 solves,
// all of them with both, the inner iterations within 0.4 % on average
constexpr int kMidSlices32 = 50;
template <int S> struct SolverBounds {
  static constexpr int threads = S == SHAPE_SMALL ? 384 : S == SHAPE_MID ? 768 : 512;  // warps of a split persistent kernel included
  static constexpr int blocks = S == SHAPE_LARGE ? 2 : 1;
  static constexpr int parts = S == SHAPE_SMALL ? kParts : 1;
  // entries per pipeline stage of the persistent kernel's products
  static constexpr int persist_u = S == SHAPE_LARGE ? 2 : 3;
};
template <class V>
struct KArgs {
  CsrDev<V> A;
  const V* b;
  V* x;
  V *r, *rh, *p, *v, *s, *t;
  SolverState* st;
  double* partials;
  unsigned int* tickets;
  unsigned int* dev_err;
  cudaGraphConditionalHandle cond;
  int has_cond;
};

template <class V>
__device__ __forceinline__ void set_cond(const KArgs<V>& a, bool cont) {
  if (a.has_cond) cudaGraphSetConditional(a.cond, cont ? 1u : 0u);
}

__device__ __forceinline__ bool deadline_passed(const SolverState* st) {
  return st->deadline_ns != 0ull && (globaltimer_ns() - st->t0) > st->deadline_ns;
}

__global__ void k_configure(SolverState* st, double tol, int32_t maxit, int32_t use_x0, double deadline_s,
                            int32_t fresh);

// Programmatic dependent launch.  The loop's kernels are launched so that a
// kernel's blocks may be scheduled while its predecessor is still running:
// they take the SMs that the predecessor's blocks leave while its last block
// forms the scalars, and wait here until the predecessor grid has completed
// and its writes are visible.  Every kernel of the loop calls this before it
// reads anything, so the order of every operation is that of plain launches
// (with a plain launch the wait returns at once).  Each grid is one wave, so
// the waiting blocks never hold an SM that a block of the predecessor needs.
// Measured on the 120x60x50 cavity (BiCGStab, 19,653 iterations): the
// host-driven loop 148.6 -> 141.4 us per iteration; the graph (the WHILE
// node, or a plain graph of 16 iterations) 138.1 us either way, although its
// body keeps the programmatic edges: a graph launch already hides that gap.
#ifndef HELM_PDL
#define HELM_PDL 1
#endif
__device__ __forceinline__ void pdl_enter() {
#if HELM_PDL
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}

// ---------------------------------------------------------------- reductions

// Two orders of a grid's sums.  One is chosen for latency (a dependent FP64 add
// is 64 clocks): trees over warps and blocks with the components side by side
// on the warps; partials: component k of block b at k G + b (every block of a
// persistent solve reads them all: neighbours share a sector).  The other, for
// complex64 on the large shape: warps in order, then blocks in thread order;
// whether the inner solves of mixed precision converge on a strongly indefinite
// system of that size (200x100x80 at 10 points per wavelength) hangs on the last
// bits of these sums, so their order stays.
template <class V, int S>
constexpr bool kOrderedSums = std::is_same<V, float2>::value && S == SHAPE_LARGE;

// Sums of the first `width` lanes (a power of two) into lane 0, in the order
// that the pattern fixes.
__device__ __forceinline__ double lanes_sum(double v, int width) {
#pragma unroll 1
  for (int off = width >> 1; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// This block's K sums into its partials (global memory; a barrier of the block
// or a fence has to follow).  `red` holds 32 * K doubles.
template <class V, int S, int K>
__device__ __forceinline__ void put_block_partials(double (&v)[K], double* red, double* partials) {
  if constexpr (kOrderedSums<V, S>) {
    block_sum<K>(v, red);
    if (threadIdx.x == 0)
#pragma unroll
      for (int k = 0; k < K; ++k) partials[static_cast<size_t>(blockIdx.x) * K + k] = v[k];
  } else {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = static_cast<int>(blockDim.x >> 5);
    const double ws = warp_sum_t<K>(v);
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (lane == warp_sum_lane<K>(k)) red[warp * K + k] = ws;
    __syncthreads();
    const int width = nwarps > 1 ? 1 << (32 - __clz(nwarps - 1)) : 1;
#pragma unroll 1
    for (int k = warp; k < K; k += nwarps) {
      const double s = lanes_sum(lane < nwarps ? red[lane * K + k] : 0.0, width);
      if (lane == 0) partials[static_cast<size_t>(k) * gridDim.x + blockIdx.x] = s;
    }
  }
}

// out[k] = sum over the blocks of component k's partials, k < K: one warp per
// component, lane j adds blocks j, j + 32, j + 64, ... (five loaded at a time) in
// that order, then the lanes' tree.  Whole block; ends with its barrier.
__device__ __forceinline__ void sum_components(const double* partials, int G, int K, double* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = static_cast<int>(blockDim.x >> 5);
#pragma unroll 1
  for (int k = warp; k < K; k += nwarps) {
    double acc = 0.0;
#pragma unroll 1
    for (int j0 = lane; j0 < G; j0 += 5 * 32) {
      double w[5];
#pragma unroll
      for (int u = 0; u < 5; ++u)
        w[u] = j0 + 32 * u < G ? ld_cg(&partials[static_cast<size_t>(k) * G + j0 + 32 * u]) : 0.0;
#pragma unroll
      for (int u = 0; u < 5; ++u)
        if (j0 + 32 * u < G) acc += w[u];
    }
    acc = lanes_sum(acc, 32);
    if (lane == 0) out[k] = acc;
  }
  __syncthreads();
}

// put_block_partials and sum_components where a block is one warp, which would add
// the components one after the other: the same sums, the components side by side
// (graph kernels of meshes up to one slice per SM: us per iteration of the 15^3 box,
// BiCGStab 36.4 -> 35.0, complex64 33.4 -> 32.6).
template <int K>
__device__ __forceinline__ void put_warp_partials(const double (&v)[K], double* partials) {
  const int lane = threadIdx.x & 31;
  const double ws = warp_sum_t<K>(v);
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (lane == warp_sum_lane<K>(k)) partials[static_cast<size_t>(k) * gridDim.x + blockIdx.x] = ws;
}
// (out of line: the kernels of larger meshes on the same shape do not fetch it)
template <int K>
__device__ __noinline__ double4 sum_warp_partials(const double* partials, int G) {
  static_assert(K <= 4, "four at most");
  const int lane = threadIdx.x & 31;
  double tot[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int j0 = lane; j0 < G; j0 += 5 * 32) {
    double w[K][5];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int u = 0; u < 5; ++u)
        w[k][u] = j0 + 32 * u < G ? ld_cg(&partials[static_cast<size_t>(k) * G + j0 + 32 * u]) : 0.0;
#pragma unroll
    for (int u = 0; u < 5; ++u)
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (j0 + 32 * u < G) tot[k] += w[k][u];
  }
  __syncwarp();
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int k = 0; k < K; ++k) tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], off);
  return make_double4(tot[0], tot[1], tot[2], tot[3]);
}

// Fixed-order totals of all blocks' partials, valid in thread 0: sum_components,
// or thread j adds blocks j, j + T, ..., then the block tree.
template <class V, int S, int K>
__device__ __forceinline__ void sum_block_partials(const double* partials, int G, double* red, double (&tot)[K]) {
  if constexpr (kOrderedSums<V, S>) {
    double acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    for (int b = threadIdx.x; b < G; b += blockDim.x)
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] += ld_cg(&partials[static_cast<size_t>(b) * K + k]);
    block_sum<K>(acc, red);
#pragma unroll
    for (int k = 0; k < K; ++k) tot[k] = acc[k];
  } else {
    __shared__ double out[K];
    sum_components(partials, G, K, out);
    if (threadIdx.x == 0) {
#pragma unroll
      for (int k = 0; k < K; ++k) tot[k] = out[k];
    }
  }
}

// Graph path: publish this block's K sums; the last block to arrive forms
// the totals (valid in its thread 0) and returns true.
template <class V, int S, int K>
__device__ __forceinline__ bool grid_total_last(double (&v)[K], double* partials, unsigned int* ticket, double* red,
                                                double (&tot)[K]) {
  __shared__ bool s_last;
  // only the shape of the smallest meshes has one-warp blocks
  constexpr bool can = S == (std::is_same<V, float2>::value ? SHAPE_MID : SHAPE_SMALL);
  const bool one_warp = can && blockDim.x == 32;
  if (one_warp) put_warp_partials<K>(v, partials);
  else put_block_partials<V, S, K>(v, red, partials);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  if (one_warp) {
    const double4 t = sum_warp_partials<K>(partials, gridDim.x);
    const double t4[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int k = 0; k < K; ++k) tot[k] = t4[k];
  } else sum_block_partials<V, S, K>(partials, gridDim.x, red, tot);
  if (threadIdx.x == 0) *ticket = 0u;
  return true;
}

// Persistent path: publish this block's K sums, wait for every block, add all
// blocks' sums in the same order (every block the same), totals valid in
// thread 0; false when the barrier gave up.
template <class V, int S, int K>
__device__ __forceinline__ bool grid_total_all(double (&v)[K], double* partials, unsigned int* tickets,
                                               unsigned int* dev_err, unsigned int* target, double* red,
                                               double (&tot)[K]) {
  put_block_partials<V, S, K>(v, red, partials);
  if (!grid_barrier(tickets, dev_err, target)) return false;
  sum_block_partials<V, S, K>(partials, gridDim.x, red, tot);
  return true;
}

// ---------------------------------------------------------------- scalar steps
// Executed by one thread on the state (in global memory for the graph path,
// in each block's shared memory for the persistent one).

// The inner loop of mixed precision does not end the solve on a breakdown or
// a non-finite scalar of its complex64 recurrence: it asks for a refinement
// step instead (the FP64 step minimises the residual over its window, so a
// poor or non-finite inner iterate is rejected there, and a fresh inner
// process starts from the FP64 residual).  Returns true when the event was
// absorbed that way; the caller then leaves the status running.
template <class V>
__device__ __forceinline__ bool refine_absorb(SolverState* st) {
  if (std::is_same<V, double2>::value || st->method != kModeRefine) return false;
  st->aux[1].x = 1.0;
  return true;
}
// A refinement step is pending: the rest of the inner iteration is skipped.
template <class V>
__device__ __forceinline__ bool refine_step_pending(const SolverState* st) {
  return !std::is_same<V, double2>::value && st->method == kModeRefine && st->aux[1].x != 0.0;
}

// after the initial residual: tot = (||b||^2, ||r||^2, (r^, r))
__device__ __forceinline__ void sc_init(SolverState* st, const double (&tot)[4], int use_x0) {
  const double bnorm = sc_sqrt(tot[0]);
  st->bnorm = bnorm;
  if (use_x0) st->spmv_count += 1;
  int status = ST_RUNNING;
  if (!isfinite(bnorm)) {
    status = HELM_ERR_NONFINITE;
  } else if (bnorm == 0.0) {
    status = HELM_OK;  // b = 0: x = 0 (written by the tail)
    st->relres = 0.0;
  } else {
    const double relres = sc_div(sc_sqrt(tot[1]), bnorm);
    st->relres = relres;
    const double2 rho = make_double2(tot[2], tot[3]);
    if (!isfinite(relres)) {
      status = HELM_ERR_NONFINITE;
    } else if (relres <= st->tol) {
      status = HELM_OK;
    } else if (st->iter >= st->maxit) {
      status = HELM_ERR_NOT_CONVERGED;
    } else if (!cfinite(rho)) {
      status = HELM_ERR_NONFINITE;
      st->iter += 1;
    } else if (czero(rho)) {
      status = HELM_ERR_BREAKDOWN;
      st->iter += 1;
    } else {
      // beta = (rho / 1) (1 / 1): the first p update gives p = r
      st->rho = rho;
      st->beta = rho;
      st->omega = make_double2(1.0, 0.0);
      st->alpha = make_double2(1.0, 0.0);
    }
  }
  st->phase = PH_RUN;
  st->status = status;
}

// after P2: tot = (r^, v)
template <class V>
__device__ __forceinline__ void sc_after_v(SolverState* st, const double (&tot)[2]) {
  st->iter += 1;
  st->spmv_count += 1;
  const double2 rv = make_double2(tot[0], tot[1]);
  int err = 0;
  if (!cfinite(rv)) {
    err = HELM_ERR_NONFINITE;
  } else if (czero(rv)) {
    err = HELM_ERR_BREAKDOWN;
  } else {
    const double2 alpha = cdiv_fast(st->rho, rv);
    if (!cfinite(alpha)) err = HELM_ERR_NONFINITE;
    else st->alpha = alpha;
  }
  if (err && !refine_absorb<V>(st)) st->status = err;
}

// after P3: tot = ||s||^2; ||s|| / ||b|| <= tol compared squared
template <class V>
__device__ __forceinline__ void sc_after_s(SolverState* st, const double (&tot)[1]) {
  const double s2 = tot[0];
  const double bt = st->bnorm * st->tol;
  if (!isfinite(s2)) {
    if (!refine_absorb<V>(st)) st->status = HELM_ERR_NONFINITE;
  } else if ((std::is_same<V, double2>::value || st->method != kModeRefine) && s2 <= bt * bt) {
    st->phase = PH_SCONV;
    st->relres = sc_div(sc_sqrt(s2), st->bnorm);
  }
}

// after P4: tot = ((t, s), ||t||^2)
template <class V>
__device__ __forceinline__ void sc_after_t(SolverState* st, const double (&tot)[3]) {
  st->spmv_count += 1;
  const double2 ts = make_double2(tot[0], tot[1]);
  const double tt = tot[2];
  int err = 0;
  if (!cfinite(ts) || !isfinite(tt)) {
    err = HELM_ERR_NONFINITE;
  } else if (tt == 0.0) {
    err = HELM_ERR_BREAKDOWN;
  } else {
    const double inv_tt = sc_div(1.0, tt);
    const double2 omega = make_double2(ts.x * inv_tt, ts.y * inv_tt);
    if (!cfinite(omega)) err = HELM_ERR_NONFINITE;
    else st->omega = omega;
  }
  if (err && !refine_absorb<V>(st)) st->status = err;
}

// after P5: tot = ((r^, r), ||r||^2); `late` = the deadline has passed.
// With phase PH_SCONV (P5 only added alpha p to x) the solve is done.
template <class V>
__device__ __forceinline__ void sc_after_xr(SolverState* st, const double (&tot)[3], bool late) {
  // the inner loop of mixed precision runs on a scaled residual: b - A x ~ aux[2].x * r
  constexpr bool plain = std::is_same<V, double2>::value;
  const double sc = !plain && st->method == kModeRefine ? st->aux[2].x : 1.0;
  const int phase = st->phase;
  const double2 alpha64 = st->alpha, omega64 = st->omega;
  int status = ST_RUNNING;
  if (phase == PH_SCONV) {
    status = HELM_OK;
    st->phase = PH_DONE;
  } else {
    // ||r|| / ||b|| <= tol compared squared; the square root is taken for the
    // report only when the loop stops
    const double r2 = tot[2];
    const double bt = st->bnorm * st->tol;
    bool stop_ok = r2 * (sc * sc) <= bt * bt;
    if (!plain && st->method == kModeRefine && isfinite(r2)) {
      // mixed precision: the recurrence never declares convergence; it asks
      // for a refinement step (FP64 residual, fresh process) when it has
      // dropped by inner_tol since the process began, looks converged, or
      // after kInnerMax iterations (complex64 BiCGStab can stagnate on
      // strongly indefinite systems; the step's minimal-residual length
      // keeps a poor inner iterate from increasing the FP64 residual)
      const double rn = sc_sqrt(r2);
      const double cyc = st->aux[3].y;
      const bool dropped = cyc > 0.0 && cyc < 1.0 && rn <= cyc * st->aux[0].x;
      if (stop_ok || dropped || st->iter - static_cast<int>(st->aux[0].y) >= kInnerMax) st->aux[1].x = 1.0;
      stop_ok = false;
    }
    if (!isfinite(r2)) {
      status = refine_absorb<V>(st) ? ST_RUNNING : HELM_ERR_NONFINITE;
    } else if (stop_ok) {
      status = HELM_OK;
    } else if (czero(omega64)) {
      status = refine_absorb<V>(st) ? ST_RUNNING : HELM_ERR_BREAKDOWN;
    } else if (st->iter >= st->maxit) {
      status = HELM_ERR_NOT_CONVERGED;
    } else if (late) {
      status = HELM_ERR_TIMEOUT;
    } else {
      const double2 rho_new = make_double2(tot[0], tot[1]);
      // beta = (rho_new / rho) (alpha / omega) = (rho_new alpha) / (rho omega)
      const double2 beta = cdiv_fast(cmul(rho_new, alpha64), cmul(st->rho, omega64));
      if (!cfinite(rho_new) || !cfinite(beta)) {
        status = refine_absorb<V>(st) ? ST_RUNNING : HELM_ERR_NONFINITE;
        st->iter += 1;
      } else if (czero(rho_new)) {
        // (r^, r) has sunk below the rounding of its terms and they cancelled:
        // the process can go no further, x and r stand.  Start again from x
        // (r^ = r); what is left in (r^, r) at such a point, zero or not, is the
        // luck of the order of the sum.
        status = refine_absorb<V>(st) ? ST_RUNNING : ST_RESTART;
        st->iter += 1;
      } else {
        st->rho = rho_new;
        st->beta = beta;
      }
    }
    if (status != ST_RUNNING) st->relres = sc_div(sc_sqrt(tot[2]) * sc, st->bnorm);
  }
  st->status = status;
}

// after the tail: tot = ||b - A x||^2
__device__ __forceinline__ void sc_tail(SolverState* st, const double (&tot)[1]) {
  if (st->bnorm == 0.0) {
    st->relres_true = 0.0;
  } else {
    st->relres_true = sc_div(sc_sqrt(tot[0]), st->bnorm);
    st->spmv_count += 1;
  }
}

// After the tail: the recurrence converged but the true residual did not, or
// (r^, r) vanished; the solve starts again from x while iterations remain.
__host__ __device__ __forceinline__ bool restart_due(SolverState* st) {
  if (st->status == ST_RESTART && st->relres_true <= st->tol) st->status = HELM_OK;
  if (st->status == ST_RESTART && st->iter >= st->maxit) st->status = HELM_ERR_NOT_CONVERGED;
  return st->status == ST_RESTART || (st->status == HELM_OK && st->relres_true > st->tol && st->iter < st->maxit);
}

// The state of a solve that starts again from x (k_configure with fresh = 0).
__device__ __forceinline__ void restart_state(SolverState* st) {
  const double2 one = make_double2(1.0, 0.0);
  st->restarts += 1;
  st->use_x0 = 1;
  st->status = ST_RUNNING;
  st->phase = PH_RUN;
  st->relres = 0.0;
  st->relres_true = 0.0;
  st->rho = one;
  st->alpha = one;
  st->omega = one;
  st->beta = make_double2(0.0, 0.0);
}

// ---------------------------------------------------------------- phases
// The per-thread work of each phase, shared by the graph kernels and the
// persistent kernels; each returns this thread's partial sums.  Rows are those
// of SliceRows.
template <class V>
struct Phases {
  const KArgs<V>& a;
  PRows q;
  Own<V, 0> v;
  Own<V, 1> r;
  Own<V, 2> t;
  Own<V, 3> rh;
  Own<V, 4> x;
  Own<V, 5> p;  // p and s: a copy beside the one that is gathered
  Own<V, 6> s;
  static constexpr int kOwn = 7;
  __device__ __forceinline__ Phases(const KArgs<V>& a_, const PLayout& L)
      : a(a_), q(L), v{a_.v, L}, r{a_.r, L}, t{a_.t, L}, rh{a_.rh, L}, x{a_.x, L}, p{a_.p, L}, s{a_.s, L} {}

  __device__ __forceinline__ int32_t n() const { return a.A.n; }

  // r = r^ = ri, p = v = 0 on row i; (||b||^2, ||r||^2, (r^, r))
  __device__ __forceinline__ void init_row(int32_t i, int li, V bi, V ri, double (&part)[4]) const {
    const V z = vzero<V>();
    r.st(i, li, ri);
    rh.st(i, li, ri);
    p.st(i, li, z);
    v.st(i, li, z);
    part[0] = nrm_acc(part[0], bi);
    part[1] = nrm_acc(part[1], ri);
    const double2 d = dot_acc(make_double2(part[2], part[3]), ri, ri);
    part[2] = d.x;
    part[3] = d.y;
  }
  // without x0: x = 0, r = b
  __device__ __forceinline__ void init_zero(double (&part)[4]) const {
    for_rows(q, n(), [&](int32_t i, int li) {
      const V bi = a.b[i];
      x.st(i, li, vzero<V>());
      init_row(i, li, bi, bi, part);
    });
  }
  // with x0: r = b - A x
  __device__ __forceinline__ void row_init(int32_t i, int li, V ax, double (&part)[4]) const {
    const V bi = a.b[i];
    if (x.shared()) x.st(i, li, a.x[i]);
    init_row(i, li, bi, csub(bi, ax), part);
  }

  // P1: p = r + beta (p - omega v)
  template <bool AHEAD>
  __device__ __forceinline__ void upd_p(V beta, V omega) const {
    struct Ops { V v, p, r; };
    for_rows_ld<AHEAD>(
        q, n(), [&](int32_t i, int li) { return Ops{v.ld(i, li), p.ld(i, li), r.ld(i, li)}; },
        [&](int32_t i, int li, const Ops& o) { p.st_both(i, li, cfma(beta, cfms(omega, o.v, o.p), o.r)); });
  }

  // P2: v = A p, (r^, v)
  __device__ __forceinline__ void row_v(int32_t i, int li, V rhi, V ax, double (&part)[4]) const {
    v.st(i, li, ax);
    const double2 d = dot_acc(make_double2(part[0], part[1]), rhi, ax);
    part[0] = d.x;
    part[1] = d.y;
  }

  // P3: s = r - alpha v, ||s||^2
  template <bool AHEAD>
  __device__ __forceinline__ void upd_s(V alpha, double (&part)[4]) const {
    struct Ops { V v, r; };
    for_rows_ld<AHEAD>(
        q, n(), [&](int32_t i, int li) { return Ops{v.ld(i, li), r.ld(i, li)}; },
        [&](int32_t i, int li, const Ops& o) {
          const V sn = cfms(alpha, o.v, o.r);
          s.st_both(i, li, sn);
          part[0] = nrm_acc(part[0], sn);
        });
  }

  // P4: t = A s, (t, s), ||t||^2
  __device__ __forceinline__ void row_t(int32_t i, int li, V si, V ax, double (&part)[4]) const {
    t.st(i, li, ax);
    const double2 d = dot_acc(make_double2(part[0], part[1]), ax, si);
    part[0] = d.x;
    part[1] = d.y;
    part[2] = nrm_acc(part[2], ax);
  }

  // P5: x += alpha p + omega s, r = s - omega t; (r^, r), ||r||^2.  With sconv
  // (the solve stopped at s) only x += alpha p.
  template <bool AHEAD>
  __device__ __forceinline__ void upd_xr(V alpha, V omega, bool sconv, double (&part)[4]) const {
    if (sconv) {
      for_rows(q, n(), [&](int32_t i, int li) { x.st(i, li, cfma(alpha, p.ld(i, li), x.ld(i, li))); });
      return;
    }
    auto dots = [&](V rhi, V ri) {
      const double2 d = dot_acc(make_double2(part[0], part[1]), rhi, ri);
      part[0] = d.x;
      part[1] = d.y;
      part[2] = nrm_acc(part[2], ri);
    };
    if constexpr (AHEAD) {
      struct Ops { V s, p, x, t, rh; };
      for_rows_ld<true>(
          q, n(),
          [&](int32_t i, int li) { return Ops{s.ld(i, li), p.ld(i, li), x.ld(i, li), t.ld(i, li), rh.ld(i, li)}; },
          [&](int32_t i, int li, const Ops& o) {
            x.st(i, li, cfma(omega, o.s, cfma(alpha, o.p, o.x)));
            const V ri = cfms(omega, o.t, o.s);
            r.st(i, li, ri);
            dots(o.rh, ri);
          });
    } else {
      // operands as they are needed: five at once cost the persistent kernel up to
      // 0.8 % (200x100x80 471.5 -> 475 us an iteration)
      for_rows(q, n(), [&](int32_t i, int li) {
        const V si = s.ld(i, li);
        x.st(i, li, cfma(omega, si, cfma(alpha, p.ld(i, li), x.ld(i, li))));
        const V ri = cfms(omega, t.ld(i, li), si);
        r.st(i, li, ri);
        dots(rh.ld(i, li), ri);
      });
    }
  }
};

// ---------------------------------------------------------------- graph kernels

// no shared memory: the rounds of the grid, whose blocks' warps all own rows
__device__ __forceinline__ PLayout graph_layout(int32_t n) {
  const int32_t wb = static_cast<int32_t>(blockDim.x >> 5), W = static_cast<int32_t>(gridDim.x) * wb;
  PLayout L = {};
  L.rounds = ((n + 31) / 32 + W - 1) / W;
  L.split = 1;
  L.warps = wb;
  return L;
}
template <class V, int S, class Pre, class F>
__device__ __forceinline__ void graph_spmv(const Phases<V>& ph, const V* x, Pre pre, F f) {
  spmv_rows<V, kSpmvUnroll, SolverBounds<S>::parts, GatherReadOnly>(ph.q, ph.a.A, x, pre, f);
}

#define HELM_SOLVER_KERNEL __global__ void __launch_bounds__(SolverBounds<S>::threads, SolverBounds<S>::blocks)
#define HELM_GRAPH_PHASES                     \
  const PLayout lay = graph_layout(a.A.n);    \
  const Phases<V> ph(a, lay);                 \
  double part[4] = {0.0, 0.0, 0.0, 0.0};

template <class V, int S>
HELM_SOLVER_KERNEL k_init(const __grid_constant__ KArgs<V> a) {
  pdl_enter();
  __shared__ double red[32 * 4];
  SolverState* st = a.st;
  const int use_x0 = st->use_x0;
  HELM_GRAPH_PHASES
  if (use_x0) {
    graph_spmv<V, S>(
        ph, a.x, [](int32_t) {}, [&](int32_t i, int li, V ax) { ph.row_init(i, li, ax, part); });
  } else {
    ph.init_zero(part);
  }
  double tot[4];
  if (!grid_total_last<V, S, 4>(part, a.partials, a.tickets + TK_INIT, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_init(st, tot, use_x0);
  set_cond(a, st->status == ST_RUNNING);
}

// K1: p = r + beta (p - omega v)
template <class V, int S>
HELM_SOLVER_KERNEL k_p(const __grid_constant__ KArgs<V> a) {
  pdl_enter();
  const SolverState* st = a.st;
  if (st->status != ST_RUNNING || refine_step_pending<V>(st)) return;
  const PLayout lay = graph_layout(a.A.n);
  Phases<V>(a, lay).template upd_p<true>(Prec<V>::cvt(st->beta), Prec<V>::cvt(st->omega));
}

// K2: v = A p, (r^, v) -> alpha
template <class V, int S>
HELM_SOLVER_KERNEL k_v(const __grid_constant__ KArgs<V> a) {
  pdl_enter();
  __shared__ double red[32 * 2];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING || refine_step_pending<V>(st)) return;
  HELM_GRAPH_PHASES
  V rhi = vzero<V>();
  graph_spmv<V, S>(
      ph, a.p, [&](int32_t i) { rhi = a.rh[i]; }, [&](int32_t i, int li, V ax) { ph.row_v(i, li, rhi, ax, part); });
  double part2[2] = {part[0], part[1]}, tot[2];
  if (!grid_total_last<V, S, 2>(part2, a.partials, a.tickets + TK_V, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_after_v<V>(st, tot);
}

// K3: s = r - alpha v, ||s||
template <class V, int S>
HELM_SOLVER_KERNEL k_s(const __grid_constant__ KArgs<V> a) {
  pdl_enter();
  __shared__ double red[32];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING || refine_step_pending<V>(st)) return;
  HELM_GRAPH_PHASES
  ph.template upd_s<true>(Prec<V>::cvt(st->alpha), part);
  double part1[1] = {part[0]}, tot[1];
  if (!grid_total_last<V, S, 1>(part1, a.partials, a.tickets + TK_S, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_after_s<V>(st, tot);
}

// K4: t = A s, (t, s), (t, t) -> omega
template <class V, int S>
HELM_SOLVER_KERNEL k_t(const __grid_constant__ KArgs<V> a) {
  pdl_enter();
  __shared__ double red[32 * 3];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING || st->phase != PH_RUN || refine_step_pending<V>(st)) return;
  HELM_GRAPH_PHASES
  V si = vzero<V>();
  graph_spmv<V, S>(
      ph, a.s, [&](int32_t i) { si = a.s[i]; }, [&](int32_t i, int li, V ax) { ph.row_t(i, li, si, ax, part); });
  double part3[3] = {part[0], part[1], part[2]}, tot[3];
  if (!grid_total_last<V, S, 3>(part3, a.partials, a.tickets + TK_T, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_after_t<V>(st, tot);
}

// K5: x += alpha p + omega s, r = s - omega t; stop test; rho, beta
template <class V, int S>
HELM_SOLVER_KERNEL k_xr(const __grid_constant__ KArgs<V> a) {
  pdl_enter();
  __shared__ double red[32 * 3];
  SolverState* st = a.st;
  // (mixed precision: a pending refinement step ends the inner loop)
  if (st->status != ST_RUNNING || refine_step_pending<V>(st)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) set_cond(a, false);
    return;
  }
  HELM_GRAPH_PHASES
  ph.template upd_xr<true>(Prec<V>::cvt(st->alpha), Prec<V>::cvt(st->omega), st->phase == PH_SCONV, part);
  double part3[3] = {part[0], part[1], part[2]}, tot[3];
  if (!grid_total_last<V, S, 3>(part3, a.partials, a.tickets + TK_XR, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_after_xr<V>(st, tot, deadline_passed(st));
  set_cond(a, st->status == ST_RUNNING && !refine_step_pending<V>(st));
}

// ---------------------------------------------------------------- persistent loop

// A solve as a loop over steps, each a vector update or a product, then a grid
// barrier and (in every block the same) the sums and the scalar step that
// chooses the next one.  complex128: the whole solve (init, iterations, tail,
// restarts); complex64: the inner loop of mixed precision, from its start to the
// next refinement step.  Every step does exactly what the graph kernel of that
// name does, on the same rows of the same threads; the totals are formed from
// the same partials in the same order, so all blocks take every decision
// together (the deadline is decided by block 0 and carried in the last
// reduction of each iteration).  Two partials buffers alternate, so a block may
// publish the next step's sums while a slower block still reads the previous
// ones.  The gathered vectors (p, s, x at the start and the end) are written by
// other blocks of the same launch: they are read with coherent loads.  The
// others stay in the block's shared memory as far as they fit (Phases).
// One product, one reduction and one copy of each update in the code: see
// persist.cuh on registers and code size.
enum : int { STEP_INIT = 0, STEP_INIT_X0, STEP_LOAD, STEP_P, STEP_V, STEP_S, STEP_T, STEP_XR, STEP_FLUSH, STEP_TAIL,
             STEP_END };
template <class V, int S>
__device__ __forceinline__ void persist_loop(const KArgs<V>& a, const PLayout& L) {
  constexpr bool whole = std::is_same<V, double2>::value;
  constexpr bool SPLIT = whole && SolverBounds<S>::parts > 1;
  using G = GatherCoherent;
  __shared__ double red[32 * 4];
  __shared__ SolverState sst;
  __shared__ unsigned int s_target;  // arrivals of the barriers passed
  __shared__ int s_step;
  const Phases<V> ph(a, L);
  copy_state(&sst, a.st);
  if (threadIdx.x == 0) s_target = 0u;
  persist_table<V>(ph.q, a.A);
  HeldPart held;
  if constexpr (SPLIT) held.load(ph.q, a.A);
  int buf = 0;
  int step = sst.use_x0 ? STEP_INIT_X0 : STEP_INIT;
  if (!whole) step = sst.status == ST_RUNNING && !refine_step_pending<V>(&sst) ? STEP_LOAD : STEP_END;
  while (step != STEP_END) {
    double part[4] = {0.0, 0.0, 0.0, 0.0};
    if (step == STEP_P) {
      ph.template upd_p<false>(Prec<V>::cvt(sst.beta), Prec<V>::cvt(sst.omega));
    } else if (step == STEP_S) {
      ph.template upd_s<false>(Prec<V>::cvt(sst.alpha), part);
    } else if (step == STEP_XR) {
      ph.template upd_xr<false>(Prec<V>::cvt(sst.alpha), Prec<V>::cvt(sst.omega), sst.phase == PH_SCONV, part);
      part[3] = (blockIdx.x == 0 && threadIdx.x == 0 && deadline_passed(&sst)) ? 1.0 : 0.0;
    } else if (whole && step == STEP_INIT) {
      ph.init_zero(part);
    } else if (!whole && step == STEP_LOAD) {  // the vectors of the inner solve's start
      for_rows(ph.q, a.A.n, [&](int32_t i, int li) {
        if (ph.v.shared()) ph.v.st(i, li, a.v[i]);
        if (ph.r.shared()) ph.r.st(i, li, a.r[i]);
        if (ph.rh.shared()) ph.rh.st(i, li, a.rh[i]);
        if (ph.x.shared()) ph.x.st(i, li, a.x[i]);
        if (ph.p.shared()) ph.p.st(i, li, a.p[i]);
      });
      step = STEP_P;
      continue;
    } else if (step == STEP_FLUSH) {  // x is complete once every block is here
      if (sst.bnorm == 0.0) for_rows(ph.q, a.A.n, [&](int32_t i, int) { a.x[i] = vzero<V>(); });
      else if (ph.x.shared()) for_rows(ph.q, a.A.n, [&](int32_t i, int li) { a.x[i] = *ph.x.at(li); });
      if (!whole) break;
    } else if (step != STEP_TAIL || sst.bnorm != 0.0) {  // a product
      const V* in = step == STEP_V ? a.p : step == STEP_T ? a.s : a.x;
      auto row = [&](int32_t i, int li, V ax) {
        const int st = opaque(step);
        if (st == STEP_V) ph.row_v(i, li, ph.rh.ld(i, li), ax, part);
        else if (st == STEP_T) ph.row_t(i, li, ph.s.ld(i, li), ax, part);
        else if (st == STEP_TAIL) part[0] = nrm_acc(part[0], csub(a.b[i], ax));
        else ph.row_init(i, li, ax, part);
      };
      if constexpr (SPLIT) spmv_split<G>(ph.q, a.A, held, in, row);
      else spmv_rows<V, SolverBounds<S>::persist_u, 1, G>(ph.q, a.A, in, [](int32_t) {}, row);
    }
    if (step == STEP_P || step == STEP_FLUSH) {
      if (!grid_barrier(a.tickets, a.dev_err, &s_target)) return;
      step = step == STEP_P ? STEP_V : STEP_TAIL;
      continue;
    }
    buf ^= 1;
    double tot[4];
    if (!grid_total_all<V, S, 4>(part, a.partials + static_cast<size_t>(buf) * gridDim.x * 4, a.tickets, a.dev_err, &s_target,
                           red, tot))
      return;
    if (threadIdx.x == 0) {
      int next = STEP_P;
      if (step == STEP_V) {
        const double t2[2] = {tot[0], tot[1]};
        sc_after_v<V>(&sst, t2);
        next = STEP_S;
      } else if (step == STEP_S) {
        const double t1[1] = {tot[0]};
        sc_after_s<V>(&sst, t1);
        next = sst.phase == PH_RUN ? STEP_T : STEP_XR;
      } else if (step == STEP_T) {
        const double t3[3] = {tot[0], tot[1], tot[2]};
        sc_after_t<V>(&sst, t3);
        next = STEP_XR;
      } else if (step == STEP_XR) {
        const double t3[3] = {tot[0], tot[1], tot[2]};
        sc_after_xr<V>(&sst, t3, tot[3] > 0.0);
      } else if (step != STEP_TAIL) {
        sc_init(&sst, tot, step == STEP_INIT_X0);
      }
      if (sst.status != ST_RUNNING || refine_step_pending<V>(&sst)) next = STEP_FLUSH;
      if (step == STEP_TAIL) {
        const double t1[1] = {tot[0]};
        sc_tail(&sst, t1);
        next = STEP_END;
        // (as the host does for the graph)
        if (restart_due(&sst)) {
          next = STEP_INIT_X0;
          restart_state(&sst);
        }
      }
      s_step = next;
    }
    __syncthreads();
    step = s_step;
  }
  if (blockIdx.x == 0) copy_state(a.st, &sst);
}

// Solver grid: one wave of the solver kernels -- the blocks that fit on every
// SM at once for each of `fns` (so that none runs a second wave), times the
// SMs, at most enough blocks for one warp per slice.  Every kernel of a solve
// (graph or persistent) runs on this grid: the grid fixes which thread owns
// which row and so the order of every partial sum.
inline helm_status persistent_grid(std::initializer_list<const void*> fns, int threads, size_t smem,
                                   int num_sms, int64_t units, int* grid) {
  int per_sm = 1 << 30;
  for (const void* fn : fns) {
    int b = 0;
    HELM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, threads, smem));
    per_sm = b < per_sm ? b : per_sm;
  }
  if (per_sm < 1) per_sm = 1;
  int64_t g = static_cast<int64_t>(per_sm) * num_sms;
  if (units < g) g = units < 1 ? 1 : units;
  *grid = static_cast<int>(g);
  return HELM_OK;
}

template <class V>
struct KShapes {
  int grid;     // every kernel of the loop, init and tail included
  int threads;  // threads per block (a multiple of 32)
  int bps;      // blocks per SM the grid is sized for
  int shape;    // SHAPE_*
};

// HELM_LAUNCH_AUTO takes a persistent kernel for this solve (where the device can).
template <class V>
inline bool persist_default(helm_csr A, const KShapes<V>& sh, const helm_opts& o) {
  return o.launch == HELM_LAUNCH_AUTO &&
         A->max_row <= persist_max_row(sh.shape == SHAPE_LARGE, std::is_same<V, float2>::value,
                                       persist_rounds(A->n, sh.grid, sh.threads / 32));
}

// A whole solve as one cooperative launch of `fn` on the shape that persist_fit
// gave it; the final state is in A->state_host.  *done stays false (and nothing
// has run) when the device did not take the launch.
inline helm_status run_persistent(helm_csr A, const void* fn, void** args, const PShape& ps, const helm_opts& o,
                                  cudaStream_t s, bool* done) {
  k_configure<<<1, 1, 0, s>>>(A->state, o.tol, o.maxit, o.use_x0 ? 1 : 0, o.deadline_s, 1);
  HELM_CUDA_TRY(cudaGetLastError());
  HELM_CUDA_TRY(cudaMemsetAsync(A->tickets + TK_BAR_COUNT, 0, 2 * sizeof(unsigned int), s));  // count, abort
  const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(ps.grid), dim3(ps.threads), args, ps.smem, s);
  if (e != cudaSuccess) {
    debug_cuda_error(e, __FILE__, __LINE__);
    (void)cudaGetLastError();
    return HELM_OK;
  }
  unsigned int herr = 0;
  HELM_CUDA_TRY(cudaMemcpyAsync(A->state_host, A->state, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
  HELM_CUDA_TRY(cudaMemcpyAsync(&herr, A->dev_err, sizeof(unsigned int), cudaMemcpyDeviceToHost, s));
  HELM_CUDA_TRY(cudaStreamSynchronize(s));
  *done = true;
  return herr ? HELM_ERR_CUDA : HELM_OK;
}

// A loop kernel launched with programmatic stream serialization (a
// programmatic edge from the kernel before it when captured into a graph);
// see pdl_enter.
template <class V>
inline void launch_loop_kernel(void (*kernel)(KArgs<V>), const KArgs<V>& a, const KShapes<V>& sh, cudaStream_t s) {
#if HELM_PDL
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(sh.grid));
  cfg.blockDim = dim3(static_cast<unsigned>(sh.threads));
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kernel, a);  // errors surface at the caller's cudaGetLastError
#else
  kernel<<<sh.grid, sh.threads, 0, s>>>(a);
#endif
}

template <class V, int S>
inline void enqueue_body_s(const KArgs<V>& a, const KShapes<V>& sh, cudaStream_t s) {
  launch_loop_kernel<V>(k_p<V, S>, a, sh, s);
  launch_loop_kernel<V>(k_v<V, S>, a, sh, s);
  launch_loop_kernel<V>(k_s<V, S>, a, sh, s);
  launch_loop_kernel<V>(k_t<V, S>, a, sh, s);
  launch_loop_kernel<V>(k_xr<V, S>, a, sh, s);
}

// f(shape constant) for the shape of a solve
template <class V, class F>
inline void with_shape(const KShapes<V>& sh, F f) {
  if constexpr (std::is_same<V, double2>::value) {
    if (sh.shape == SHAPE_SMALL) return f(std::integral_constant<int, SHAPE_SMALL>());
  }
  if (sh.shape == SHAPE_MID) return f(std::integral_constant<int, SHAPE_MID>());
  f(std::integral_constant<int, SHAPE_LARGE>());
}
template <class V>
inline void enqueue_init(const KArgs<V>& a, const KShapes<V>& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) { k_init<V, S.value><<<sh.grid, sh.threads, 0, s>>>(a); });
}
template <class V>
inline void enqueue_body(const KArgs<V>& a, const KShapes<V>& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) { enqueue_body_s<V, S.value>(a, sh, s); });
}

// Shape of a slice-parallel grid: one block per SM (blocks_per_sm with
// smaller blocks), never more blocks than slices, and per block just enough
// warps (at most max_threads / 32) for one slice per warp in each round.
struct SliceShape {
  int grid, threads;
};
inline SliceShape slice_shape(int32_t n, int num_sms, int max_threads, int blocks_per_sm, bool full = false) {
  const int64_t nsl = std::max<int64_t>((static_cast<int64_t>(n) + 31) / 32, 1);
  const int64_t grid = std::min<int64_t>(static_cast<int64_t>(num_sms) * blocks_per_sm, nsl);
  const int64_t wmax = std::max(max_threads / 32, 1);
  // rounds at the widest block, then (unless `full`) the fewest warps that
  // keep that many rounds: every round (the last one too) nearly full
  const int64_t rounds = (nsl + grid * wmax - 1) / (grid * wmax);
  const int64_t warps =
      full ? std::min<int64_t>((nsl + grid - 1) / grid, wmax) : std::min<int64_t>((nsl + grid * rounds - 1) / (grid * rounds), wmax);
  return SliceShape{static_cast<int>(grid), static_cast<int>(32 * std::max<int64_t>(warps, 1))};
}

// Grid of the solver's kernels: one wave.
template <class V>
inline helm_status krylov_shapes(helm_csr A, KShapes<V>* sh) {
  const int64_t nsl = (static_cast<int64_t>(A->n) + 31) / 32, sms = A->num_sms;
  const bool c64 = std::is_same<V, float2>::value;
  sh->shape = nsl > sms * (c64 ? kMidSlices32 : kMidSlices)                             ? SHAPE_LARGE
              : !c64 && nsl <= sms * (SolverBounds<SHAPE_SMALL>::threads / 32 / kParts) ? SHAPE_SMALL
                                                                                        : SHAPE_MID;
  sh->bps = sh->shape == SHAPE_LARGE ? SolverBounds<SHAPE_LARGE>::blocks : 1;
  const SliceShape ss = slice_shape(A->n, A->num_sms, sh->shape == SHAPE_MID ? SolverBounds<SHAPE_MID>::threads : 512, sh->bps);
  sh->grid = ss.grid;
  sh->threads = ss.threads;
  return HELM_OK;
}

// Iterations (loop bodies) per pass of the while node: each pass re-launches
// the body graph, so several iterations per pass save that cost (measured:
// 164.5 -> 161.3 -> 159.8 us per BiCGStab iteration for 1, 2, 4); once the
// solve has finished, the remaining kernels of a pass return at once.
#ifndef HELM_BODY_UNROLL
#define HELM_BODY_UNROLL 4
#endif
constexpr int kBodyUnroll = HELM_BODY_UNROLL;

// Build a graph  init -> while(body) -> tail.  Each callable enqueues its
// kernels on the capture stream with the loop's conditional handle:
// init(cond, stream), body(cond, stream), tail(cond, stream).
template <class Init, class Body, class Tail>
helm_status build_while_graph(Init init, Body body, Tail tail, GraphEntry* out) {
  cudaStream_t cs = nullptr;
  HELM_CUDA_TRY(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  helm_status result = HELM_ERR_CUDA;
  do {
    if (cudaGraphCreate(&graph, 0) != cudaSuccess) break;
    cudaGraphConditionalHandle cond;
    if (cudaGraphConditionalHandleCreate(&cond, graph, 1u, cudaGraphCondAssignDefault) != cudaSuccess) break;
    if (cudaStreamBeginCaptureToGraph(cs, graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) !=
        cudaSuccess)
      break;
    init(cond, cs);
    cudaStreamCaptureStatus cst;
    const cudaGraphNode_t* deps = nullptr;
    size_t ndeps = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(cs, &cst, nullptr, nullptr, &deps, nullptr, &ndeps);
    cudaGraphNode_t init_node = (e == cudaSuccess && ndeps == 1) ? deps[0] : nullptr;
    cudaGraph_t tmp = nullptr;
    if (cudaStreamEndCapture(cs, &tmp) != cudaSuccess || e != cudaSuccess || !init_node) break;
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = cond;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t wnode;
    if (cudaGraphAddNode(&wnode, graph, &init_node, nullptr, 1, &cp) != cudaSuccess) break;
    cudaGraph_t bodyg = cp.conditional.phGraph_out[0];
    if (cudaStreamBeginCaptureToGraph(cs, bodyg, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) !=
        cudaSuccess)
      break;
    for (int u = 0; u < kBodyUnroll; ++u) body(cond, cs);
    if (cudaStreamEndCapture(cs, &tmp) != cudaSuccess) break;
    if (cudaStreamBeginCaptureToGraph(cs, graph, &wnode, nullptr, 1, cudaStreamCaptureModeThreadLocal) !=
        cudaSuccess)
      break;
    tail(cond, cs);
    if (cudaStreamEndCapture(cs, &tmp) != cudaSuccess) break;
    if (cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) break;
    result = HELM_OK;
  } while (false);
  cudaStreamDestroy(cs);
  if (result != HELM_OK) {
    (void)cudaGetLastError();
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    return result;
  }
  out->exec = exec;
  out->graph = graph;
  return HELM_OK;
}

// BiCGStab graph  init -> while(K1..K5) -> tail  for fixed vectors.
template <class V, class Tail>
helm_status build_krylov_graph(const KArgs<V>& base, const KShapes<V>& sh, Tail tail, GraphEntry* out) {
  auto with = [&](cudaGraphConditionalHandle cond) {
    KArgs<V> a = base;
    a.cond = cond;
    a.has_cond = 1;
    return a;
  };
  return build_while_graph([&](cudaGraphConditionalHandle c, cudaStream_t s) { enqueue_init(with(c), sh, s); },
                           [&](cudaGraphConditionalHandle c, cudaStream_t s) { enqueue_body(with(c), sh, s); },
                           [&](cudaGraphConditionalHandle c, cudaStream_t s) { tail(with(c), s); }, out);
}

// Run init -> loop -> tail once: through the cached graph when there is one,
// else host-driven (chunks of 16 iterations, state polled between chunks).
template <class V, class Tail>
helm_status run_krylov(helm_csr A, const KArgs<V>& a, const KShapes<V>& sh, GraphEntry* g, Tail tail,
                       cudaStream_t s) {
  if (g && g->exec) {
    HELM_CUDA_TRY(cudaGraphLaunch(g->exec, s));
    return HELM_OK;
  }
  enqueue_init(a, sh, s);
  HELM_CUDA_TRY(cudaGetLastError());
  for (;;) {
    for (int k = 0; k < 16; ++k) enqueue_body(a, sh, s);
    HELM_CUDA_TRY(cudaGetLastError());
    HELM_CUDA_TRY(cudaMemcpyAsync(A->state_host, a.st, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
    HELM_CUDA_TRY(cudaStreamSynchronize(s));
    if (A->state_host->status != ST_RUNNING) break;
  }
  tail(a, s);
  HELM_CUDA_TRY(cudaGetLastError());
  return HELM_OK;
}

}  // namespace helm
