// Persistent solvers: a Krylov loop as one cooperative kernel whose steps are
// separated by grid barriers (Section 4's iterations without a launch or a
// host step between their kernels).
//
// What bounds a small or medium solve is not bytes or FP64 but the chain of
// latencies between its kernels: launch, ramp, L2 round trips, the sums, the
// scalars.  Here a step is one grid barrier, and a block keeps in shared memory
// what only it needs: the positions of its slices, its rows' lengths and the
// vectors that are never gathered (v, r, t, r^, x).
//
// What a step costs on GB300 (measured): L2 round trip 300-470 clocks,
// fence.acq_rel.gpu 325 (650 with stores in flight), a dependent FP64 add 64,
// the whole barrier 3,600.  Two things that are easy to lose more with:
//   * the acquire fence drops the SM's L1, so that a spilled register costs an
//     L2 round trip after every barrier: the kernels must not spill;
//   * code that is run once per step comes from the instruction cache: at 147
//     kB of it every step ran two to three times slower than at 88 kB.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.hpp"
#include "persist_plan.hpp"
#include "spmv.cuh"

namespace helm {

// ---------------------------------------------------------------- grid barrier

__device__ __forceinline__ unsigned int ld_relaxed_u32(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// A grid barrier for a cooperative launch (all blocks resident).  The count
// word only grows (zero before the launch): thread 0 of each block adds one
// and waits until the count reaches gridDim.x times the number of barriers
// passed, compared modulo 2^32, so arriving is the block's only write and the
// last arrival itself releases the others.  `target` is the block's own count
// of arrivals to wait for, in shared memory.  Every wait is bounded; a block
// that gives up sets the abort word and DEVERR_BARRIER_TIMEOUT, and returns
// false in all its threads: every block leaves the kernel.
// Measured on GB300, whatever the grid (16 to 304 blocks): 1.7-1.9 us; every
// block polling a slot of every other one: 2.9 to 6 us; with the global timer
// and the abort word read in every poll: about 5 us.
__device__ __forceinline__ bool grid_barrier(unsigned int* tickets, unsigned int* dev_err, unsigned int* target) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int* count = tickets + TK_BAR_COUNT;
    unsigned int* abort = tickets + TK_BAR_ABORT;
    const unsigned int tg = *target + gridDim.x;
    *target = tg;
    int ok = 1;
    asm volatile("fence.acq_rel.gpu;" ::: "memory");  // release: this block's writes (ordered by the __syncthreads)
    asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
#pragma unroll 1
    for (int it = 0; static_cast<int>(ld_relaxed_u32(count) - tg) < 0; ++it) {
      if ((it & 255) == 255 && ld_relaxed_u32(abort) != 0u) {
        ok = 0;
        break;
      }
      if (it >= kBarrierPolls) {
        atomicOr(dev_err, DEVERR_BARRIER_TIMEOUT);
        atomicExch(abort, 1u);
        ok = 0;
        break;
      }
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");  // acquire: the other blocks' writes
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// The solver's state between global and shared memory, word by word over the
// block's threads (a barrier of the block has to follow or precede).
__device__ __forceinline__ void copy_state(SolverState* to, const SolverState* from) {
  static_assert(sizeof(SolverState) % 8 == 0, "copied in 8-byte words");
#pragma unroll 1
  for (int i = threadIdx.x; i < static_cast<int>(sizeof(SolverState) / 8); i += blockDim.x)
    reinterpret_cast<unsigned long long*>(to)[i] = reinterpret_cast<const unsigned long long*>(from)[i];
}

// ---------------------------------------------------------------- a block's rows and vectors

// The block's warps: unsplit, each warp owns its slices' rows; split (small
// meshes: one slice a warp), the first third own the rows and each row's sum is
// shared out to three warps.  The block's dynamic shared memory is laid out by
// persist_plan.hpp.
struct RoundTab {
  SlicePos pos;
  int32_t s, pad_[3];
};
static_assert(sizeof(RoundTab) == kRoundTabBytes && sizeof(double2) == kExchangeBytes, "as the host lays them out");

extern __shared__ __align__(128) unsigned char persist_smem[];

// v, as a value that the compiler does not know to be the same from one row to
// the next: it would copy a loop over the rows for each combination of such
// conditions.
__device__ __forceinline__ int32_t opaque(int32_t v) {
  asm volatile("" : "+r"(v));
  return v;
}

// The rows of this thread: those SliceRows gives it on a grid of the owner
// warps, round by round.
struct PRows {
  const PLayout& L;
  int32_t owner;  // the owner warp whose slices this warp works on
  int32_t share;  // and its share of their sums
  __device__ __forceinline__ explicit PRows(const PLayout& l) : L(l) {
    const int32_t w = static_cast<int32_t>(threadIdx.x >> 5);
    share = w >= 2 * L.warps ? 2 : w >= L.warps ? 1 : 0;
    owner = w - share * L.warps;
  }
  __device__ __forceinline__ int lane() const { return static_cast<int>(threadIdx.x & 31); }
  __device__ __forceinline__ bool table() const { return opaque(L.tab) != 0; }
  __device__ __forceinline__ RoundTab* round(int32_t k) const {
    return reinterpret_cast<RoundTab*>(persist_smem) + k * L.warps + owner;
  }
  // place of round k's row of the owner in the block's shared vectors
  __device__ __forceinline__ int place(int32_t k) const { return (k * L.warps + owner) * 32 + lane(); }
  __device__ __forceinline__ int32_t* tlen(int32_t k) const {
    return reinterpret_cast<int32_t*>(persist_smem + L.tlen_at) + place(k);
  }

  __device__ __forceinline__ int32_t compute_slice(int32_t n, int32_t k) const {
    const uint32_t G = gridDim.x, WB = static_cast<uint32_t>(L.warps), W = G * WB,
                   m = static_cast<uint32_t>((n + 31) >> 5);
    const uint32_t base = static_cast<uint32_t>(k) * W, b = blockIdx.x, w = static_cast<uint32_t>(owner);
    if (base >= m) return -1;
    uint32_t lo = base + b * WB, hi = lo + WB;
    if (m - base < W) {
      lo = base + b * (m - base) / G;
      hi = base + (b + 1) * (m - base) / G;
    }
    return lo + w < hi ? static_cast<int32_t>(lo + w) : -1;
  }
  __device__ __forceinline__ int32_t slice(int32_t n, int32_t k) const {
    return table() ? round(k)->s : compute_slice(n, k);
  }
};

// Fill the table (all threads; ends with a barrier of the block).
template <class V>
__device__ __forceinline__ void persist_table(const PRows& q, const CsrDev<V>& A) {
  if (q.table() && q.share == 0) {
#pragma unroll 1
    for (int32_t k = 0; k < q.L.rounds; ++k) {
      const int32_t s = q.compute_slice(A.n, k);
      const int32_t r = s * 32 + q.lane();
      if (q.lane() == 0) {
        RoundTab* t = q.round(k);
        t->s = s;
        if (s >= 0) t->pos = slice_pos(A, s);
      }
      *q.tlen(k) = (s >= 0 && r < A.n) ? A.rowptr[r + 1] - A.rowptr[r] : 0;
    }
  }
  __syncthreads();
}

// Calls f(row, li) for every row of this thread, li = its place in the
// block's shared vectors.
template <class F>
__device__ __forceinline__ void for_rows(const PRows& q, int32_t n, F f) {
  if (q.share != 0) return;
#pragma unroll 1
  for (int32_t k = 0; k < q.L.rounds; ++k) {
    const int32_t s = q.slice(n, k);
    const int32_t r = s * 32 + q.lane();
    if (s >= 0 && r < n) f(r, q.place(k));
  }
}

// f(row, li, ld(row, li)) for every row of this thread; with AHEAD (graph kernels,
// which have the registers) the next row's loads are issued before a row is worked
// on.
template <bool AHEAD, class Ld, class F>
__device__ __forceinline__ void for_rows_ld(const PRows& q, int32_t n, Ld ld, F f) {
  if constexpr (!AHEAD) {
    for_rows(q, n, [&](int32_t r, int li) { f(r, li, ld(r, li)); });
  } else {
    int32_t s = q.slice(n, 0), r = s * 32 + q.lane();
    if (s < 0 || r >= n) return;  // only the last round has none for some warps
    auto cur = ld(r, q.place(0));
#pragma unroll 1
    for (int32_t k = 0;; ++k) {
      const int32_t s1 = k + 1 < q.L.rounds ? q.slice(n, k + 1) : -1;
      const int32_t r1 = s1 * 32 + q.lane();
      const bool more = s1 >= 0 && r1 < n;
      auto next = cur;
      if (more) next = ld(r1, q.place(k + 1));
      f(r, q.place(k), cur);
      if (!more) return;
      cur = next;
      r = r1;
    }
  }
}

// Calls f(row, li, sum_k a_rk x_k) for every row of this thread; pre(row) first
// (its loads are in flight with the sum's).  A split solver's rows are summed
// in three parts (sell_row_part): here by the row's thread (sell_row_parts).
template <class V, int U, int PARTS, class G, class Pre, class F>
__device__ __forceinline__ void spmv_rows(const PRows& q, const CsrDev<V>& A, const V* x, Pre pre, F f) {
#pragma unroll 1
  for (int32_t k = 0; k < q.L.rounds; ++k) {
    const int32_t s = q.slice(A.n, k);
    if (s < 0) continue;
    const int32_t r = s * 32 + q.lane();
    const SlicePos sp = q.table() ? q.round(k)->pos : slice_pos(A, s);
    const int32_t len = q.table() ? *q.tlen(k) : r < A.n ? A.rowptr[r + 1] - A.rowptr[r] : 0;
    if (r < A.n) pre(r);
    V acc;
    if constexpr (std::is_same<V, float2>::value) {
      acc = A.ndia > 0 ? dia_row<G>(A, s, q.lane(), r, x) : sell_row<V, G, U>(A, sp, q.lane(), r, len, x);
    } else if constexpr (PARTS == 1) {
      acc = sell_row<V, G, U>(A, sp, q.lane(), r, len, x);
    } else {
      static_assert(PARTS == kParts, "as the split kernels sum them");
      acc = sell_row_parts<V, G>(A, sp, q.lane(), r, len, x);
    }
    if (r < A.n) f(r, q.place(k), acc);
  }
}

// The entries of this warp's share of its slice, kept in registers for the
// whole solve (split kernels: one slice a warp): a product then starts with
// its gathers.  Rows of more than kHeld entries a part read them at every
// product instead.
constexpr int kHeld = 9, kHeldImag = 3;
struct HeldPart {
  double a[kHeld], b[kHeldImag];
  int32_t c[kHeld], d[kHeldImag];
  int32_t n, m;  // entries of this lane's row, real and imaginary
  bool held;     // the warp's share fits
  __device__ __forceinline__ void load(const PRows& q, const CsrDev<double2>& A) {
    n = m = 0;
    held = true;
    const int32_t s = q.round(0)->s;
    if (s >= 0) {
      const SlicePos sp = q.round(0)->pos;
      const int32_t r = s * 32 + q.lane(), len = *q.tlen(0), il = sp.iw > 0 && r < A.n ? A.ilen[r] : 0;
      const int32_t ch = part_width(sp.w), ci = part_width(sp.iw);
      held = ch <= kHeld && ci <= kHeldImag;
      n = max(min(len - q.share * ch, ch), 0);
      m = max(min(il - q.share * ci, ci), 0);
      const int32_t at = sp.base + q.share * ch * 32 + q.lane(), ai = sp.ib + q.share * ci * 32 + q.lane();
#pragma unroll
      for (int u = 0; u < kHeld; ++u) {
        a[u] = held && u < n ? A.sval[at + u * 32] : 0.0;
        c[u] = held && u < n ? A.scol[at + u * 32] : 0;
      }
#pragma unroll
      for (int u = 0; u < kHeldImag; ++u) {
        b[u] = held && u < m ? A.ival[ai + u * 32] : 0.0;
        d[u] = held && u < m ? A.icol[ai + u * 32] : 0;
      }
    }
  }
  // sell_row_part of this share
  template <class G>
  __device__ __forceinline__ double2 sum(const double2* x) const {
    double2 xv[kHeld], xi[kHeldImag];
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < kHeld; ++u)
      if (u < n) xv[u] = G::ld(x + c[u]);
#pragma unroll
    for (int u = 0; u < kHeldImag; ++u)
      if (u < m) xi[u] = G::ld(x + d[u]);
#pragma unroll
    for (int u = 0; u < kHeld; ++u)
      if (u < n) acc = mac_real(a[u], xv[u], acc);
#pragma unroll
    for (int u = 0; u < kHeldImag; ++u)
      if (u < m) acc = mac_imag(b[u], xi[u], acc);
    return acc;
  }
};

// The product with split warps (whole block; one round): each warp sums its
// share of its slice's rows, the owners add the parts in order.
template <class G, class F>
__device__ __forceinline__ void spmv_split(const PRows& q, const CsrDev<double2>& A, const HeldPart& H,
                                           const double2* x, F f) {
  const int32_t s = q.round(0)->s;
  const int32_t r = s * 32 + q.lane();
  double2 acc = make_double2(0.0, 0.0);
  if (s >= 0)
    acc = H.held ? H.sum<G>(x) : sell_row_part<double2, G, 2>(A, q.round(0)->pos, q.lane(), r, *q.tlen(0), q.share, x);
  double2* xc = reinterpret_cast<double2*>(persist_smem + q.L.xchg_at) + q.owner * 32 + q.lane();
  if (q.share > 0) xc[(q.share - 1) * q.L.warps * 32] = acc;
  __syncthreads();
  if (q.share == 0 && s >= 0 && r < A.n) {
#pragma unroll
    for (int p = 0; p < kParts - 1; ++p) acc = cadd(acc, xc[p * q.L.warps * 32]);
    f(r, q.place(0), acc);
  }
}

// Vector I of those that a thread keeps for its rows: in the block's shared
// memory when I < nown, else (and then only) in global memory.
template <class V, int I>
struct Own {
  V* const& gl;
  const PLayout& L;
  __device__ __forceinline__ bool shared() const { return I < L.nown; }
  __device__ __forceinline__ V* at(int li) const {
    return reinterpret_cast<V*>(persist_smem + L.own_at) + I * L.own_len + li;
  }
  __device__ __forceinline__ V* ptr(int32_t row, int li) const { return I < opaque(L.nown) ? at(li) : gl + row; }
  __device__ __forceinline__ V ld(int32_t row, int li) const { return *ptr(row, li); }
  __device__ __forceinline__ void st(int32_t row, int li, V v) const { *ptr(row, li) = v; }
  // both, for a vector that other blocks gather
  __device__ __forceinline__ void st_both(int32_t row, int li, V v) const {
    gl[row] = v;
    if (I < opaque(L.nown)) *at(li) = v;
  }
};

// ---------------------------------------------------------------- host side

struct PShape {
  int grid = 0, threads = 0;
  PLayout L = {};
  size_t smem = 0;
};

// Fit a persistent kernel for the system A on a grid of `grid` blocks (bps per SM)
// of `owners` owner threads, times `split` warps a slice: the table and as many of
// `want` own vectors of `elem` bytes as there is room for.  False when the kernel
// cannot run so.
inline bool persist_fit(const void* fn, const helm_csr_s* A, int grid, int owners, int bps, int split, int want,
                        size_t elem, PShape* p) {
  int dev = 0, per_sm = 0, optin = 0, reserved = 0, coop = 0;
  cudaFuncAttributes fa;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
      cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, fn) != cudaSuccess)
    return false;
  p->grid = grid;
  p->threads = owners * split;
  const size_t room = persist_room(per_sm, optin, reserved, fa.sharedSizeBytes, bps, A->ndia > 0);
  if (!persist_plan(A->n, grid, owners, split, want, elem, room, &p->L, &p->smem)) return false;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           optin - static_cast<int>(fa.sharedSizeBytes)) != cudaSuccess)
    return false;
  int fit = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, fn, p->threads, p->smem) != cudaSuccess) return false;
  return fit >= bps;
}

}  // namespace helm
