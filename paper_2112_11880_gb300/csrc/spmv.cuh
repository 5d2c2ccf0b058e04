// CSR SpMV engine (Section 3, Table 8 of the paper: CSR SpMV, 8 flops per
// stored entry in complex arithmetic), for complex128 and complex64.
//
// The handle keeps the caller's CSR arrays and derives from them, once, a
// sliced-ELLPACK copy (SELL-32, Kreutzer et al. 2014, without row sorting):
//   * a slice is 32 consecutive rows; its width w is the longest row in it;
//     entry k of the slice's row l sits at soff[s] + 32 k + l, so when the 32
//     lanes of a warp each take one row, every load of a value or column
//     index is one contiguous, fully coalesced 256-byte (values) or 128-byte
//     (columns) access, and the gathered x[col] of neighbouring rows share
//     cache lines;
//   * the real parts of the values are stored there (8 bytes per entry for
//     complex128, 4 for complex64) and multiplied with the real x complex
//     product (2 FMA per entry instead of 4);
//   * the entries with a nonzero imaginary part are kept again, as a second
//     SELL of imaginary parts (for Helmholtz FEM, A = K - k^2 M + i k B, only
//     the rows of the impedance face: 65,341 of 9.7 M entries on the
//     120x60x50 cavity), each adding i Im(a) x with 2 more FMA.
//   Padding entries (rows shorter than the slice width) are never read: each
//   lane stops at its own row length.
// A row's sum runs in CSR order over the real parts, then over the imaginary
// parts, so that for a row whose entries are all real it is the CSR-order FP64 sum
// bit for bit.  Two users sum it in parts instead, each part so, the parts added in
// order: the solvers on the smallest meshes (kParts) and the stand-alone product of
// matrices of few slices (k_spmv_split).
//
// Schedule (SliceRows): rounds of consecutive slices, each round split into
// equal contiguous sub-ranges, one per block (one block per SM), one slice
// per warp: the whole GPU works on one front of consecutive slices
// (sequential HBM streams; x gathers that hit in L2 and, within a block, in
// L1) and every SM has the same work.  The
// loads of the next U entries are issued before the FMAs of the current U
// (software pipeline), so each warp keeps 2U matrix loads and U gathers in
// flight.  Measured on GB300 (120x60x50 cavity, nnz 9.7 M): 43.1 us, against
// 47.6 us for 32-row CSR tiles staged into shared memory by TMA bulk copies
// (the previous engine); per-warp contiguous slice ranges were 1.3-8x slower.
// On GB300 the FP64 pipe (about two FMA lanes per clock per SM), not HBM,
// bounds this kernel: 2 FMA per stored entry.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "internal.hpp"

// Entries per pipeline stage of a row (matrix loads in flight: 2U per lane).
#ifndef HELM_SPMV_UNROLL
#define HELM_SPMV_UNROLL 4
#endif

namespace helm {

constexpr int kSpmvUnroll = HELM_SPMV_UNROLL;

// Real type of a complex type.
template <class V> struct RealOf;
template <> struct RealOf<double2> { using T = double; };
template <> struct RealOf<float2> { using T = float; };

// Device view of a matrix: the CSR arrays and the SELL-32 copy.
template <class V>
struct CsrDev {
  using R = typename RealOf<V>::T;
  int32_t n;
  int64_t nnz;
  const int32_t* rowptr;  // CSR row pointers (row lengths are read from here)
  const int32_t* colind;  // CSR column indices (not read by the SpMV)
  const V* vals;          // CSR values (not read by the SpMV)
  int32_t nsl;            // slices: ceil(n / 32)
  const int32_t* soff;    // [nsl + 1] first entry of each slice (multiples of 32)
  const int32_t* scol;    // [soff[nsl]] columns, slice-major
  const R* sval;          // [soff[nsl]] real parts, slice-major
  const int32_t* isoff;   // [nsl + 1] the same for the imaginary entries
  const int32_t* icol;
  const R* ival;
  const int32_t* ilen;    // [n] imaginary entries per row (read only in slices that have some)
  int32_t ndia;           // complex64 with a diagonal copy: the real parts on ndia diagonals, else 0
  const int32_t* doff;    // [ndia] ascending offsets col - row
  int64_t dld;            // row length of dval: n rounded up to a multiple of 4
  const R* dval;          // [ndia][dld] real part of entry (r, r + doff[d]), 0 where none
};
__host__ __device__ __forceinline__ int64_t dia_ld(int32_t n) { return (static_cast<int64_t>(n) + 3) & ~int64_t(3); }

template <class V> __device__ __forceinline__ V vzero();
template <> __device__ __forceinline__ double2 vzero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 vzero<float2>() { return make_float2(0.f, 0.f); }
template <class V> __device__ __forceinline__ V vadd(V a, V b) { return cadd(a, b); }

// acc + a x for real a
__device__ __forceinline__ double2 mac_real(double a, double2 x, double2 acc) {
  acc.x = fma(a, x.x, acc.x);
  acc.y = fma(a, x.y, acc.y);
  return acc;
}
__device__ __forceinline__ float2 mac_real(float a, float2 x, float2 acc) {
  acc.x = fmaf(a, x.x, acc.x);
  acc.y = fmaf(a, x.y, acc.y);
  return acc;
}
// acc + a x, complex a
__device__ __forceinline__ double2 mac(double2 a, double2 x, double2 acc) { return cfma(a, x, acc); }
__device__ __forceinline__ float2 mac(float2 a, float2 x, float2 acc) { return cfma32(a, x, acc); }
// acc + i b x for real b
__device__ __forceinline__ double2 mac_imag(double b, double2 x, double2 acc) {
  acc.x = fma(-b, x.y, acc.x);
  acc.y = fma(b, x.x, acc.y);
  return acc;
}
__device__ __forceinline__ float2 mac_imag(float b, float2 x, float2 acc) {
  acc.x = fmaf(-b, x.y, acc.x);
  acc.y = fmaf(b, x.x, acc.y);
  return acc;
}

// How the gathered vector is loaded.  Kernels that only read x take the
// read-only path; a kernel that writes the vector it later gathers (the
// persistent solvers, across their grid barriers) must use coherent loads.
struct GatherReadOnly {
  template <class V> __device__ __forceinline__ static V ld(const V* p) { return __ldg(p); }
};
struct GatherCoherent {
  // an ordinary load: the acquire fence of the grid barrier before it orders
  // it after the other blocks' stores (and drops this SM's L1 lines), and
  // within a phase neighbouring rows share the lines in L1
  template <class V> __device__ __forceinline__ static V ld(const V* p) { return *p; }
};

// Where a slice lies: its first entry and width, and those of its imaginary
// entries.
struct SlicePos {
  int32_t base, w, ib, iw;
};
template <class V>
__device__ __forceinline__ SlicePos slice_pos(const CsrDev<V>& A, int32_t s) {
  const int32_t base = A.soff[s], ib = A.isoff[s];
  return SlicePos{base, (A.soff[s + 1] - base) >> 5, ib, (A.isoff[s + 1] - ib) >> 5};
}

// acc + sum over the row's `len` entries of (IMAG ? i : 1) v_k x[c_k], entry k
// at stride 32 from v and c, at most w entries in the slice: a U-entry
// software pipeline (the next stage's entries are loaded before this one's
// products; the gathers of a stage are in flight together).
template <class V, class G, int U, bool IMAG>
__device__ __forceinline__ V sell_acc(const typename RealOf<V>::T* v, const int32_t* c, int32_t w, int32_t len,
                                      const V* x, V acc) {
  using R = typename RealOf<V>::T;
  R a[U];
  int32_t cc[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    a[u] = R(0);
    cc[u] = 0;
    if (u < len) {
      a[u] = __ldcs(v + u * 32);
      cc[u] = __ldcs(c + u * 32);
    }
  }
#pragma unroll 1
  for (int32_t k = 0; k < w; k += U) {
    V xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k + u < len) xv[u] = G::ld(x + cc[u]);
    R an[U];
    int32_t cn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      an[u] = R(0);
      cn[u] = 0;
      if (k + U + u < len) {
        an[u] = __ldcs(v + (k + U + u) * 32);
        cn[u] = __ldcs(c + (k + U + u) * 32);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k + u < len) acc = IMAG ? mac_imag(a[u], xv[u], acc) : mac_real(a[u], xv[u], acc);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      a[u] = an[u];
      cc[u] = cn[u];
    }
  }
  return acc;
}

// acc + the row's imaginary entries (iw in its slice at most, from ib).
template <class V, class G>
__device__ __forceinline__ V imag_row(const CsrDev<V>& A, int32_t ib, int32_t iw, int lane, int32_t r, const V* x,
                                      V acc) {
  if (iw > 0) {
    const int32_t il = r < A.n ? A.ilen[r] : 0;
    for (int32_t q = 0; q < iw; ++q) {
      if (q < il) {
        const typename RealOf<V>::T b = A.ival[ib + q * 32 + lane];
        acc = mac_imag(b, G::ld(x + A.icol[ib + q * 32 + lane]), acc);
      }
    }
  }
  return acc;
}

// Sum of row r = 32 s + lane (len entries) of the slice at `sp`: real parts in
// CSR order, then the row's imaginary entries.
template <class V, class G = GatherReadOnly, int U = kSpmvUnroll>
__device__ __forceinline__ V sell_row(const CsrDev<V>& A, const SlicePos& sp, int lane, int32_t r, int32_t len,
                                      const V* x) {
  const V acc = sell_acc<V, G, U, false>(A.sval + sp.base + lane, A.scol + sp.base + lane, sp.w, len, x, vzero<V>());
  return imag_row<V, G>(A, sp.ib, sp.iw, lane, r, x, acc);
}

// A row's sum in PARTS parts, for kernels that share it out to as many warps and
// add the parts in order (solvers: kParts, in every form of the solve): part p is
// entries [p w', (p + 1) w') with w' = ceil(w / PARTS) for slice width w, real
// parts, then imaginary ones likewise.
constexpr int kParts = 3;
template <int PARTS = kParts>
__host__ __device__ __forceinline__ int32_t part_width(int32_t w) {
  return (w + PARTS - 1) / PARTS;
}
template <class V, class G, int U, int PARTS = kParts, int UI = 2>
__device__ __forceinline__ V sell_row_part(const CsrDev<V>& A, const SlicePos& sp, int lane, int32_t r, int32_t len,
                                           int32_t p, const V* x) {
  const int32_t ch = part_width<PARTS>(sp.w), ci = part_width<PARTS>(sp.iw);
  const int32_t il = sp.iw > 0 && r < A.n ? A.ilen[r] : 0;
  const int32_t at = sp.base + p * ch * 32 + lane, ai = sp.ib + p * ci * 32 + lane;
  V acc = sell_acc<V, G, U, false>(A.sval + at, A.scol + at, ch, max(min(len - p * ch, ch), 0), x, vzero<V>());
  if (sp.iw > 0) acc = sell_acc<V, G, UI, true>(A.ival + ai, A.icol + ai, ci, max(min(il - p * ci, ci), 0), x, acc);
  return acc;
}

// A row's kParts parts by one thread, added in order: the same sums, the parts'
// pipelines side by side, two entries of each a stage (one part after the other: a
// BiCGStab iteration of the 20^3 box as a graph 43.7 us, so 39.0).
template <class V, class G>
__device__ __forceinline__ V sell_row_parts(const CsrDev<V>& A, const SlicePos& sp, int lane, int32_t r, int32_t len,
                                            const V* x) {
  using R = typename RealOf<V>::T;
  constexpr int U = 2;
  const int32_t ch = part_width(sp.w), ci = part_width(sp.iw);
  V acc[kParts];
  R a[kParts][U];
  int32_t c[kParts][U];
  auto entry = [&](int p, int u, int32_t k) {
    const int32_t e = p * ch + k;
    a[p][u] = R(0);
    c[p][u] = 0;
    if (k < ch && e < len) {
      a[p][u] = __ldcs(A.sval + sp.base + e * 32 + lane);
      c[p][u] = __ldcs(A.scol + sp.base + e * 32 + lane);
    }
  };
#pragma unroll
  for (int p = 0; p < kParts; ++p) {
    acc[p] = vzero<V>();
#pragma unroll
    for (int u = 0; u < U; ++u) entry(p, u, u);
  }
#pragma unroll 1
  for (int32_t k = 0; k < ch; k += U) {
    V xv[kParts][U];
    R av[kParts][U];
#pragma unroll
    for (int p = 0; p < kParts; ++p)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (k + u < ch && p * ch + k + u < len) xv[p][u] = G::ld(x + c[p][u]);
        av[p][u] = a[p][u];
      }
#pragma unroll
    for (int p = 0; p < kParts; ++p)
#pragma unroll
      for (int u = 0; u < U; ++u) entry(p, u, k + U + u);
#pragma unroll
    for (int p = 0; p < kParts; ++p)
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u < ch && p * ch + k + u < len) acc[p] = mac_real(av[p][u], xv[p][u], acc[p]);
  }
  if (sp.iw > 0) {
    const int32_t il = r < A.n ? A.ilen[r] : 0;
#pragma unroll 1
    for (int32_t k = 0; k < ci; ++k) {
      R b[kParts];
      V xv[kParts];
#pragma unroll
      for (int p = 0; p < kParts; ++p)
        if (p * ci + k < il) {
          b[p] = A.ival[sp.ib + (p * ci + k) * 32 + lane];
          xv[p] = G::ld(x + A.icol[sp.ib + (p * ci + k) * 32 + lane]);
        }
#pragma unroll
      for (int p = 0; p < kParts; ++p)
        if (p * ci + k < il) acc[p] = mac_imag(b[p], xv[p], acc[p]);
    }
  }
  V sum = acc[0];
#pragma unroll
  for (int p = 1; p < kParts; ++p) sum = vadd(sum, acc[p]);
  return sum;
}

// Rows of this thread.  The slices are taken in rounds of W = G WB
// consecutive slices (G blocks of WB warps); in round k, whose R slices
// start at k W, block b takes the contiguous sub-range
// [k W + floor(b R / G), k W + floor((b + 1) R / G)), one slice per warp in
// warp order.  So at any moment the grid works on one front of consecutive
// slices (sequential HBM streams, x gathers that hit in L2), the warps of a
// block work on neighbouring slices (their x gathers share L1 lines), every
// block gets the same number of slices to one, also when the last round is
// partial, and the thread that owns a row depends only on the grid's shape:
// every kernel of a solver that launches on the same grid gives a row to
// the same thread, so element-wise phases find their operands where the
// SpMV phase left them, and each thread's partial sums do not depend on the
// schedule.
struct SliceRows {
  int32_t s, lane, nsl, k;
  __device__ __forceinline__ explicit SliceRows(int32_t n)
      : s(0), lane(static_cast<int32_t>(threadIdx.x & 31)), nsl((n + 31) >> 5), k(-1) {
    advance();
  }
  // Move to this warp's slice of the next round that gives it one; s = nsl
  // when there is none.
  __device__ __forceinline__ bool advance() {
    // 32-bit arithmetic: nsl < 2^26, W <= 2^17 warps and b R < 2^31 on this
    // GPU's grids; a full round (R = W) gives block b its WB slices without a
    // division
    const uint32_t G = gridDim.x, WB = blockDim.x >> 5, W = G * WB, m = static_cast<uint32_t>(nsl);
    const uint32_t b = blockIdx.x, w = threadIdx.x >> 5;
    uint32_t base = static_cast<uint32_t>(++k) * W;
    for (; base < m; base += W, ++k) {
      uint32_t lo = base + b * WB, hi = lo + WB;
      if (m - base < W) {
        lo = base + b * (m - base) / G;
        hi = base + (b + 1) * (m - base) / G;
      }
      if (lo + w < hi) {
        s = static_cast<int32_t>(lo + w);
        return true;
      }
    }
    s = nsl;
    return false;
  }
  __device__ __forceinline__ bool active() const { return s < nsl; }
  __device__ __forceinline__ int32_t row() const { return s * 32 + lane; }
};

// Row r of a complex64 matrix with a diagonal copy: the real parts from the
// diagonals, in ascending column order (the CSR order of a sorted row), then
// the row's imaginary entries as in sell_row.  Every diagonal's value and
// gather are loaded independently of one another (no load waits on another
// one); a diagonal without an entry in this row (value 0) leaves the sum
// untouched, so the result is that of sell_row for finite x.  The complex64
// product is bound by HBM on this GPU (its arithmetic is FP32): the diagonal
// copy reads 4 bytes per stored real part and no column index, against 8
// for the sliced copy.
template <class G = GatherReadOnly>
__device__ __forceinline__ float2 dia_row(const CsrDev<float2>& A, int32_t s, int lane, int32_t r, const float2* x) {
  float2 acc = make_float2(0.f, 0.f);
  if (r < A.n) {
    const float* dv = A.dval + r;
#pragma unroll 9
    for (int32_t d = 0; d < A.ndia; ++d) {
      const int32_t j = r + __ldg(A.doff + d);
      const float a = __ldcs(dv + static_cast<size_t>(d) * A.dld);
      float2 xv = make_float2(0.f, 0.f);
      if (static_cast<uint32_t>(j) < static_cast<uint32_t>(A.n)) xv = G::ld(x + j);
      const float sx = fmaf(a, xv.x, acc.x), sy = fmaf(a, xv.y, acc.y);
      const bool nz = a != 0.f;
      acc.x = nz ? sx : acc.x;
      acc.y = nz ? sy : acc.y;
    }
  }
  const int32_t ib = A.isoff[s];
  return imag_row<float2, G>(A, ib, (A.isoff[s + 1] - ib) >> 5, lane, r, x, acc);
}

// Walk this thread's rows; for each row r < n call epi.prefetch(r) (before
// the row's sum, so the epilogue's own loads are in flight with it) and then
// epi.row(r, sum_k a_rk x_k).
template <class V, class Epi, class G = GatherReadOnly, int U = kSpmvUnroll>
__device__ __forceinline__ void spmv_run(const CsrDev<V>& A, const V* __restrict__ x, Epi& epi) {
  for (SliceRows q(A.n); q.active(); q.advance()) {
    const int32_t r = q.row();
    int32_t len = 0;
    if (r < A.n) {
      len = A.rowptr[r + 1] - A.rowptr[r];
      epi.prefetch(r);
    }
    V acc;
    if constexpr (std::is_same<V, float2>::value) {
      if (A.ndia > 0) acc = dia_row<G>(A, q.s, q.lane, r, x);
      else acc = sell_row<V, G, U>(A, slice_pos(A, q.s), q.lane, r, len, x);
    } else {
      acc = sell_row<V, G, U>(A, slice_pos(A, q.s), q.lane, r, len, x);
    }
    if (r < A.n) epi.row(r, acc);
  }
}

// Launch shape of the stand-alone product and the FP64 products of a refinement
// step: 1024 threads (32 warps), one block per SM (64 registers per thread at most).
// Measured on GB300 (120x60x50 cavity): with 256-thread blocks, four per SM, the warps'
// slice counts differed by one round and SMs idled 19 % of the SpMV.
template <class V> struct Engine {
  static constexpr int R = 32;  // rows per slice
  static constexpr int kThreads = 1024;
  static constexpr int kMinBlocks = 1;
};

// Device view of one value array of a handle (the caller's values, the
// complex64 copy or A D^-1) with the handle's SELL pattern.
template <class V>
inline CsrDev<V> csr_dev(const helm_csr_s* A, const V* vals, const SellVals& sv) {
  using R = typename RealOf<V>::T;
  const bool dia = sv.dval != nullptr && A->ndia > 0;
  return CsrDev<V>{A->n,        A->nnz,   A->rowptr,
                   A->colind,   vals,     A->nsl,
                   A->sell_off, A->sell_col, static_cast<const R*>(sv.sval),
                   sv.isoff,    sv.icol,  static_cast<const R*>(sv.ival),
                   sv.ilen,     dia ? A->ndia : 0, dia ? A->dia_off : nullptr, dia_ld(A->n),
                   dia ? static_cast<const R*>(sv.dval) : nullptr};
}

}  // namespace helm
