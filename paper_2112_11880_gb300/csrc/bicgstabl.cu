// Complex128 BiCGStab(l) with device-resident scalars: the "P-BiCGSTAB(l)"
// of Section 4 (identity preconditioner), after Sleijpen & Fokkema 1993.
//
// One iteration = one cycle = l BiCG steps (2 l products with A) and one
// minimal-residual step.  BiCG step j (B1..B4):
//   B1  u_i = r_i - beta u_i, i <= j
//   B2  u_{j+1} = A u_j          + (r~, u_{j+1})       -> alpha = rho0 / gamma
//   B3  r_i -= alpha u_{i+1}, i <= j;  x += alpha u_0  + ||r_0||^2 -> stop test
//   B4  r_{j+1} = A r_j          + (r~, r_{j+1})       -> rho1, beta
// Minimal-residual step (after B4 of j = l-1, r_{i+1} = A r_i and
// u_{i+1} = A u_i hold for i < l):
//   M1  Gram entries G_ik = (r_i, r_k), 0 <= i <= k, 1 <= k <= l, with the last
//       B4 (whose own sum is not needed: M2 forms the next rho1);
//       sum_k G_ik g_k = G_i0 (i = 1..l) is solved by Cholesky in FP64:
//       g minimises ||r_0 - sum g_k r_k||, omega = g_l
//   M2  x += sum g_k r_{k-1};  r_0 -= sum g_k r_k;  u_0 -= sum g_k u_k
//       + ||r_0||^2 and (r~, r_0) -> stop test, rho1 and beta of the next cycle
// The minimal-residual coefficients come from the normal equations instead of
// the modified Gram-Schmidt of the original algorithm: the same minimiser in
// exact arithmetic, one reduction pass instead of l(l-1)/2 dependent ones.
//
// The loop runs as one persistent cooperative kernel (4 l + 1 grid barriers a
// cycle), or as a graph or a host-driven loop of one kernel per step; same
// shapes, rows and sums as BiCGStab's (krylov.cuh), the same bits in each.  A
// small mesh is bound by the latency between steps, a large one by the FP64
// pipe (l = 4: 8 products of 39 us and some 230 FP64 instructions a row for the
// vectors on the 120x60x50 cavity, 0.49 ms a cycle).
// Measured, us per cycle, l = 4, persistent / graph / before (22 graph kernels,
// four of one thread): 20^3 box 123 / 158 / 282, 60x30x25 165 / 174 / 319,
// 80x40x32 246 / 263 / 375, 120x60x50 550 / 578 / 735, 200x100x80 2164 / 2167 /
// 2310.
#include <cmath>
#include <cstring>

#include "krylov.cuh"

namespace helm {

namespace {

using V = double2;
constexpr int kMaxEll = 8;
constexpr int kGram = kMaxEll * (kMaxEll + 3) / 2;  // Gram entries: 44
// Gram entries summed in one pass over the rows: (i0 .. i0 + 3, k)
constexpr int kGramPass = 4;

// Vectors by slot: x, r~, then r_0, u_0, r_1, u_1, ...: the first ones, used
// most, are kept in shared memory by a persistent kernel.
constexpr int SLOT_X = 0, SLOT_RT = 1;
__host__ __device__ __forceinline__ constexpr int slot_r(int i) { return 2 + 2 * i; }
__host__ __device__ __forceinline__ constexpr int slot_u(int i) { return 3 + 2 * i; }
constexpr int kSlots = slot_u(kMaxEll) + 1;

struct BlArgs {
  CsrDev<V> A;
  const V* b;
  V* vec[kSlots];
  int ell;
  SolverState* st;     // rho = rho0, alpha, omega, beta; aux[0] = rho1
  double* partials;
  double* gram;        // block partials of the Gram entries
  V* coef;             // g_1 .. g_l (graph)
  unsigned int* tickets;
  unsigned int* dev_err;
  cudaGraphConditionalHandle cond;
  int has_cond;
};

__device__ __forceinline__ void bl_cond(const BlArgs& a, bool cont) {
  if (a.has_cond) cudaGraphSetConditional(a.cond, cont ? 1u : 0u);
}

// ---------------------------------------------------------------- scalar steps

// after ||r_0||^2 is known: stop test (status) -- the caller keeps running otherwise
__device__ __noinline__ void bl_stop_test(SolverState* st, double r2) {
  const double bt = st->tol * st->bnorm;
  st->relres = sc_div(sc_sqrt(r2), st->bnorm);
  if (!isfinite(r2)) st->status = HELM_ERR_NONFINITE;
  else if (r2 <= bt * bt) st->status = HELM_OK;
}

// Before B1 of step j: at the start of a cycle rho0 = -omega rho0; then
// beta = alpha rho1 / rho0 and rho0 = rho1.
__device__ __noinline__ void sc_bl_beta(SolverState* st, int j) {
  if (j == 0) {
    st->iter += 1;
    st->rho = cmul(make_double2(-st->omega.x, -st->omega.y), st->rho);
  }
  const double2 rho1 = st->aux[0];
  if (!cfinite(rho1)) {
    st->status = HELM_ERR_NONFINITE;
    return;
  }
  if (czero(st->rho)) {
    st->status = HELM_ERR_BREAKDOWN;
    return;
  }
  st->beta = cmul(st->alpha, cdiv_fast(rho1, st->rho));
  st->rho = rho1;
}

// after the initial residual: tot = (||b||^2, ||r_0||^2, (r~, r_0)); rho0 = 1,
// alpha = 0, omega = 1; rho1 = (r~, r_0) for the first step
__device__ __forceinline__ void sc_bl_init(SolverState* st, const double (&tot)[4], int use_x0) {
  const double bnorm = sc_sqrt(tot[0]);
  st->bnorm = bnorm;
  if (use_x0) st->spmv_count += 1;
  st->status = ST_RUNNING;
  if (!isfinite(bnorm)) {
    st->status = HELM_ERR_NONFINITE;
  } else if (bnorm == 0.0) {
    st->status = HELM_OK;
  } else {
    bl_stop_test(st, tot[1]);
    if (st->status == ST_RUNNING && st->maxit <= 0) st->status = HELM_ERR_NOT_CONVERGED;
    st->rho = make_double2(1.0, 0.0);    // rho0
    st->alpha = make_double2(0.0, 0.0);
    st->omega = make_double2(1.0, 0.0);
    st->aux[0] = make_double2(tot[2], tot[3]);  // rho1 = (r~, r_0)
    if (st->status == ST_RUNNING) sc_bl_beta(st, 0);
  }
}

// after B2: tot = gamma
__device__ __forceinline__ void sc_bl_au(SolverState* st, const double (&tot)[2]) {
  st->spmv_count += 1;
  const double2 gamma = make_double2(tot[0], tot[1]);
  if (!cfinite(gamma)) st->status = HELM_ERR_NONFINITE;
  else if (czero(gamma)) st->status = HELM_ERR_BREAKDOWN;
  else st->alpha = cdiv_fast(st->rho, gamma);
}

// after B4 of step j < l - 1: tot = rho1 of the next BiCG step
__device__ __forceinline__ void sc_bl_ar(SolverState* st, const double (&tot)[2], int j) {
  st->spmv_count += 1;
  st->aux[0] = make_double2(tot[0], tot[1]);
  sc_bl_beta(st, j + 1);
}

// entry (i, k), i <= k, k >= 1, in the order of the passes
__device__ __forceinline__ int gram_entry(int i, int k) { return (k - 1) * (k + 2) / 2 + i; }

// after M1: the Gram entries -> coef (one thread; coef and the factor M in
// shared memory)
__device__ __noinline__ void sc_bl_gram(SolverState* st, const double* gram, int l, double2* coef,
                                        double2 (*M)[kMaxEll]) {
  st->spmv_count += 1;  // the B4 that it came with
  // G_ki = conj(G_ik)
  auto G = [&](int i, int k) -> double2 {
    const bool sw = i > k;
    const int e = sw ? gram_entry(k, i) : gram_entry(i, k);
    return make_double2(gram[2 * e], sw ? -gram[2 * e + 1] : gram[2 * e + 1]);
  };
  // Cholesky of the Hermitian matrix M_ik = G_ik (i, k = 1..l), column by
  // column, the diagonal's reciprocal on the diagonal; solve M g = c, c_i = G_i0
#pragma unroll 1
  for (int k = 0; k < l; ++k) {
#pragma unroll 1
    for (int i = k; i < l; ++i) {
      double2 s = G(i + 1, k + 1);
#pragma unroll 1
      for (int m = 0; m < k; ++m) s = csub(s, cmul(M[i][m], make_double2(M[k][m].x, -M[k][m].y)));
      if (i == k) {
        if (!(s.x > 0.0) || !isfinite(s.x)) {
          st->status = HELM_ERR_BREAKDOWN;
          return;
        }
        M[k][k] = make_double2(sc_div(1.0, sc_sqrt(s.x)), 0.0);
      } else {
        M[i][k] = make_double2(s.x * M[k][k].x, s.y * M[k][k].x);
      }
    }
  }
#pragma unroll 1
  for (int i = 0; i < l; ++i) {  // L y = c
    double2 s = G(i + 1, 0);
#pragma unroll 1
    for (int m = 0; m < i; ++m) s = csub(s, cmul(M[i][m], coef[m]));
    coef[i] = make_double2(s.x * M[i][i].x, s.y * M[i][i].x);
  }
  bool finite = true;
#pragma unroll 1
  for (int i = l - 1; i >= 0; --i) {  // L^H g = y
    double2 s = coef[i];
#pragma unroll 1
    for (int m = i + 1; m < l; ++m) s = csub(s, cmul(make_double2(M[m][i].x, -M[m][i].y), coef[m]));
    coef[i] = make_double2(s.x * M[i][i].x, s.y * M[i][i].x);
    finite = finite && cfinite(coef[i]);
  }
  if (!finite) {
    st->status = HELM_ERR_NONFINITE;
    return;
  }
  st->omega = coef[l - 1];
  if (czero(st->omega)) st->status = HELM_ERR_BREAKDOWN;
}

// after M2: tot = (||r_0||^2, (r~, r_0)); `late` = the deadline has passed
__device__ __forceinline__ void sc_bl_mr(SolverState* st, const double (&tot)[3], bool late) {
  bl_stop_test(st, tot[0]);
  st->aux[0] = make_double2(tot[1], tot[2]);
  if (st->status != ST_RUNNING) return;
  if (st->iter >= st->maxit) st->status = HELM_ERR_NOT_CONVERGED;
  else if (late) st->status = HELM_ERR_TIMEOUT;
  else sc_bl_beta(st, 0);
}

// ---------------------------------------------------------------- steps
// The per-row work of each step, shared by all forms of the loop.  B1 to M2 of
// a row are the same thread's, so only what a product gathers (u_j, r_j, x) has
// to be in global memory.
struct BlPhases {
  const BlArgs& a;
  PRows q;
  __device__ __forceinline__ BlPhases(const BlArgs& a_, const PLayout& L) : a(a_), q(L) {}
  __device__ __forceinline__ bool shared(int slot) const { return slot < opaque(q.L.nown); }
  __device__ __forceinline__ V* at(int slot, int li) const {
    return reinterpret_cast<V*>(persist_smem + q.L.own_at) + slot * q.L.own_len + li;
  }
  __device__ __forceinline__ V* ptr(int slot, int32_t i, int li) const {
    return shared(slot) ? at(slot, li) : a.vec[slot] + i;
  }
  __device__ __forceinline__ V ld(int slot, int32_t i, int li) const { return *ptr(slot, i, li); }
  __device__ __forceinline__ void st(int slot, int32_t i, int li, V v) const { *ptr(slot, i, li) = v; }
  __device__ __forceinline__ void st_both(int slot, int32_t i, int li, V v) const {
    a.vec[slot][i] = v;
    if (shared(slot)) *at(slot, li) = v;
  }

  // r_0 = r~ = ri, u_0 = 0; (||b||^2, ||r_0||^2, (r~, r_0))
  __device__ __forceinline__ void init_row(int32_t i, int li, V bi, V ri, double (&part)[4]) const {
    st(slot_r(0), i, li, ri);
    st(SLOT_RT, i, li, ri);
    st(slot_u(0), i, li, vzero<V>());
    part[0] = cabs2_acc(bi, part[0]);
    part[1] = cabs2_acc(ri, part[1]);
    const V s = cfma_conj(ri, ri, make_double2(part[2], part[3]));
    part[2] = s.x;
    part[3] = s.y;
  }
  __device__ __forceinline__ void init_zero(double (&part)[4]) const {
    for_rows(q, a.A.n, [&](int32_t i, int li) {
      const V bi = a.b[i];
      st(SLOT_X, i, li, vzero<V>());
      init_row(i, li, bi, bi, part);
    });
  }
  __device__ __forceinline__ void row_init(int32_t i, int li, V ax, double (&part)[4]) const {
    const V bi = a.b[i];
    if (shared(SLOT_X)) *at(SLOT_X, li) = a.vec[SLOT_X][i];
    init_row(i, li, bi, csub(bi, ax), part);
  }
  // B1
  __device__ __forceinline__ void upd_u(int j, V beta) const {
    for_rows(q, a.A.n, [&](int32_t i, int li) {
#pragma unroll 1
      for (int k = 0; k < j; ++k) st(slot_u(k), i, li, cfms(beta, ld(slot_u(k), i, li), ld(slot_r(k), i, li)));
      st_both(slot_u(j), i, li, cfms(beta, ld(slot_u(j), i, li), ld(slot_r(j), i, li)));
    });
  }
  // B2 and B4: out = ax, (r~, ax)
  __device__ __forceinline__ void row_prod(int out, int32_t i, int li, V ax, double (&part)[4]) const {
    st(out, i, li, ax);
    const V s = cfma_conj(ld(SLOT_RT, i, li), ax, make_double2(part[0], part[1]));
    part[0] = s.x;
    part[1] = s.y;
  }
  // B3
  __device__ __forceinline__ void upd_r(int j, V alpha, double (&part)[4]) const {
    for_rows(q, a.A.n, [&](int32_t i, int li) {
#pragma unroll 1
      for (int k = 0; k <= j; ++k) {
        const V rk = cfms(alpha, ld(slot_u(k + 1), i, li), ld(slot_r(k), i, li));
        if (k == 0) part[0] = cabs2_acc(rk, part[0]);
        if (k == j) st_both(slot_r(k), i, li, rk);
        else st(slot_r(k), i, li, rk);
      }
      st(SLOT_X, i, li, cfma(alpha, ld(slot_u(0), i, li), ld(SLOT_X, i, li)));
    });
  }
  // M1: this block's partials of every entry, component-major (whole block);
  // red holds 2 x 32 x 4 doubles
  template <int S>
  __device__ __forceinline__ void gram(double* red) const {
    const int l = a.ell;
    const size_t G = gridDim.x;
    double* out = a.gram;
    int half = 0;
#pragma unroll 1
    for (int k = 1; k <= l; ++k) {
#pragma unroll 1
      for (int i0 = 0; i0 <= k; i0 += kGramPass) {
        double g[kGramPass][2];
#pragma unroll
        for (int u = 0; u < kGramPass; ++u) g[u][0] = g[u][1] = 0.0;
        for_rows(q, a.A.n, [&](int32_t i, int li) {
          const V rk = ld(slot_r(k), i, li);
#pragma unroll
          for (int u = 0; u < kGramPass; ++u) {
            if (i0 + u < k) {
              const V s = cfma_conj(ld(slot_r(i0 + u), i, li), rk, make_double2(g[u][0], g[u][1]));
              g[u][0] = s.x;
              g[u][1] = s.y;
            } else if (i0 + u == k) {
              g[u][0] = cabs2_acc(rk, g[u][0]);
            }
          }
        });
        // two entries at a time; the two halves of `red` alternate, so a half is
        // written again only after a barrier that its readers have passed
#pragma unroll
        for (int u = 0; u < kGramPass; u += 2) {
          if (i0 + u + 1 <= k) {
            double v[4] = {g[u][0], g[u][1], g[u + 1][0], g[u + 1][1]};
            put_block_partials<V, S, 4>(v, red + half, out);
            out += 4 * G;
          } else if (i0 + u <= k) {
            double v[2] = {g[u][0], g[u][1]};
            put_block_partials<V, S, 2>(v, red + half, out);
            out += 2 * G;
          } else {
            continue;
          }
          half ^= 128;
        }
      }
    }
  }
  // M2
  __device__ __forceinline__ void upd_mr(const V* g, double (&part)[4]) const {
    for_rows(q, a.A.n, [&](int32_t i, int li) {
      V xq = ld(SLOT_X, i, li), r0 = ld(slot_r(0), i, li), u0 = ld(slot_u(0), i, li);
      V rprev = r0;
#pragma unroll 1
      for (int k = 1; k <= a.ell; ++k) {
        const V gk = g[k - 1], rk = ld(slot_r(k), i, li);
        xq = cfma(gk, rprev, xq);
        r0 = cfms(gk, rk, r0);
        u0 = cfms(gk, ld(slot_u(k), i, li), u0);
        rprev = rk;
      }
      st(SLOT_X, i, li, xq);
      st(slot_r(0), i, li, r0);
      st(slot_u(0), i, li, u0);
      part[0] = cabs2_acc(r0, part[0]);
      const V s = cfma_conj(ld(SLOT_RT, i, li), r0, make_double2(part[1], part[2]));
      part[1] = s.x;
      part[2] = s.y;
    });
  }
  __device__ __forceinline__ void row_res(int32_t i, V ax, double (&part)[4]) const {
    part[0] = cabs2_acc(csub(a.b[i], ax), part[0]);
  }
};

// ---------------------------------------------------------------- graph kernels

template <int S, class F>
__device__ __forceinline__ void bl_spmv(const BlPhases& ph, const V* x, F f) {
  spmv_rows<V, kSpmvUnroll, SolverBounds<S>::parts, GatherReadOnly>(ph.q, ph.a.A, x, [](int32_t) {}, f);
}
#define HELM_BL_PHASES                      \
  const PLayout lay = graph_layout(a.A.n);  \
  const BlPhases ph(a, lay);                \
  double part[4] = {0.0, 0.0, 0.0, 0.0};

template <int S>
HELM_SOLVER_KERNEL k_bl_init(const __grid_constant__ BlArgs a) {
  __shared__ double red[32 * 4];
  SolverState* st = a.st;
  const int use_x0 = st->use_x0;
  HELM_BL_PHASES
  if (use_x0) bl_spmv<S>(ph, a.vec[SLOT_X], [&](int32_t i, int li, V ax) { ph.row_init(i, li, ax, part); });
  else ph.init_zero(part);
  double tot[4];
  if (!grid_total_last<V, S, 4>(part, a.partials, a.tickets + TK_INIT, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_bl_init(st, tot, use_x0);
  bl_cond(a, st->status == ST_RUNNING);
}

// B1
template <int S>
HELM_SOLVER_KERNEL k_bl_u(const __grid_constant__ BlArgs a, int j) {
  const SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  const PLayout lay = graph_layout(a.A.n);
  BlPhases(a, lay).upd_u(j, st->beta);
}

// B2
template <int S>
HELM_SOLVER_KERNEL k_bl_au(const __grid_constant__ BlArgs a, int j) {
  __shared__ double red[32 * 2];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  HELM_BL_PHASES
  bl_spmv<S>(ph, a.vec[slot_u(j)], [&](int32_t i, int li, V ax) { ph.row_prod(slot_u(j + 1), i, li, ax, part); });
  double part2[2] = {part[0], part[1]}, tot[2];
  if (!grid_total_last<V, S, 2>(part2, a.partials, a.tickets + TK_V, red, tot)) return;
  if (threadIdx.x == 0) sc_bl_au(st, tot);
}

// B3
template <int S>
HELM_SOLVER_KERNEL k_bl_r(const __grid_constant__ BlArgs a, int j) {
  __shared__ double red[32];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  HELM_BL_PHASES
  ph.upd_r(j, st->alpha, part);
  double part1[1] = {part[0]}, tot[1];
  if (!grid_total_last<V, S, 1>(part1, a.partials, a.tickets + TK_S, red, tot)) return;
  if (threadIdx.x == 0) bl_stop_test(st, tot[0]);
}

// B4, and M1 with the last one
template <int S>
HELM_SOLVER_KERNEL k_bl_ar(const __grid_constant__ BlArgs a, int j) {
  __shared__ double red[2 * 32 * 4];
  __shared__ double gram[2 * kGram];
  __shared__ double2 M[kMaxEll][kMaxEll], coef[kMaxEll];
  __shared__ bool s_last;
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  HELM_BL_PHASES
  bl_spmv<S>(ph, a.vec[slot_r(j)], [&](int32_t i, int li, V ax) { ph.row_prod(slot_r(j + 1), i, li, ax, part); });
  if (j + 1 < a.ell) {
    double part2[2] = {part[0], part[1]}, tot[2];
    if (!grid_total_last<V, S, 2>(part2, a.partials, a.tickets + TK_T, red, tot)) return;
    if (threadIdx.x == 0) sc_bl_ar(st, tot, j);
    return;
  }
  ph.gram<S>(red);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(a.tickets + TK_AUX2, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  sum_components(a.gram, gridDim.x, a.ell * (a.ell + 3), gram);
  if (threadIdx.x != 0) return;
  a.tickets[TK_AUX2] = 0u;
  sc_bl_gram(st, gram, a.ell, coef, M);
  for (int k = 0; k < a.ell; ++k) a.coef[k] = coef[k];
}

// M2
template <int S>
HELM_SOLVER_KERNEL k_bl_mr(const __grid_constant__ BlArgs a) {
  __shared__ double red[32 * 3];
  __shared__ V gs[kMaxEll];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) {
    if (blockIdx.x == 0 && threadIdx.x == 0) bl_cond(a, false);
    return;
  }
  if (threadIdx.x < a.ell) gs[threadIdx.x] = a.coef[threadIdx.x];
  __syncthreads();
  HELM_BL_PHASES
  ph.upd_mr(gs, part);
  double part3[3] = {part[0], part[1], part[2]}, tot[3];
  if (!grid_total_last<V, S, 3>(part3, a.partials, a.tickets + TK_XR, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_bl_mr(st, tot, deadline_passed(st));
  bl_cond(a, st->status == ST_RUNNING);
}

// tail: true residual (x = 0 when b = 0)
template <int S>
HELM_SOLVER_KERNEL k_bl_tail(const __grid_constant__ BlArgs a) {
  __shared__ double red[32];
  SolverState* st = a.st;
  HELM_BL_PHASES
  if (st->bnorm == 0.0) for_rows(ph.q, a.A.n, [&](int32_t i, int) { a.vec[SLOT_X][i] = vzero<V>(); });
  else bl_spmv<S>(ph, a.vec[SLOT_X], [&](int32_t i, int, V ax) { ph.row_res(i, ax, part); });
  double part1[1] = {part[0]}, tot[1];
  if (!grid_total_last<V, S, 1>(part1, a.partials, a.tickets + TK_TAIL, red, tot)) return;
  if (threadIdx.x == 0) sc_tail(st, tot);
}

// ---------------------------------------------------------------- persistent loop

// The whole solve, restarts included, as one cooperative kernel: a state machine
// over the steps above (step kind + 16 j) like BiCGStab's persist_loop
// (krylov.cuh), which says why it is built so.
enum : int { BL_INIT = 0, BL_INIT_X0, BL_U, BL_AU, BL_R, BL_AR, BL_MR, BL_FLUSH, BL_TAIL, BL_END };
template <int S>
HELM_SOLVER_KERNEL k_bl_persistent(const __grid_constant__ BlArgs a, const __grid_constant__ PLayout L) {
  constexpr bool SPLIT = SolverBounds<S>::parts > 1;
  using G = GatherCoherent;
  __shared__ double red[2 * 32 * 4];
  __shared__ double gram[2 * kGram];
  __shared__ double2 M[kMaxEll][kMaxEll], coef[kMaxEll];
  __shared__ SolverState sst;
  __shared__ unsigned int s_target;  // arrivals of the barriers passed
  __shared__ int s_step;
  const BlPhases ph(a, L);
  copy_state(&sst, a.st);
  if (threadIdx.x == 0) s_target = 0u;
  persist_table<V>(ph.q, a.A);
  HeldPart held;
  if constexpr (SPLIT) held.load(ph.q, a.A);
  int buf = 0;
  int step = sst.use_x0 ? BL_INIT_X0 : BL_INIT;
  while (step != BL_END) {
    const int kind = step & 15, j = step >> 4;
    const bool m1 = kind == BL_AR && j + 1 == a.ell;
    double part[4] = {0.0, 0.0, 0.0, 0.0};
    if (kind == BL_U) {
      ph.upd_u(j, sst.beta);
    } else if (kind == BL_R) {
      ph.upd_r(j, sst.alpha, part);
    } else if (kind == BL_MR) {
      ph.upd_mr(coef, part);
      part[3] = (blockIdx.x == 0 && threadIdx.x == 0 && deadline_passed(&sst)) ? 1.0 : 0.0;
    } else if (kind == BL_INIT) {
      ph.init_zero(part);
    } else if (kind == BL_FLUSH) {  // x is complete once every block is here
      if (sst.bnorm == 0.0) for_rows(ph.q, a.A.n, [&](int32_t i, int) { a.vec[SLOT_X][i] = vzero<V>(); });
      else if (ph.shared(SLOT_X))
        for_rows(ph.q, a.A.n, [&](int32_t i, int li) { a.vec[SLOT_X][i] = *ph.at(SLOT_X, li); });
    } else if (kind != BL_TAIL || sst.bnorm != 0.0) {  // a product
      const int in = kind == BL_AU ? slot_u(j) : kind == BL_AR ? slot_r(j) : SLOT_X;
      auto row = [&](int32_t i, int li, V ax) {
        const int st = opaque(kind);
        if (st == BL_AU || st == BL_AR) ph.row_prod(in + 2, i, li, ax, part);  // u_{j+1}, r_{j+1}
        else if (st == BL_INIT_X0) ph.row_init(i, li, ax, part);
        else ph.row_res(i, ax, part);
      };
      if constexpr (SPLIT) spmv_split<G>(ph.q, a.A, held, a.vec[in], row);
      else spmv_rows<V, SolverBounds<S>::persist_u, 1, G>(ph.q, a.A, a.vec[in], [](int32_t) {}, row);
    }
    if (m1) ph.gram<S>(red);
    if (kind == BL_U || kind == BL_FLUSH || m1) {
      if (!grid_barrier(a.tickets, a.dev_err, &s_target)) return;
      if (!m1) {
        step = kind == BL_U ? BL_AU + 16 * j : BL_TAIL;
        continue;
      }
      sum_components(a.gram, gridDim.x, a.ell * (a.ell + 3), gram);
    }
    double tot[4] = {0.0, 0.0, 0.0, 0.0};
    if (!m1) {
      buf ^= 1;
      if (!grid_total_all<V, S, 4>(part, a.partials + static_cast<size_t>(buf) * gridDim.x * 4, a.tickets, a.dev_err,
                                   &s_target, red, tot))
        return;
    }
    if (threadIdx.x == 0) {
      const double t1[1] = {tot[0]}, t2[2] = {tot[0], tot[1]}, t3[3] = {tot[0], tot[1], tot[2]};
      int next = BL_U;
      if (kind == BL_AU) {
        sc_bl_au(&sst, t2);
        next = BL_R + 16 * j;
      } else if (kind == BL_R) {
        bl_stop_test(&sst, tot[0]);
        next = BL_AR + 16 * j;
      } else if (m1) {
        sc_bl_gram(&sst, gram, a.ell, coef, M);
        next = BL_MR;
      } else if (kind == BL_AR) {
        sc_bl_ar(&sst, t2, j);
        next = BL_U + 16 * (j + 1);
      } else if (kind == BL_MR) {
        sc_bl_mr(&sst, t3, tot[3] > 0.0);
      } else if (kind != BL_TAIL) {
        sc_bl_init(&sst, tot, kind == BL_INIT_X0);
      }
      if (sst.status != ST_RUNNING) next = BL_FLUSH;
      if (kind == BL_TAIL) {
        sc_tail(&sst, t1);
        next = BL_END;
        if (restart_due(&sst)) {  // (as the host does for the graph)
          next = BL_INIT_X0;
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

void bl_init(const BlArgs& a, const KShapes<V>& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) { k_bl_init<S.value><<<sh.grid, sh.threads, 0, s>>>(a); });
}
void bl_body(const BlArgs& a, const KShapes<V>& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) {
    for (int j = 0; j < a.ell; ++j) {
      k_bl_u<S.value><<<sh.grid, sh.threads, 0, s>>>(a, j);
      k_bl_au<S.value><<<sh.grid, sh.threads, 0, s>>>(a, j);
      k_bl_r<S.value><<<sh.grid, sh.threads, 0, s>>>(a, j);
      k_bl_ar<S.value><<<sh.grid, sh.threads, 0, s>>>(a, j);
    }
    k_bl_mr<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
  });
}
void bl_tail(const BlArgs& a, const KShapes<V>& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) { k_bl_tail<S.value><<<sh.grid, sh.threads, 0, s>>>(a); });
}

}  // namespace

helm_status bicgstabl_fp64(helm_csr A, const double2* b, double2* x, const helm_opts& o, helm_info* info,
                           cudaStream_t s) {
  const int ell = o.ell;
  if (ell < 1 || ell > kMaxEll) return HELM_ERR_INVALID;
  const int nvec = 2 * (ell + 1) + 1;
  helm_status st = ensure_vectors(A, nvec > kNumVec ? nvec : kNumVec);
  if (st != HELM_OK) return st;
  KShapes<V> sh;
  HELM_TRY(krylov_shapes<V>(A, &sh));
  const size_t N = static_cast<size_t>(A->n);
  double2* W = A->vec;
  BlArgs a;
  std::memset(&a, 0, sizeof(a));
  a.A = csr_for(A, o);
  a.b = b;
  a.vec[SLOT_X] = x;
  for (int k = SLOT_RT; k <= slot_u(ell); ++k) a.vec[k] = W + (k - SLOT_RT) * N;
  a.ell = ell;
  a.st = A->state;
  // partials: two buffers of four sums a block, the Gram entries, the coefficients
  a.partials = A->partials;
  a.gram = a.partials + 2 * 4 * static_cast<size_t>(sh.grid);
  a.coef = reinterpret_cast<V*>(a.gram + 2 * kGram * static_cast<size_t>(sh.grid));
  static_assert((2 * 4 + 2 * kGram) * SolverBounds<SHAPE_LARGE>::blocks + 2 * kMaxEll <= kPartialsPerSm,
                "the handle's partial sums hold them");
  a.tickets = A->tickets;
  a.dev_err = A->dev_err;

  SolverState* hs = A->state_host;
  HELM_CUDA_TRY(cudaMemsetAsync(A->dev_err, 0, sizeof(unsigned int), s));
  bool done = false;
  if (persist_default(A, sh, o)) {
    const void* fn = nullptr;
    int split = 1;
    with_shape(sh, [&](auto S) {
      fn = reinterpret_cast<const void*>(&k_bl_persistent<S.value>);
      split = SolverBounds<S.value>::parts;
    });
    PShape ps;
    if (persist_fit(fn, A, sh.grid, sh.threads, sh.bps, split, slot_u(ell) + 1, sizeof(V), &ps)) {
      void* args[] = {&a, &ps.L};
      HELM_TRY(run_persistent(A, fn, args, ps, o, s, &done));
    }
  }

  GraphEntry* g = nullptr;
  auto key = graph_key(b, x, 4 + ell, o);
  auto it = A->graphs.find(key);
  if (done || o.launch == HELM_LAUNCH_HOST) {
  } else if (it != A->graphs.end()) {
    g = &it->second;
  } else {
    auto with = [&](cudaGraphConditionalHandle c) {
      BlArgs aa = a;
      aa.cond = c;
      aa.has_cond = 1;
      return aa;
    };
    GraphEntry e;
    if (build_while_graph(
            [&](cudaGraphConditionalHandle c, cudaStream_t cs) {
              bl_init(with(c), sh, cs);
            },
            [&](cudaGraphConditionalHandle c, cudaStream_t cs) { bl_body(with(c), sh, cs); },
            [&](cudaGraphConditionalHandle c, cudaStream_t cs) { bl_tail(with(c), sh, cs); },
            &e) == HELM_OK) {
      bound_graphs(A, 1);
      g = &(A->graphs[key] = e);
    }
  }

  // an explicit graph request does not fall back to the host-driven loop
  if (!g && o.launch == HELM_LAUNCH_GRAPH) return HELM_ERR_CUDA;
  // restart from x while the recurrence converged but the true residual did
  // not (and iterations remain), as for BiCGStab
  for (int32_t use_x0 = o.use_x0 ? 1 : 0, fresh = 1; !done; use_x0 = 1, fresh = 0) {
    k_configure<<<1, 1, 0, s>>>(A->state, o.tol, o.maxit, use_x0, o.deadline_s, fresh);
    HELM_CUDA_TRY(cudaGetLastError());
    if (g) {
      HELM_CUDA_TRY(cudaGraphLaunch(g->exec, s));
    } else {
      bl_init(a, sh, s);
      for (;;) {
        for (int q = 0; q < 4; ++q) bl_body(a, sh, s);
        HELM_CUDA_TRY(cudaGetLastError());
        HELM_CUDA_TRY(cudaMemcpyAsync(hs, A->state, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
        HELM_CUDA_TRY(cudaStreamSynchronize(s));
        if (hs->status != ST_RUNNING) break;
      }
      bl_tail(a, sh, s);
    }
    unsigned int herr = 0;
    HELM_CUDA_TRY(cudaMemcpyAsync(hs, A->state, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
    HELM_CUDA_TRY(cudaMemcpyAsync(&herr, A->dev_err, sizeof(unsigned int), cudaMemcpyDeviceToHost, s));
    HELM_CUDA_TRY(cudaStreamSynchronize(s));
    if (herr) return HELM_ERR_CUDA;
    if (!(hs->status == HELM_OK && hs->relres_true > o.tol && hs->iter < o.maxit)) break;
  }
  helm_status result = hs->status == ST_RUNNING ? HELM_ERR_CUDA : static_cast<helm_status>(hs->status);
  if (result == HELM_OK && !(hs->relres_true <= o.tol)) result = HELM_ERR_NOT_CONVERGED;
  if (info) {
    info->iters = hs->iter;
    info->restarts = hs->restarts;
    info->relres_recur = hs->relres;
    info->relres_true = hs->relres_true;
    info->status = result;
    info->spmv_count = hs->spmv_count;
  }
  return result;
}

}  // namespace helm
