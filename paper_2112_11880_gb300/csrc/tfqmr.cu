// Complex128 TFQMR with device-resident scalars: the "P-TFQMR" of Section 4
// (identity preconditioner), following Freund 1993 / Saad 2003 Algorithm 7.8
// with conjugated inner products (r0, y) = sum conj(r0_i) y_i.
//
// One iteration = two half-steps = two products with A, in four steps:
//   T1  un = u - alpha v, w -= alpha Au, d = u + gamma d   + ||w||^2
//         -> theta, c, tau, eta (even half-step), quasi-residual bound
//   T2  Aun = A un;  x += eta d  (the even half-step's x update);
//       w -= alpha Aun, d = un + gamma d       + ||w||^2, (r0, w)
//         -> theta, c, tau, eta (odd half-step), rho, beta
//   T3  u = w + beta un;  x += eta d
//   T4  Au = A u;  v = Au + beta (Aun + beta v) + (r0, v) -> alpha, gamma
//   T5  only when a half-step's bound tau sqrt(m + 2) fell below tol ||b||:
//       true residual ||b - A x|| (one SpMV), convergence.  Then the iteration
//       cap, the deadline, the loop condition.
// The true-residual check runs once per iteration, after the odd half-step,
// so a solve can end one half-step later than a check after every half-step.
//
// The loop runs as one persistent cooperative kernel (four grid barriers an
// iteration), or as a graph or a host-driven loop of one kernel per step; same
// shapes, rows and sums as BiCGStab's (krylov.cuh), the same bits in each.
// What bounds it up to some 100,000 unknowns is the latency between steps.
// Measured, us per iteration, persistent / graph / before (six graph kernels on
// a grid of 1024-thread blocks): 20^3 box 28.7 / 39.8 / 53.0, 60x30x25 39.9 /
// 44.4 / 63.5, 80x40x32 57.3 / 63.4 / 77.4, 120x60x50 130 / 139 / 170,
// 200x100x80 519 / 533 / 552.
#include <cmath>
#include <cstring>

#include "krylov.cuh"

namespace helm {

namespace {

using V = double2;

struct TqArgs {
  CsrDev<V> A;
  const V* b;
  V* x;
  V *r0, *w, *u, *un, *v, *Au, *Aun, *d;
  SolverState* st;  // rho, alpha, beta; aux[0] = eta, aux[1] = (theta, tau), aux[2] = gamma, aux[3] = (check, start iteration)
  double* partials;
  unsigned int* tickets;
  unsigned int* dev_err;
  cudaGraphConditionalHandle cond;
  int has_cond;
};

__device__ __forceinline__ void tq_cond(const TqArgs& a, bool cont) {
  if (a.has_cond) cudaGraphSetConditional(a.cond, cont ? 1u : 0u);
}

// ---------------------------------------------------------------- scalar steps

// After a half-step: theta = ||w|| / tau, c = 1/sqrt(1 + theta^2),
// tau = tau theta c, eta = c^2 alpha; the bound tau sqrt(m + 2) <= tol ||b||
// (m = half-step index) raises the check flag.
__device__ __noinline__ void tq_half_step_scalars(SolverState* st, double ww, int m) {
  const double tau0 = st->aux[1].y;
  const double theta = sc_div(sc_sqrt(ww), tau0);
  const double c = sc_div(1.0, sc_sqrt(1.0 + theta * theta));
  const double tau = tau0 * theta * c;
  const double2 alpha = st->alpha;
  const double2 eta = make_double2(c * c * alpha.x, c * c * alpha.y);
  if (!isfinite(theta) || !isfinite(tau) || !cfinite(eta)) {
    st->status = HELM_ERR_NONFINITE;
    return;
  }
  st->aux[1] = make_double2(theta, tau);
  st->aux[0] = eta;
  const double bt = st->tol * st->bnorm;
  if (tau * tau * static_cast<double>(m + 2) <= bt * bt) st->aux[3].x = 1.0;
  st->relres = sc_div(tau * sc_sqrt(static_cast<double>(m + 2)), st->bnorm);
}

// gamma = (theta^2 / alpha) eta for the next d update
__device__ __noinline__ void tq_gamma(SolverState* st) {
  const double th = st->aux[1].x;
  const double2 q = cdiv_fast(make_double2(th * th, 0.0), st->alpha);
  st->aux[2] = cmul(q, st->aux[0]);
}
// half-step index of the even half-step of the current iteration
__device__ __forceinline__ int tq_m(const SolverState* st) {
  return 2 * (st->iter - 1 - static_cast<int32_t>(st->aux[3].y));
}

// after the initial residual: tot = (||b||^2, ||r0||^2, (r0, r0))
__device__ __forceinline__ void sc_tq_init(SolverState* st, const double (&tot)[4], int use_x0) {
  const double bnorm = sc_sqrt(tot[0]);
  st->bnorm = bnorm;
  if (use_x0) st->spmv_count += 1;
  int status = ST_RUNNING;
  if (!isfinite(bnorm)) {
    status = HELM_ERR_NONFINITE;
  } else if (bnorm == 0.0) {
    status = HELM_OK;
  } else {
    const double rn = sc_sqrt(tot[1]);
    st->relres = sc_div(rn, bnorm);
    if (!isfinite(rn)) status = HELM_ERR_NONFINITE;
    else if (rn <= st->tol * bnorm) status = HELM_OK;
    else if (st->maxit <= 0) status = HELM_ERR_NOT_CONVERGED;
    st->rho = make_double2(tot[2], tot[3]);
    st->aux[1] = make_double2(0.0, rn);  // theta = 0, tau = ||r0||
    st->aux[0] = make_double2(0.0, 0.0);  // eta
    st->aux[2] = make_double2(0.0, 0.0);  // gamma
    // check flag; iteration at which this (re)start began (the half-step
    // index m of the bound tau sqrt(m + 2) counts from there)
    st->aux[3] = make_double2(0.0, static_cast<double>(st->iter));
  }
  st->status = status;
}

// after v = A u of the start: tot = (r0, v)
__device__ __forceinline__ void sc_tq_sigma0(SolverState* st, const double (&tot)[2]) {
  st->spmv_count += 1;
  const double2 sigma = make_double2(tot[0], tot[1]);
  int status = ST_RUNNING;
  if (!cfinite(sigma) || !cfinite(st->rho)) status = HELM_ERR_NONFINITE;
  else if (czero(sigma) || czero(st->rho)) { status = HELM_ERR_BREAKDOWN; st->iter += 1; }
  else {
    st->alpha = cdiv_fast(st->rho, sigma);
    if (!cfinite(st->alpha)) status = HELM_ERR_NONFINITE;
  }
  st->status = status;
}

// after T1: tot = ||w||^2
__device__ __forceinline__ void sc_tq_even(SolverState* st, const double (&tot)[1]) {
  st->iter += 1;
  tq_half_step_scalars(st, tot[0], tq_m(st));
  if (st->status == ST_RUNNING) tq_gamma(st);  // gamma of the odd half-step's d update (same alpha)
}

// after T2: tot = (||w||^2, (r0, w))
__device__ __forceinline__ void sc_tq_odd(SolverState* st, const double (&tot)[3]) {
  st->spmv_count += 1;
  tq_half_step_scalars(st, tot[0], tq_m(st) + 1);
  if (st->status != ST_RUNNING) return;
  const double2 rho_new = make_double2(tot[1], tot[2]);
  if (!cfinite(rho_new)) {
    st->status = HELM_ERR_NONFINITE;
    return;
  }
  if (czero(st->rho)) {
    st->status = HELM_ERR_BREAKDOWN;
    return;
  }
  st->beta = cdiv_fast(rho_new, st->rho);
  st->rho = rho_new;
}

// after T4: tot = (r0, v)
__device__ __forceinline__ void sc_tq_sigma(SolverState* st, const double (&tot)[2]) {
  st->spmv_count += 1;
  const double2 sigma = make_double2(tot[0], tot[1]);
  if (!cfinite(sigma)) st->status = HELM_ERR_NONFINITE;
  else if (czero(sigma) || czero(st->rho)) st->status = HELM_ERR_BREAKDOWN;
  else {
    st->alpha = cdiv_fast(st->rho, sigma);
    if (!cfinite(st->alpha)) st->status = HELM_ERR_NONFINITE;
    else tq_gamma(st);
  }
}

__device__ __forceinline__ bool tq_check_due(const SolverState* st) {
  return st->status == ST_RUNNING && st->aux[3].x != 0.0;
}
// end of an iteration without a check; `late` = the deadline has passed
__device__ __forceinline__ void sc_tq_end(SolverState* st, bool late) {
  if (st->status != ST_RUNNING) return;
  if (st->iter >= st->maxit) st->status = HELM_ERR_NOT_CONVERGED;
  else if (late) st->status = HELM_ERR_TIMEOUT;
}
// after the check: rr = ||b - A x||^2
__device__ __forceinline__ void sc_tq_check(SolverState* st, double rr, bool late) {
  st->spmv_count += 1;
  const double rt = sc_div(sc_sqrt(rr), st->bnorm);
  st->aux[3].x = 0.0;
  int status = ST_RUNNING;
  if (!isfinite(rt)) status = HELM_ERR_NONFINITE;
  else if (rt <= st->tol) status = HELM_OK;
  else if (st->iter >= st->maxit) status = HELM_ERR_NOT_CONVERGED;
  else if (late) status = HELM_ERR_TIMEOUT;
  // the bound is below tol but the true residual is not: the recurrence has
  // drifted from b - A x, so the solve starts again from the current x
  else status = ST_RESTART;
  st->status = status;
}

// ---------------------------------------------------------------- steps
// The per-row work of each step, shared by all forms of the loop.
struct TqPhases {
  const TqArgs& a;
  PRows q;
  Own<V, 0> w;
  Own<V, 1> d;
  Own<V, 2> x;
  Own<V, 3> v;
  Own<V, 4> Aun;
  Own<V, 5> Au;
  Own<V, 6> r0;
  Own<V, 7> un;  // un and u: a copy beside the one that is gathered
  Own<V, 8> u;
  static constexpr int kOwn = 9;
  __device__ __forceinline__ TqPhases(const TqArgs& a_, const PLayout& L)
      : a(a_), q(L), w{a_.w, L}, d{a_.d, L}, x{a_.x, L}, v{a_.v, L}, Aun{a_.Aun, L}, Au{a_.Au, L}, r0{a_.r0, L},
        un{a_.un, L}, u{a_.u, L} {}

  // r0 = w = u = ri, d = 0 on row i; (||b||^2, ||r0||^2, (r0, r0))
  __device__ __forceinline__ void init_row(int32_t i, int li, V bi, V ri, double (&part)[4]) const {
    r0.st(i, li, ri);
    w.st(i, li, ri);
    u.st_both(i, li, ri);
    d.st(i, li, vzero<V>());
    part[0] = cabs2_acc(bi, part[0]);
    part[1] = cabs2_acc(ri, part[1]);
    const V s = cfma_conj(ri, ri, make_double2(part[2], part[3]));
    part[2] = s.x;
    part[3] = s.y;
  }
  // without x0: x = 0, r0 = b
  __device__ __forceinline__ void init_zero(double (&part)[4]) const {
    for_rows(q, a.A.n, [&](int32_t i, int li) {
      const V bi = a.b[i];
      x.st(i, li, vzero<V>());
      init_row(i, li, bi, bi, part);
    });
  }
  // with x0: r0 = b - A x
  __device__ __forceinline__ void row_init(int32_t i, int li, V ax, double (&part)[4]) const {
    const V bi = a.b[i];
    if (x.shared()) x.st(i, li, a.x[i]);
    init_row(i, li, bi, csub(bi, ax), part);
  }
  // v = Au = A u, (r0, v)
  __device__ __forceinline__ void row_sigma0(int32_t i, int li, V ax, double (&part)[4]) const {
    v.st(i, li, ax);
    Au.st(i, li, ax);
    const V s = cfma_conj(r0.ld(i, li), ax, make_double2(part[0], part[1]));
    part[0] = s.x;
    part[1] = s.y;
  }
  // T1
  __device__ __forceinline__ void upd_even(V alpha, V gamma, double (&part)[4]) const {
    for_rows(q, a.A.n, [&](int32_t i, int li) {
      const V ui = u.ld(i, li);
      un.st_both(i, li, cfms(alpha, v.ld(i, li), ui));
      const V wi = cfms(alpha, Au.ld(i, li), w.ld(i, li));
      w.st(i, li, wi);
      d.st(i, li, cfma(gamma, d.ld(i, li), ui));
      part[0] = cabs2_acc(wi, part[0]);
    });
  }
  // T2
  __device__ __forceinline__ void row_odd(int32_t i, int li, V ax, V alpha, V gamma, V eta, double (&part)[4]) const {
    Aun.st(i, li, ax);
    const V di = d.ld(i, li), uni = un.ld(i, li), r0i = r0.ld(i, li);
    x.st(i, li, cfma(eta, di, x.ld(i, li)));
    const V wi = cfms(alpha, ax, w.ld(i, li));
    w.st(i, li, wi);
    d.st(i, li, cfma(gamma, di, uni));
    part[0] = cabs2_acc(wi, part[0]);
    const V s = cfma_conj(r0i, wi, make_double2(part[1], part[2]));
    part[1] = s.x;
    part[2] = s.y;
  }
  // T3
  __device__ __forceinline__ void upd_u(V beta, V eta) const {
    for_rows(q, a.A.n, [&](int32_t i, int li) {
      u.st_both(i, li, cfma(beta, un.ld(i, li), w.ld(i, li)));
      x.st(i, li, cfma(eta, d.ld(i, li), x.ld(i, li)));
    });
  }
  // T4
  __device__ __forceinline__ void row_u(int32_t i, int li, V ax, V beta, double (&part)[4]) const {
    Au.st(i, li, ax);
    const V vn = cfma(beta, cfma(beta, v.ld(i, li), Aun.ld(i, li)), ax);
    v.st(i, li, vn);
    const V s = cfma_conj(r0.ld(i, li), vn, make_double2(part[0], part[1]));
    part[0] = s.x;
    part[1] = s.y;
  }
  // ||b - A x||^2
  __device__ __forceinline__ void row_res(int32_t i, V ax, double (&part)[4]) const {
    part[0] = cabs2_acc(csub(a.b[i], ax), part[0]);
  }
};

// ---------------------------------------------------------------- graph kernels

template <int S, class F>
__device__ __forceinline__ void tq_spmv(const TqPhases& ph, const V* x, F f) {
  spmv_rows<V, kSpmvUnroll, SolverBounds<S>::parts, GatherReadOnly>(ph.q, ph.a.A, x, [](int32_t) {}, f);
}
#define HELM_TQ_PHASES                      \
  const PLayout lay = graph_layout(a.A.n);  \
  const TqPhases ph(a, lay);                \
  double part[4] = {0.0, 0.0, 0.0, 0.0};

template <int S>
HELM_SOLVER_KERNEL k_tq_init_a(const __grid_constant__ TqArgs a) {
  __shared__ double red[32 * 4];
  SolverState* st = a.st;
  const int use_x0 = st->use_x0;
  HELM_TQ_PHASES
  if (use_x0) tq_spmv<S>(ph, a.x, [&](int32_t i, int li, V ax) { ph.row_init(i, li, ax, part); });
  else ph.init_zero(part);
  double tot[4];
  if (!grid_total_last<V, S, 4>(part, a.partials, a.tickets + TK_INIT, red, tot)) return;
  if (threadIdx.x == 0) sc_tq_init(st, tot, use_x0);
}

template <int S>
HELM_SOLVER_KERNEL k_tq_init_b(const __grid_constant__ TqArgs a) {
  __shared__ double red[32 * 2];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) {
    if (blockIdx.x == 0 && threadIdx.x == 0) tq_cond(a, false);
    return;
  }
  HELM_TQ_PHASES
  tq_spmv<S>(ph, a.u, [&](int32_t i, int li, V ax) { ph.row_sigma0(i, li, ax, part); });
  double part2[2] = {part[0], part[1]}, tot[2];
  if (!grid_total_last<V, S, 2>(part2, a.partials, a.tickets + TK_V, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_tq_sigma0(st, tot);
  tq_cond(a, st->status == ST_RUNNING);
}

// T1
template <int S>
HELM_SOLVER_KERNEL k_tq_even(const __grid_constant__ TqArgs a) {
  __shared__ double red[32];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  HELM_TQ_PHASES
  ph.upd_even(st->alpha, st->aux[2], part);
  double part1[1] = {part[0]}, tot[1];
  if (!grid_total_last<V, S, 1>(part1, a.partials, a.tickets + TK_S, red, tot)) return;
  if (threadIdx.x == 0) sc_tq_even(st, tot);
}

// T2
template <int S>
HELM_SOLVER_KERNEL k_tq_odd(const __grid_constant__ TqArgs a) {
  __shared__ double red[32 * 3];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  HELM_TQ_PHASES
  const V alpha = st->alpha, gamma = st->aux[2], eta = st->aux[0];
  tq_spmv<S>(ph, a.un, [&](int32_t i, int li, V ax) { ph.row_odd(i, li, ax, alpha, gamma, eta, part); });
  double part3[3] = {part[0], part[1], part[2]}, tot[3];
  if (!grid_total_last<V, S, 3>(part3, a.partials, a.tickets + TK_T, red, tot)) return;
  if (threadIdx.x == 0) sc_tq_odd(st, tot);
}

// T3
template <int S>
HELM_SOLVER_KERNEL k_tq_u(const __grid_constant__ TqArgs a) {
  const SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  const PLayout lay = graph_layout(a.A.n);
  TqPhases(a, lay).upd_u(st->beta, st->aux[0]);
}

// T4
template <int S>
HELM_SOLVER_KERNEL k_tq_spmv_u(const __grid_constant__ TqArgs a) {
  __shared__ double red[32 * 2];
  SolverState* st = a.st;
  if (st->status != ST_RUNNING) return;
  HELM_TQ_PHASES
  const V beta = st->beta;
  tq_spmv<S>(ph, a.u, [&](int32_t i, int li, V ax) { ph.row_u(i, li, ax, beta, part); });
  double part2[2] = {part[0], part[1]}, tot[2];
  if (!grid_total_last<V, S, 2>(part2, a.partials, a.tickets + TK_AUX1, red, tot)) return;
  if (threadIdx.x == 0) sc_tq_sigma(st, tot);
}

// T5
template <int S>
HELM_SOLVER_KERNEL k_tq_check(const __grid_constant__ TqArgs a) {
  __shared__ double red[32];
  SolverState* st = a.st;
  if (!tq_check_due(st)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      sc_tq_end(st, deadline_passed(st));
      tq_cond(a, st->status == ST_RUNNING);
    }
    return;
  }
  HELM_TQ_PHASES
  tq_spmv<S>(ph, a.x, [&](int32_t i, int, V ax) { ph.row_res(i, ax, part); });
  double part1[1] = {part[0]}, tot[1];
  if (!grid_total_last<V, S, 1>(part1, a.partials, a.tickets + TK_AUX2, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_tq_check(st, tot[0], deadline_passed(st));
  tq_cond(a, st->status == ST_RUNNING);
}

// tail: ||b - A x|| / ||b|| (x = 0 when b = 0)
template <int S>
HELM_SOLVER_KERNEL k_tq_tail(const __grid_constant__ TqArgs a) {
  __shared__ double red[32];
  SolverState* st = a.st;
  HELM_TQ_PHASES
  if (st->bnorm == 0.0) for_rows(ph.q, a.A.n, [&](int32_t i, int) { a.x[i] = vzero<V>(); });
  else tq_spmv<S>(ph, a.x, [&](int32_t i, int, V ax) { ph.row_res(i, ax, part); });
  double part1[1] = {part[0]}, tot[1];
  if (!grid_total_last<V, S, 1>(part1, a.partials, a.tickets + TK_TAIL, red, tot)) return;
  if (threadIdx.x == 0) sc_tail(st, tot);
}

// ---------------------------------------------------------------- persistent loop

// The whole solve, restarts included, as one cooperative kernel: a state machine
// over the steps above like BiCGStab's persist_loop (krylov.cuh), which says why
// it is built so.
enum : int { TQ_INIT = 0, TQ_INIT_X0, TQ_SIGMA0, TQ_EVEN, TQ_ODD, TQ_U, TQ_SPMV_U, TQ_FLUSH, TQ_CHECK, TQ_TAIL, TQ_END };
template <int S>
HELM_SOLVER_KERNEL k_tq_persistent(const __grid_constant__ TqArgs a, const __grid_constant__ PLayout L) {
  constexpr bool SPLIT = SolverBounds<S>::parts > 1;
  using G = GatherCoherent;
  __shared__ double red[32 * 4];
  __shared__ SolverState sst;
  __shared__ unsigned int s_target;  // arrivals of the barriers passed
  __shared__ int s_step;
  const TqPhases ph(a, L);
  copy_state(&sst, a.st);
  if (threadIdx.x == 0) s_target = 0u;
  persist_table<V>(ph.q, a.A);
  HeldPart held;
  if constexpr (SPLIT) held.load(ph.q, a.A);
  int buf = 0;
  int step = sst.use_x0 ? TQ_INIT_X0 : TQ_INIT;
  while (step != TQ_END) {
    double part[4] = {0.0, 0.0, 0.0, 0.0};
    if (step == TQ_EVEN) {
      ph.upd_even(sst.alpha, sst.aux[2], part);
    } else if (step == TQ_U) {
      ph.upd_u(sst.beta, sst.aux[0]);
    } else if (step == TQ_INIT) {
      ph.init_zero(part);
    } else if (step == TQ_FLUSH) {  // x is complete once every block is here
      if (sst.bnorm == 0.0) for_rows(ph.q, a.A.n, [&](int32_t i, int) { a.x[i] = vzero<V>(); });
      else if (ph.x.shared()) for_rows(ph.q, a.A.n, [&](int32_t i, int li) { a.x[i] = *ph.x.at(li); });
    } else if (step != TQ_TAIL || sst.bnorm != 0.0) {  // a product
      const V* in = step == TQ_ODD ? a.un : step == TQ_SPMV_U || step == TQ_SIGMA0 ? a.u : a.x;
      auto row = [&](int32_t i, int li, V ax) {
        const int st = opaque(step);
        if (st == TQ_ODD) ph.row_odd(i, li, ax, sst.alpha, sst.aux[2], sst.aux[0], part);
        else if (st == TQ_SPMV_U) ph.row_u(i, li, ax, sst.beta, part);
        else if (st == TQ_SIGMA0) ph.row_sigma0(i, li, ax, part);
        else if (st == TQ_INIT_X0) ph.row_init(i, li, ax, part);
        else ph.row_res(i, ax, part);
      };
      if constexpr (SPLIT) spmv_split<G>(ph.q, a.A, held, in, row);
      else spmv_rows<V, SolverBounds<S>::persist_u, 1, G>(ph.q, a.A, in, [](int32_t) {}, row);
      // the deadline is decided by block 0 and carried in the sums
      if (step == TQ_SPMV_U || step == TQ_CHECK)
        part[3] = (blockIdx.x == 0 && threadIdx.x == 0 && deadline_passed(&sst)) ? 1.0 : 0.0;
    }
    if (step == TQ_U || step == TQ_FLUSH) {
      if (!grid_barrier(a.tickets, a.dev_err, &s_target)) return;
      step = step == TQ_U ? TQ_SPMV_U : sst.status == ST_RUNNING ? TQ_CHECK : TQ_TAIL;
      continue;
    }
    buf ^= 1;
    double tot[4];
    if (!grid_total_all<V, S, 4>(part, a.partials + static_cast<size_t>(buf) * gridDim.x * 4, a.tickets, a.dev_err,
                                 &s_target, red, tot))
      return;
    if (threadIdx.x == 0) {
      const double t1[1] = {tot[0]}, t2[2] = {tot[0], tot[1]}, t3[3] = {tot[0], tot[1], tot[2]};
      const bool late = tot[3] > 0.0;
      int next = TQ_EVEN;
      if (step == TQ_EVEN) {
        sc_tq_even(&sst, t1);
        next = TQ_ODD;
      } else if (step == TQ_ODD) {
        sc_tq_odd(&sst, t3);
        next = TQ_U;
      } else if (step == TQ_SPMV_U) {
        sc_tq_sigma(&sst, t2);
        if (tq_check_due(&sst)) next = TQ_FLUSH;  // then the check
        else sc_tq_end(&sst, late);
      } else if (step == TQ_CHECK) {
        sc_tq_check(&sst, tot[0], late);
      } else if (step == TQ_SIGMA0) {
        sc_tq_sigma0(&sst, t2);
      } else if (step != TQ_TAIL) {
        sc_tq_init(&sst, tot, step == TQ_INIT_X0);
        next = TQ_SIGMA0;
      }
      if (sst.status != ST_RUNNING) next = step == TQ_CHECK ? TQ_TAIL : TQ_FLUSH;
      if (step == TQ_TAIL) {
        sc_tail(&sst, t1);
        next = TQ_END;
        if (sst.status == ST_RESTART) {  // (as the host does for the graph)
          next = TQ_INIT_X0;
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

using TqShapes = KShapes<V>;

void tq_init(const TqArgs& a, const TqShapes& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) {
    k_tq_init_a<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
    k_tq_init_b<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
  });
}
void tq_body(const TqArgs& a, const TqShapes& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) {
    k_tq_even<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
    k_tq_odd<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
    k_tq_u<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
    k_tq_spmv_u<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
    k_tq_check<S.value><<<sh.grid, sh.threads, 0, s>>>(a);
  });
}
void tq_tail(const TqArgs& a, const TqShapes& sh, cudaStream_t s) {
  with_shape(sh, [&](auto S) { k_tq_tail<S.value><<<sh.grid, sh.threads, 0, s>>>(a); });
}

}  // namespace

helm_status tfqmr_fp64(helm_csr A, const double2* b, double2* x, const helm_opts& o, helm_info* info,
                       cudaStream_t s) {
  helm_status st = ensure_vectors(A, kNumVec);
  if (st != HELM_OK) return st;
  TqShapes sh;
  HELM_TRY(krylov_shapes<V>(A, &sh));
  const size_t N = static_cast<size_t>(A->n);
  double2* W = A->vec;
  TqArgs a;
  std::memset(&a, 0, sizeof(a));
  a.A = csr_for(A, o);
  a.b = b;
  a.x = x;
  a.r0 = W;
  a.w = W + N;
  a.u = W + 2 * N;
  a.un = W + 3 * N;
  a.v = W + 4 * N;
  a.Au = W + 5 * N;
  a.Aun = W + 6 * N;
  a.d = W + 7 * N;
  a.st = A->state;
  a.partials = A->partials;
  a.tickets = A->tickets;
  a.dev_err = A->dev_err;

  SolverState* hs = A->state_host;
  unsigned int herr = 0;
  int32_t use_x0 = o.use_x0 ? 1 : 0, fresh = 1;
  HELM_CUDA_TRY(cudaMemsetAsync(A->dev_err, 0, sizeof(unsigned int), s));
  bool done = false;
  if (persist_default(A, sh, o)) {
    const void* fn = nullptr;
    int split = 1;
    with_shape(sh, [&](auto S) {
      fn = reinterpret_cast<const void*>(&k_tq_persistent<S.value>);
      split = SolverBounds<S.value>::parts;
    });
    PShape ps;
    if (persist_fit(fn, A, sh.grid, sh.threads, sh.bps, split, TqPhases::kOwn, sizeof(V), &ps)) {
      void* args[] = {&a, &ps.L};
      HELM_TRY(run_persistent(A, fn, args, ps, o, s, &done));
    }
  }

  // graph cache: key (b, x, variant), the variant tagged as TFQMR
  GraphEntry* g = nullptr;
  auto key = graph_key(b, x, 1, o);
  auto it = A->graphs.find(key);
  if (done || o.launch == HELM_LAUNCH_HOST) {
  } else if (it != A->graphs.end()) {
    g = &it->second;
  } else {
    auto with = [&](cudaGraphConditionalHandle c) {
      TqArgs aa = a;
      aa.cond = c;
      aa.has_cond = 1;
      return aa;
    };
    GraphEntry e;
    if (build_while_graph([&](cudaGraphConditionalHandle c, cudaStream_t cs) { tq_init(with(c), sh, cs); },
                          [&](cudaGraphConditionalHandle c, cudaStream_t cs) { tq_body(with(c), sh, cs); },
                          [&](cudaGraphConditionalHandle c, cudaStream_t cs) { tq_tail(with(c), sh, cs); },
                          &e) == HELM_OK) {
      bound_graphs(A, 1);
      g = &(A->graphs[key] = e);
    }
  }

  // an explicit graph request does not fall back to the host-driven loop
  if (!g && o.launch == HELM_LAUNCH_GRAPH) return HELM_ERR_CUDA;
  while (!done) {
    k_configure<<<1, 1, 0, s>>>(A->state, o.tol, o.maxit, use_x0, o.deadline_s, fresh);
    HELM_CUDA_TRY(cudaGetLastError());
    if (g) {
      HELM_CUDA_TRY(cudaGraphLaunch(g->exec, s));
    } else {
      tq_init(a, sh, s);
      for (;;) {
        for (int k = 0; k < 8; ++k) tq_body(a, sh, s);
        HELM_CUDA_TRY(cudaGetLastError());
        HELM_CUDA_TRY(cudaMemcpyAsync(hs, A->state, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
        HELM_CUDA_TRY(cudaStreamSynchronize(s));
        if (hs->status != ST_RUNNING) break;
      }
      tq_tail(a, sh, s);
    }
    HELM_CUDA_TRY(cudaMemcpyAsync(hs, A->state, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
    HELM_CUDA_TRY(cudaMemcpyAsync(&herr, A->dev_err, sizeof(unsigned int), cudaMemcpyDeviceToHost, s));
    HELM_CUDA_TRY(cudaStreamSynchronize(s));
    if (herr) return HELM_ERR_CUDA;
    if (hs->status != ST_RESTART) break;
    use_x0 = 1;  // start again from the current x, iterations counted on
    fresh = 0;
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
