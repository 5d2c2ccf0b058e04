// Complex128 BiCGStab solver (Section 4 of the paper: P-BiCGSTAB, residual
// tolerance, zero initial guess, iteration cap; identity preconditioner).
// The kernels are the precision-generic ones of krylov.cuh instantiated for
// complex128; this file adds the true-residual tail, the persistent
// (cooperative) form of the whole solve, the graph cache and the restart
// rule: a solve reports HELM_OK only when the true residual
// ||b - A x|| / ||b|| recomputed in FP64 is at most tol; when the recurrence
// converged but the true residual did not, the solve restarts from the
// current x while iterations remain.
#include <cmath>
#include <cstring>

#include "krylov.cuh"

namespace helm {

__global__ void k_configure(SolverState* st, double tol, int32_t maxit, int32_t use_x0, double deadline_s,
                            int32_t fresh) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  if (fresh) {
    st->iter = 0;
    st->spmv_count = 0;
    st->restarts = 0;
    st->t0 = globaltimer_ns();
  } else {
    st->restarts += 1;
  }
  st->tol = tol;
  st->maxit = maxit;
  st->use_x0 = use_x0;
  st->method = kModePlain;
  st->deadline_ns = deadline_s > 0.0 ? static_cast<unsigned long long>(deadline_s * 1e9) : 0ull;
  st->status = ST_RUNNING;
  st->phase = PH_RUN;
  st->relres = 0.0;
  st->relres_true = 0.0;
  const double2 one = make_double2(1.0, 0.0);
  st->rho = one;
  st->alpha = one;
  st->omega = one;
  st->beta = make_double2(0.0, 0.0);
}

namespace {

using V = double2;

// Tail: ||b - A x|| / ||b|| (x = 0 when b = 0).
template <class V, int S>
HELM_SOLVER_KERNEL k_tail(const __grid_constant__ KArgs<V> a) {
  __shared__ double red[32];
  SolverState* st = a.st;
  HELM_GRAPH_PHASES
  if (st->bnorm == 0.0) {
    for_rows(ph.q, a.A.n, [&](int32_t i, int) { a.x[i] = vzero<V>(); });
  } else {
    V bi = vzero<V>();
    graph_spmv<V, S>(
        ph, a.x, [&](int32_t i) { bi = a.b[i]; },
        [&](int32_t, int, V ax) { part[0] = cabs2_acc(csub(bi, ax), part[0]); });
  }
  double part1[1] = {part[0]}, tot[1];
  if (!grid_total_last<V, S, 1>(part1, a.partials, a.tickets + TK_TAIL, red, tot)) return;
  if (threadIdx.x != 0) return;
  sc_tail(st, tot);
}

// The whole solve (init, iterations, tail, restarts) as one cooperative kernel:
// persist_loop (krylov.cuh) on the solver grid.
template <int S>
HELM_SOLVER_KERNEL k_bicgstab_persistent(const __grid_constant__ KArgs<V> a, const __grid_constant__ PLayout L) {
  persist_loop<V, S>(a, L);
}

}  // namespace

helm_status bicgstab_fp64(helm_csr A, const double2* b, double2* x, const helm_opts& o, helm_info* info,
                          cudaStream_t s) {
  helm_status st = ensure_vectors(A, kNumVec);
  if (st != HELM_OK) return st;
  KShapes<V> sh;
  st = krylov_shapes<V>(A, &sh);
  if (st != HELM_OK) return st;
  const int32_t n = A->n;
  double2* W = A->vec;
  KArgs<V> a;
  std::memset(&a, 0, sizeof(a));
  a.A = csr_for(A, o);
  a.b = b;
  a.x = x;
  a.r = W;
  a.rh = W + (size_t)n;
  a.p = W + 2 * (size_t)n;
  a.v = W + 3 * (size_t)n;
  a.s = W + 4 * (size_t)n;
  a.t = W + 5 * (size_t)n;
  a.st = A->state;
  a.partials = A->partials;
  a.tickets = A->tickets;
  a.dev_err = A->dev_err;
  HELM_CUDA_TRY(cudaMemsetAsync(A->dev_err, 0, sizeof(unsigned int), s));
  const int32_t use_x0_first = o.use_x0 ? 1 : 0;
  SolverState* hs = A->state_host;
  unsigned int herr = 0;

  // persistent: the whole solve, restarts included, is one cooperative
  // launch; HELM_LAUNCH_AUTO takes it unless rows are long (persist_max_row)
  // or the device cannot run it
  bool done = false;
  if (o.launch == HELM_LAUNCH_PERSISTENT || persist_default(A, sh, o)) {
    const void* fn = nullptr;
    int split = 1;
    with_shape(sh, [&](auto S) {
      fn = reinterpret_cast<const void*>(&k_bicgstab_persistent<S.value>);
      split = SolverBounds<S.value>::parts;
    });
    PShape ps;
    if (persist_fit(fn, A, sh.grid, sh.threads, sh.bps, split, Phases<V>::kOwn, sizeof(V), &ps)) {
      void* args[] = {&a, &ps.L};
      HELM_TRY(run_persistent(A, fn, args, ps, o, s, &done));
    }
    if (!done && o.launch == HELM_LAUNCH_PERSISTENT) return HELM_ERR_CUDA;
  }

  if (!done) {
    struct Tail {
      KShapes<V> sh;
      void operator()(const KArgs<V>& ka, cudaStream_t ss) const {
        with_shape(sh, [&](auto S) { k_tail<V, S.value><<<sh.grid, sh.threads, 0, ss>>>(ka); });
      }
    } tail{sh};
    // Graph for this (b, x), built once and reused.
    GraphEntry* g = nullptr;
    const bool use_graph = o.launch != HELM_LAUNCH_HOST;
    auto key = graph_key(b, x, 0, o);
    auto it = A->graphs.find(key);
    if (!use_graph) {
    } else if (it != A->graphs.end()) {
      g = &it->second;
    } else {
      GraphEntry e;
      if (build_krylov_graph<V>(a, sh, tail, &e) == HELM_OK) {
        bound_graphs(A, 1);
        g = &(A->graphs[key] = e);
      }
    }
    // an explicit graph request does not fall back to the host-driven loop
    if (!g && o.launch == HELM_LAUNCH_GRAPH) return HELM_ERR_CUDA;
    int32_t use_x0 = use_x0_first;
    int32_t fresh = 1;
    for (;;) {
      k_configure<<<1, 1, 0, s>>>(A->state, o.tol, o.maxit, use_x0, o.deadline_s, fresh);
      HELM_CUDA_TRY(cudaGetLastError());
      st = run_krylov<V>(A, a, sh, g, tail, s);
      if (st != HELM_OK) return st;
      HELM_CUDA_TRY(cudaMemcpyAsync(hs, A->state, sizeof(SolverState), cudaMemcpyDeviceToHost, s));
      HELM_CUDA_TRY(cudaMemcpyAsync(&herr, A->dev_err, sizeof(unsigned int), cudaMemcpyDeviceToHost, s));
      HELM_CUDA_TRY(cudaStreamSynchronize(s));
      if (herr) return HELM_ERR_CUDA;
      if (restart_due(hs)) {
        use_x0 = 1;
        fresh = 0;
        continue;
      }
      break;
    }
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
