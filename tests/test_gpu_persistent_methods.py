"""TFQMR and BiCGStab(l) as persistent kernels (the default loop) against their
graph loop, on each shape of the solver grid: the same bits, and a solution
that meets the tolerance by the oracle's product."""
import numpy as np
import pytest

import helmgen as g
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402
from test_gpu_solver_shapes import SMS, _banded, _check  # noqa: E402

DEV = torch.device("cuda:0")
METHODS = [(helm.HELM_TFQMR, 2)] + [(helm.HELM_BICGSTABL, ell) for ell in (1, 2, 3, 4, 5, 8)]


def _both(rp, ci, v, seed, **kw):
    n = rp.size - 1
    A = helm.CsrMatrix.from_host(rp, ci, v, device=DEV)
    b = torch.as_tensor(g.complex_vector(n, seed), device=DEV)
    x0 = torch.as_tensor(0.1 * g.complex_vector(n, seed + 1), device=DEV)
    out = []
    for launch in (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_AUTO):
        x = x0.clone()
        out.append((x, helm.helm_bicgstab_solve(A.handle, b, x, helm.default_opts(launch=launch, **kw))))
    A.close()
    (xg, ig), (xa, ia) = out
    assert ia == ig
    assert torch.equal(torch.view_as_real(xg), torch.view_as_real(xa))
    bh, xh = b.cpu().numpy(), xa.cpu().numpy()
    return ia, np.linalg.norm(bh - oracle.spmv(rp, ci, v, xh)) / np.linalg.norm(bh)


@pytest.mark.parametrize("method,ell", METHODS)
@pytest.mark.parametrize("slices,extra", [(1, -31), (3, -5), (SMS, 1), (4 * SMS, 0), (4 * SMS, 33), (20 * SMS, 1),
                                          (150 * SMS, 1)])
@pytest.mark.parametrize("use_x0", [0, 1])
def test_persistent_is_the_graph(slices, extra, method, ell, use_x0):
    n = 32 * slices + extra
    offs = [o for o in (-70, -1, 0, 1, 70) if abs(o) < n]
    info, r = _both(*_banded(n, offs, lambda q: (q % 97 == 0) * 1.0, 3), seed=11, tol=1e-10, method=method, ell=ell,
                    use_x0=use_x0)
    # one unknown: the process may end exactly, on a zero Gram entry
    assert info["status"] == "ok" or (n == 1 and info["status"] == "breakdown"), info
    assert info["status"] != "ok" or r <= 1e-10 * (1 + 1e-6)


@pytest.mark.parametrize("method,ell", [(helm.HELM_TFQMR, 2), (helm.HELM_BICGSTABL, 4)])
@pytest.mark.parametrize("kw", [dict(tol=2e-16, maxit=60), dict(tol=1e-30, maxit=3), dict(tol=1e-10, maxit=0),
                                dict(tol=1e-15, deadline_s=1e-9), dict(tol=1e-9, precond=helm.HELM_PRECOND_JACOBI)])
def test_restarts_caps_and_options(method, ell, kw):
    """Restarts and checks near rounding level, iteration caps, an expired
    deadline, right Jacobi."""
    rp, ci, v = _banded(9000, [-40, -1, 0, 1, 40], lambda r: (r % 3 == 0) * 1.0, 7)
    _both(rp, ci, v, seed=8, method=method, ell=ell, use_x0=0, **kw)


@pytest.mark.parametrize("method,ell", [(helm.HELM_TFQMR, 2), (helm.HELM_BICGSTABL, 3)])
def test_zero_right_hand_side(method, ell):
    rp, ci, v = _banded(2000, [-1, 0, 1], lambda r: 1.0 * (r >= 0), 9)
    A = helm.CsrMatrix.from_host(rp, ci, v, device=DEV)
    b = torch.zeros(2000, dtype=torch.complex128, device=DEV)
    x = torch.ones_like(b)
    info = helm.helm_bicgstab_solve(A.handle, b, x, helm.default_opts(method=method, ell=ell, use_x0=1))
    assert info["status"] == "ok" and info["relres_true"] == 0.0
    assert not x.any()
    A.close()


@pytest.mark.parametrize("extra", [0, 1, 32 * SMS])
def test_bicgstab_at_a_full_round_of_the_mid_shape(extra):
    """24 slices per SM are one round of its warps."""
    _check(*_banded(32 * 24 * SMS + extra, [-70, -1, 0, 1, 70], lambda r: (r % 97 == 0) * 1.0, 3), seed=11)
