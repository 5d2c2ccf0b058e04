"""FP64 BiCGStab when (r^, r) vanishes exactly after an iteration: every loop form
starts again from x, at the same iteration, on each shape of the grid, and ends at
the cap where that comes first; the oracle does the same."""
import os
import sys

import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
from vanishing_rho import blocks  # noqa: E402

DEV = torch.device("cuda:0")
FORMS = (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_HOST, helm.HELM_LAUNCH_PERSISTENT, helm.HELM_LAUNCH_AUTO)


def _solve_all(A, b, **kw):
    out = [helm.solve(A, b, launch=l, **kw) for l in FORMS]
    for x, i in out[1:]:
        assert i == out[0][1]
        assert torch.equal(torch.view_as_real(x), torch.view_as_real(out[0][0]))
    return out[0]


@pytest.mark.parametrize("m,pad", [(1, 0), (4, 5), (1024, 77), (65536, 1), (262144, 0)])
def test_every_form_restarts(m, pad):
    rp, ci, v, bh = blocks(m, pad)
    A = helm.CsrMatrix.from_host(rp, ci, v, device=DEV)
    b = torch.as_tensor(bh, device=DEV)
    x, info = _solve_all(A, b, tol=1e-12, maxit=100)
    assert info["status"] == "ok" and info["restarts"] >= 1
    r = b - A.matvec(x)
    assert torch.linalg.vector_norm(r).item() <= 1.000001e-12 * torch.linalg.vector_norm(b).item()
    if m <= 1024:
        _, ref = oracle.bicgstab(rp, ci, v, bh, tol=1e-12, maxit=100)
        assert ref["status"] == "ok" and abs(ref["iters"] - info["iters"]) <= 1
    # the cap on, just after and one past the iteration that meets the zero
    for maxit, restarts in ((1, 0), (2, 0), (3, 1)):
        x, info = _solve_all(A, b, tol=1e-12, maxit=maxit)
        assert (info["status"], info["iters"], info["restarts"]) == ("not_converged", maxit, restarts)
        if maxit < 3:
            first = torch.tensor([1.0, -0.3, -0.3], dtype=torch.float64, device=DEV)
            assert torch.allclose(x.real[: 3 * m].reshape(m, 3), first.expand(m, 3), atol=1e-14, rtol=0)
    A.close()


def test_met_within_the_tolerance():
    """(r^, r) vanishes at an x that already meets the tolerance: ok, no restart."""
    rp, ci, v, bh = blocks(4)
    A = helm.CsrMatrix.from_host(rp, ci, v, device=DEV)
    b = torch.as_tensor(bh, device=DEV)
    x, info = _solve_all(A, b, tol=0.5, maxit=100)  # ||r|| / ||b|| = sqrt(0.2) after one iteration
    assert info["status"] == "ok" and info["iters"] == 1 and info["restarts"] == 0
    A.close()
