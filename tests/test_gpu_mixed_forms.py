"""Mixed precision: the persistent complex64 inner solve (the default up to 50
slices per SM) against the graph and the host-driven loop of the same kernels.
Every inner iterate, and so every refinement step and x, has to agree bit for bit:
at one slice, with a partial last slice, in several rounds of the grid and on both
sides of 50 slices per SM; on a diagonal copy and on the sliced copy; with a warm
start; and on a Helmholtz system that takes thousands of inner iterations."""
import numpy as np
import pytest

import helmgen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")
SMS = torch.cuda.get_device_properties(0).multi_processor_count


def _banded(n, seed):
    """Up to nine diagonals, diagonally dominant, every 53rd row complex."""
    rng = np.random.default_rng(seed)
    offs = np.array([o for o in (-400, -21, -20, -1, 0, 1, 20, 21, 400) if abs(o) < n])
    cols = np.arange(n)[:, None] + offs[None, :]
    ok = (cols >= 0) & (cols < n)
    v = rng.uniform(-1, 1, cols.shape) + 1j * rng.uniform(-1, 1, cols.shape) * (np.arange(n) % 53 == 0)[:, None]
    v[:, offs == 0] = (8.0 * (1 + 0.3 * rng.uniform(-1, 1, n)))[:, None]
    rowptr = np.zeros(n + 1, np.int32)
    rowptr[1:] = ok.sum(1).cumsum()
    return rowptr, cols[ok].astype(np.int32), v[ok]


def _forms(A, b, x0=None, **kw):
    out = []
    for launch in (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_HOST, helm.HELM_LAUNCH_AUTO):
        x = torch.empty_like(b) if x0 is None else x0.clone()
        o = helm.default_opts(precision=helm.HELM_PREC_MIXED, launch=launch, use_x0=0 if x0 is None else 1, **kw)
        out.append((x, helm.helm_bicgstab_solve(A.handle, b, x, o)))
    (xg, ig) = out[0]
    for x, i in out[1:]:
        assert i == ig
        assert torch.equal(torch.view_as_real(x), torch.view_as_real(xg))
    return ig


@pytest.mark.parametrize("sliced_only", [False, True])
@pytest.mark.parametrize("slices,extra", [
    (1, -31), (1, -5), (3, 0), (SMS, 1), (4 * SMS, 33), (24 * SMS, 0), (24 * SMS, 1), (49 * SMS, -7), (50 * SMS, 0),
    (50 * SMS, 1),
])
def test_inner_solve_forms(slices, extra, sliced_only):
    n = 32 * slices + extra
    A = helm.CsrMatrix.from_host(*_banded(n, 9), device=DEV, sliced_only=sliced_only)
    b = torch.as_tensor(g.complex_vector(n, 10), device=DEV)
    x0 = torch.as_tensor(0.1 * g.complex_vector(n, 11), device=DEV)
    for kw in (dict(), dict(x0=x0), dict(inner_tol=0.3)):
        info = _forms(A, b, tol=1e-11, **kw)
        assert info["status"] == "ok"
        assert info["restarts"] >= (1 if n > 1 else 0)
    _forms(A, b, tol=1e-11, maxit=3)  # the cap inside an inner solve
    A.close()


@pytest.mark.parametrize("sliced_only", [False, True])
def test_helmholtz_forms(sliced_only):
    cfg = g.CONFIGS["box20_10ppw"]
    p = g.assemble(cfg)
    A = helm.CsrMatrix.from_host(p.rowptr, p.colind, g.helmholtz_values(p, cfg.F), device=DEV, sliced_only=sliced_only)
    info = _forms(A, torch.as_tensor(g.source(p), device=DEV), tol=1e-10, maxit=100000)
    assert info["status"] == "ok" and info["restarts"] >= 3
    A.close()
