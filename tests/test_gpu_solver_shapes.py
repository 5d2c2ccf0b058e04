"""The BiCGStab loop on each shape of its grid: small meshes (a row summed in
three parts by three warps), mid and large ones, at the sizes where the rule
changes, with partial last slices, rows longer than a thread holds and complex
rows.  The persistent and the graph form have to agree bit for bit, and the
solution has to meet the tolerance by the oracle's product."""
import numpy as np
import pytest

import helmgen as g
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")


def _banded(n, offsets, complex_rows, seed):
    """CSR with the given diagonals, diagonally dominant; imaginary parts on the
    entries of `complex_rows` only."""
    rng = np.random.default_rng(seed)
    offsets = np.asarray(sorted(offsets))
    cols = np.arange(n)[:, None] + offsets[None, :]
    ok = (cols >= 0) & (cols < n)
    v = rng.uniform(-1, 1, cols.shape) + 1j * rng.uniform(-1, 1, cols.shape) * complex_rows(np.arange(n))[:, None]
    diag = offsets == 0
    v[:, diag] = (1.5 * len(offsets) * (1 + 0.3 * rng.uniform(-1, 1, n)))[:, None]
    rowptr = np.zeros(n + 1, np.int32)
    rowptr[1:] = ok.sum(1).cumsum()
    return rowptr, cols[ok].astype(np.int32), v[ok]


def _check(rp, ci, v, seed, tol=1e-10, **kw):
    n = rp.size - 1
    A = helm.CsrMatrix.from_host(rp, ci, v, device=DEV)
    b = torch.as_tensor(g.complex_vector(n, seed), device=DEV)
    x0 = torch.as_tensor(0.1 * g.complex_vector(n, seed + 1), device=DEV)
    out = []
    for launch in (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_PERSISTENT, helm.HELM_LAUNCH_AUTO):
        x = x0.clone()
        out.append((x, helm.helm_bicgstab_solve(A.handle, b, x, helm.default_opts(tol=tol, launch=launch, use_x0=1, **kw))))
    A.close()
    (xg, ig) = out[0]
    assert ig["status"] == "ok", ig
    for x, i in out[1:]:
        assert i == ig
        assert torch.equal(torch.view_as_real(x), torch.view_as_real(xg))
    bh, xh = b.cpu().numpy(), xg.cpu().numpy()
    r = np.linalg.norm(bh - oracle.spmv(rp, ci, v, xh)) / np.linalg.norm(bh)
    assert r <= tol * (1 + 1e-6)


SMS = torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("slices,extra", [
    (1, -31), (1, 0), (3, -5), (SMS, 0), (SMS, 1), (4 * SMS, 0), (4 * SMS, 1), (4 * SMS, 33), (20 * SMS, -1),
    (20 * SMS, 1), (150 * SMS, 0), (150 * SMS, 1),
])
def test_shape_boundaries(slices, extra):
    """Small up to four slices per SM, large from 150; `extra` rows beyond."""
    n = 32 * slices + extra
    offs = [o for o in (-70, -1, 0, 1, 70) if abs(o) < n]
    _check(*_banded(n, offs, lambda r: (r % 97 == 0) * 1.0, 3), seed=11)


@pytest.mark.parametrize("width,part", [(9, 1), (25, 0), (27, 0), (29, 1), (41, 1)])
def test_rows_held_in_parts(width, part):
    """Rows of the small shape: short ones, three times nine, one more, and too
    many to hold; `part` of the rows complex in every entry."""
    half = width // 2
    offs = list(range(-half, half + 1))
    _check(*_banded(2500, offs, lambda r: (r < 400) * float(part), 5), seed=21)


def test_restart_and_deadline_on_the_small_shape():
    """A tolerance near rounding level (restarts) and an expired deadline, in
    parts."""
    rp, ci, v = _banded(5000, [-40, -1, 0, 1, 40], lambda r: (r % 3 == 0) * 1.0, 7)
    A = helm.CsrMatrix.from_host(rp, ci, v, device=DEV)
    b = torch.as_tensor(g.complex_vector(5000, 8), device=DEV)
    res = []
    for launch in (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_PERSISTENT):
        x, info = helm.solve(A, b, tol=2e-16, maxit=200, launch=launch)
        res.append((x, info))
    assert res[0][1] == res[1][1]
    assert torch.equal(torch.view_as_real(res[0][0]), torch.view_as_real(res[1][0]))
    _, info = helm.solve(A, b, tol=1e-15, deadline_s=1e-9)
    assert info["status"] == "timeout" and info["iters"] == 1
    A.close()
