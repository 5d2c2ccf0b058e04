"""How a sweep deals its frequencies to threads: counts around the multiples of 32
(and 96, which does not divide a block), systems down to one row, frequencies
that stop at very different iterations, so that the running ones are dealt out
anew many times.  Every frequency has to meet the tolerance by the oracle's
product, and a repeat has to give the same bits."""
import numpy as np
import pytest

import helmgen as g
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402
from test_gpu_sweep import DEV, _method, _relres  # noqa: E402


@pytest.mark.parametrize("dims", [(3, 2, 2), (9, 7, 6)])
@pytest.mark.parametrize("freqs", [1, 2, 3, 7, 16, 31, 32, 33, 45, 63, 64, 97, 127, 128])
@pytest.mark.parametrize("method", ["bicgstab", "tfqmr", "bicgstabl2"])
def test_every_count_of_frequencies(dims, freqs, method):
    if method != "bicgstab" and freqs not in (3, 31, 45, 128):
        pytest.skip("fewer counts")
    cfg = g.tiny_config(*dims, h=0.1, seed=3)
    p = g.assemble(cfg)
    b = g.source(p) + 0.1 * g.complex_vector(p.n, 4) * (~p.dirichlet)
    w = [g.omega(f) for f in np.linspace(80.0, 900.0, freqs)]
    S = helm.Sweep(p.rowptr, p.colind, p.K, p.Mc, p.Bc, device=DEV)
    bt = torch.as_tensor(b, device=DEV)
    X, infos = S.solve(w, bt, tol=1e-9, maxit=4000, **_method(method))
    X2, infos2 = S.solve(w, bt, tol=1e-9, maxit=4000, **_method(method))
    Xh = X.cpu().numpy()
    assert np.array_equal(Xh, X2.cpu().numpy()) and infos == infos2
    for j in range(freqs):
        assert infos[j]["status"] == "ok", (j, infos[j])
        vals = oracle.helmholtz_values(p.K, p.Mc, p.Bc, w[j])
        assert _relres(p, vals, b, Xh[:, j]) <= 1e-9 * (1 + 1e-6)
    # the stand-alone product dealt the same way: 28 roundings a row at most
    Y = S.matvec(w, X).cpu().numpy()
    for j in range(0, freqs, 5):
        vals = oracle.helmholtz_values(p.K, p.Mc, p.Bc, w[j])
        ab = oracle.spmv(p.rowptr, p.colind, np.abs(vals), np.abs(Xh[:, j])).real
        assert np.all(np.abs(Y[:, j] - oracle.spmv(p.rowptr, p.colind, vals, Xh[:, j])) <= 1e-13 * ab + 1e-300)
    S.close()


@pytest.mark.parametrize("n", [1, 2, 3])
@pytest.mark.parametrize("freqs", [1, 31, 63, 127])
def test_fewer_rows_than_slots(n, freqs):
    """Diagonal systems: x = b / (K - w^2 M + i w B), eight roundings and the
    solver's tolerance."""
    rng = np.random.default_rng(n)
    K, M, B = 5 + rng.uniform(0, 1, n), rng.uniform(0.1, 0.2, n), rng.uniform(0.5, 1, n)
    w = np.linspace(0.5, 2.0, freqs)
    b = g.complex_vector(n, 5)
    S = helm.Sweep(np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), K, M, B, device=DEV)
    X, infos = S.solve(list(w), torch.as_tensor(b, device=DEV), tol=1e-12, maxit=200)
    d = K[:, None] - w[None, :] ** 2 * M[:, None] + 1j * w[None, :] * B[:, None]
    err = np.linalg.norm(X.cpu().numpy() * d - b[:, None], axis=0) / np.linalg.norm(b)
    assert all(i["status"] == "ok" for i in infos)
    assert err.max() <= 1e-12 + 8 * 2.0 ** -53
    S.close()
