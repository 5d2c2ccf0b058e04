"""The stand-alone product of a sweep, Y_j = (K - w_j^2 M + i w_j B) X_j, at the counts
of frequencies where the split of a block into groups of 32 changes, on fewer rows than
a block has slots and on several blocks."""
import numpy as np
import pytest

import helmgen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("freqs", [1, 32, 33, 64, 65, 80, 95, 96, 97, 128])
@pytest.mark.parametrize("dims", [(1, 1, 1), (9, 7, 6)])
def test_product(dims, freqs):
    p = g.assemble(g.tiny_config(*dims, h=0.1, seed=4))
    S = helm.Sweep(p.rowptr, p.colind, p.K, p.Mc, p.Bc, device=DEV)
    w = 2 * np.pi * np.linspace(50.0, 400.0, freqs)
    X = g.complex_vector(p.n * freqs, 5).reshape(p.n, freqs)
    Y = S.matvec(w, torch.as_tensor(X, device=DEV)).cpu().numpy()
    rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
    terms = (p.K[:, None] - w**2 * p.Mc[:, None] + 1j * w * p.Bc[:, None]) * X[p.colind]
    size = (np.abs(p.K)[:, None] + w**2 * np.abs(p.Mc)[:, None] + w * np.abs(p.Bc)[:, None]) * np.abs(X[p.colind])
    ref, bound = np.zeros((p.n, freqs), complex), np.zeros((p.n, freqs))
    np.add.at(ref, rows, terms)
    np.add.at(bound, rows, size)
    # entries: three roundings; products and a row's sum: one each per term, on both sides
    m = np.diff(p.rowptr).max()
    assert np.all(np.abs(Y - ref) <= 4 * (m + 6) * 2.0**-53 * bound)
    S.close()
