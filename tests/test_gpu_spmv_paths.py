"""Stand-alone products at the sizes where their path changes: complex64 matrices
on diagonals from 200,000 rows on."""
import numpy as np
import pytest

import helmgen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")
AXPBY = [(1.0, 0.0), (0.5 - 2.0j, 0.0), (1.5 + 0.5j, -0.25 + 1.0j)]


@pytest.mark.parametrize("n", [200_000, 200_001, 200_003, 262_147])
@pytest.mark.parametrize("offsets", [[0], [-1, 0, 1], [-300, -299, -1, 0, 1, 2, 300], [-7, -6, -5, -4, 0, 1, 1000]])
def test_diagonals_two_rows_a_thread(n, offsets):
    """The bits of the sliced copy, for every run of neighbouring diagonals, odd
    sizes, vectors aligned to an element only, and rows with imaginary parts."""
    rng = np.random.default_rng(7)
    cols = np.arange(n)[:, None] + np.asarray(offsets)[None, :]
    ok = (cols >= 0) & (cols < n)
    v = rng.uniform(-1, 1, cols.shape) + 1j * rng.uniform(-1, 1, cols.shape) * (np.arange(n) % 1000 < 40)[:, None]
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = ok.sum(1).cumsum()
    args = (rp, cols[ok].astype(np.int32), v[ok].astype(np.complex64))
    A = helm.CsrMatrix.from_host(*args, device=DEV)
    B = helm.CsrMatrix.from_host(*args, device=DEV, sliced_only=True)
    assert A.diagonals() == len(offsets) and B.diagonals() == 0
    x = torch.as_tensor(g.complex_vector(n + 1, 8), device=DEV).to(torch.complex64)[1:]
    y0 = torch.as_tensor(g.complex_vector(n + 1, 9), device=DEV).to(torch.complex64)[1:]
    for al, be in AXPBY:
        ya, yb = torch.empty(n + 1, dtype=torch.complex64, device=DEV)[1:], y0.clone()
        ya.copy_(y0)
        A.matvec(x, ya, alpha=al, beta=be)
        B.matvec(x, yb, alpha=al, beta=be)
        assert torch.equal(torch.view_as_real(ya), torch.view_as_real(yb))
    A.close()
    B.close()
