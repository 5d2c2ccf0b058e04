"""Stand-alone products at the sizes where their path changes: matrices whose few
slices are shared out to several warps, complex64 matrices on
diagonals from 200,000 rows on."""
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
AXPBY = [(1.0, 0.0), (0.5 - 2.0j, 0.0), (1.5 + 0.5j, -0.25 + 1.0j)]


def _ragged(n, most, complex_part, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, most + 1, n)
    lens[rng.random(n) < 0.1] = 0
    lens = np.minimum(lens, n)
    lens[0] = min(most, n)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = lens.cumsum()
    start = rng.integers(0, np.maximum(n - lens + 1, 1))
    ci = np.concatenate([np.arange(s, s + k) for s, k in zip(start, lens)] or [np.zeros(0)]).astype(np.int32)
    v = rng.uniform(-1, 1, ci.size) + 1j * rng.uniform(-1, 1, ci.size) * (rng.random(ci.size) < complex_part)
    return rp, ci, v


@pytest.mark.parametrize("slices,extra", [(1, -31), (1, 0), (SMS, 0), (SMS, 1), (5 * SMS, -7), (5 * SMS, 1)])
@pytest.mark.parametrize("most,complex_part", [(1, 1.0), (3, 0.0), (27, 0.05), (61, 1.0)])
@pytest.mark.parametrize("dtype", [np.complex128, np.complex64])
def test_slices_shared_out(slices, extra, most, complex_part, dtype):
    """A row of m entries: 2 m products and sums of parts, m + 12 roundings a
    component at most, and six of alpha and beta."""
    n = 32 * slices + extra
    rp, ci, v = _ragged(n, most, complex_part, 3)
    v, x, y0 = v.astype(dtype), g.complex_vector(n, 4).astype(dtype), g.complex_vector(n, 5).astype(dtype)
    eps = 2.0 ** -53 if dtype == np.complex128 else 2.0 ** -24
    A = helm.CsrMatrix.from_host(rp, ci, v, device=DEV)
    xd = torch.as_tensor(x, device=DEV)
    rows = np.repeat(np.arange(n), np.diff(rp))

    def rowsum(t):
        return np.bincount(rows, weights=t, minlength=n)
    t = v.astype(np.complex128) * x[ci]
    ax = rowsum(t.real) + 1j * rowsum(t.imag)
    ab = rowsum(np.abs(v).astype(np.float64) * np.abs(x[ci]))
    for al, be in AXPBY:
        y = torch.as_tensor(y0, device=DEV)
        A.matvec(xd, y, alpha=al, beta=be)
        bound = 4 * (most + 18) * eps * (abs(al) * ab + abs(be) * np.abs(y0).astype(np.float64))
        assert np.all(np.abs(y.cpu().numpy() - (al * ax + be * y0)) <= bound)
    A.close()


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
