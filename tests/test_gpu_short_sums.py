"""Dot products and norms of vectors up to 32,768 elements (one cluster of
eight blocks) and one past it: against FP64 sums on the host.

Bounds: a complex128 sum is a tree of at most 40 roundings above products of
two each, so within 50 eps of sum |x_i| |y_i|; complex64 forms each product in
FP32 (4 roundings) and adds in FP64."""
import numpy as np
import pytest

import helmgen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("n", [0, 1, 33, 256, 257, 2047, 2049, 8193, 9261, 32_767, 32_768, 32_769,
                               65_537])
def test_short_dot_and_norm(n, dtype):
    x = torch.as_tensor(g.complex_vector(n + 1, 7), device=DEV).to(dtype)[1:]  # aligned to an element only
    y = torch.as_tensor(g.complex_vector(n + 1, 8), device=DEV).to(dtype)[1:]
    out = torch.full((3,), complex("nan+nanj"), dtype=torch.complex128, device=DEV)
    nrm = torch.full((1,), float("nan"), dtype=torch.float64, device=DEV)
    helm.helm_dot(x, y, out[0:1], True)
    helm.helm_dot(x, y, out[1:2], False)
    helm.helm_dot_noalloc(x, y, out[2:3], True)
    helm.helm_nrm2(x, nrm)
    d = out.cpu().numpy()
    xe, ye = x.cpu().numpy().astype(np.complex128), y.cpu().numpy().astype(np.complex128)
    tol = 50 * 2.0 ** -53 if dtype == torch.complex128 else 4 * 2.0 ** -24
    bound = tol * float(np.sum(np.abs(xe) * np.abs(ye)))
    assert abs(d[0] - np.vdot(xe, ye)) <= bound
    assert abs(d[1] - np.dot(xe, ye)) <= bound
    assert d[2] == d[0]
    assert abs(float(nrm[0]) - np.linalg.norm(xe)) <= tol * float(np.linalg.norm(xe))


def test_short_sums_carry_nan_and_infinity():
    x = torch.as_tensor(g.complex_vector(1000, 7), device=DEV)
    x[700] = complex("inf")
    nrm = torch.zeros(1, dtype=torch.float64, device=DEV)
    helm.helm_nrm2(x, nrm)
    assert float(nrm[0]) == float("inf")
    x[3] = complex("nan")
    helm.helm_nrm2(x, nrm)
    assert np.isnan(float(nrm[0]))
