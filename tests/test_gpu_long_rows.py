"""Solves of matrices with one very long row: a step of the solve then takes as long
as that row's chain of loads, a second and more."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")


def long_row(n, length, seed=3):
    """A diagonal matrix whose middle row also has `length` - 1 small entries."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    r = n // 2
    cols = torch.randperm(n - 1, generator=gen, device=DEV)[: length - 1]
    cols = torch.cat([cols + (cols >= r), torch.tensor([r], device=DEV)]).sort().values
    vals = (torch.rand(length, generator=gen, device=DEV, dtype=torch.float64) - 0.5) / length
    vals[cols == r] = 3.0
    lens = torch.ones(n, dtype=torch.int64, device=DEV)
    lens[r] = length
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = lens.cumsum(0).to(torch.int32)
    d = 2.0 + torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    colind = torch.cat([torch.arange(r, device=DEV), cols, torch.arange(r + 1, n, device=DEV)]).to(torch.int32)
    return rowptr, colind, torch.cat([d[:r], vals, d[r + 1:]]).to(torch.complex128)


def test_a_step_of_more_than_a_second():
    """The waits of the grid barrier last 2 s: a product of some 1.1 s, for which
    every block but one waits, is no time-out."""
    n = 3_400_000
    A = helm.CsrMatrix(*long_row(n, 3_300_000))
    gen = torch.Generator(device=DEV).manual_seed(1)
    b = torch.view_as_complex(torch.rand(n, 2, generator=gen, device=DEV, dtype=torch.float64))
    out = [helm.solve(A, b, tol=1e-30, maxit=1, launch=l) for l in (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_PERSISTENT)]
    assert out[0][1]["status"] == "not_converged" and out[0][1] == out[1][1]
    assert torch.equal(torch.view_as_real(out[0][0]), torch.view_as_real(out[1][0]))
    A.close()


@pytest.mark.parametrize("n,length,precision", [
    (300_000, 128, helm.HELM_PREC_MIXED), (200_000, 129, helm.HELM_PREC_MIXED), (200_000, 3000, helm.HELM_PREC_MIXED),
    (15_000, 15_000, helm.HELM_PREC_FP64), (300_000, 1 << 16, helm.HELM_PREC_FP64),
    (300_000, 1 << 18, helm.HELM_PREC_FP64), (1_000_000, 192, helm.HELM_PREC_FP64),
    (1_000_000, 193, helm.HELM_PREC_FP64),
])
def test_forms_agree_on_both_sides_of_the_rule(n, length, precision):
    A = helm.CsrMatrix(*long_row(n, length))
    gen = torch.Generator(device=DEV).manual_seed(2)
    b = torch.view_as_complex(torch.rand(n, 2, generator=gen, device=DEV, dtype=torch.float64))
    for method in (helm.HELM_BICGSTAB, helm.HELM_TFQMR, helm.HELM_BICGSTABL)[: 1 if precision else 3]:
        out = [helm.solve(A, b, tol=1e-10, maxit=60, method=method, precision=precision, launch=l)
               for l in (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_AUTO)]
        assert out[0][1]["status"] == "ok" and out[0][1] == out[1][1]
        assert torch.equal(torch.view_as_real(out[0][0]), torch.view_as_real(out[1][0]))
    A.close()
