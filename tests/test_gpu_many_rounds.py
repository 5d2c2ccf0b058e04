"""Solves with so many rounds of slices that a block's table does not fit into its
shared memory: the persistent kernel runs all the same and agrees with the graph
form bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")
SMS = torch.cuda.get_device_properties(0).multi_processor_count
ROUND = 2 * SMS * 512  # rows of one round: two blocks of 16 warps per SM


def _banded(n, seed):
    """Five diagonals, diagonally dominant; every 97th row complex."""
    offs = torch.tensor([-3000, -1, 0, 1, 3000], device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    cols = torch.arange(n, device=DEV)[:, None] + offs
    ok = (cols >= 0) & (cols < n)
    re = torch.rand(n, 5, generator=gen, device=DEV, dtype=torch.float64) - 0.5
    im = torch.rand(n, 5, generator=gen, device=DEV, dtype=torch.float64) - 0.5
    im[torch.arange(n, device=DEV) % 97 != 0] = 0.0
    re[:, 2] += 4.0
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = ok.sum(1).cumsum(0).to(torch.int32)
    return rowptr, cols[ok].to(torch.int32).contiguous(), torch.complex(re, im)[ok].contiguous()


@pytest.mark.parametrize("rounds,extra", [(18, 0), (19, 1), (20, 0), (44, 0), (44, 1), (45, -7), (64, -31), (64, 1)])
@pytest.mark.parametrize("method", [helm.HELM_BICGSTAB, helm.HELM_TFQMR, helm.HELM_BICGSTABL])
def test_rounds_without_a_table(rounds, extra, method):
    n = rounds * ROUND + extra
    A = helm.CsrMatrix(*_banded(n, rounds))
    gen = torch.Generator(device=DEV).manual_seed(1)
    b = torch.view_as_complex(torch.rand(n, 2, generator=gen, device=DEV, dtype=torch.float64) - 0.5)
    xg, ig = helm.solve(A, b, tol=1e-10, maxit=200, method=method, launch=helm.HELM_LAUNCH_GRAPH)
    assert ig["status"] == "ok"
    forms = [helm.HELM_LAUNCH_AUTO]
    if method == helm.HELM_BICGSTAB:
        forms.append(helm.HELM_LAUNCH_PERSISTENT)
    for launch in forms:
        x, info = helm.solve(A, b, tol=1e-10, maxit=200, method=method, launch=launch)
        assert info == ig
        assert torch.equal(torch.view_as_real(x), torch.view_as_real(xg))
    r = b - A.matvec(xg)
    assert torch.linalg.vector_norm(r).item() <= 1.000001e-10 * torch.linalg.vector_norm(b).item()
    A.close()
