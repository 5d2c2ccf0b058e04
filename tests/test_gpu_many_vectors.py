"""Graph solves for more pairs of vectors than a handle keeps graphs for, the methods
interleaved: every solve gives the bits of the first one."""
import pytest

import helmgen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")


def test_more_vectors_than_graphs():
    p = g.assemble(g.tiny_config(6, 5, 4, h=0.1, F=350.0))
    A = helm.CsrMatrix.from_host(p.rowptr, p.colind, g.helmholtz_values(p, 350.0), device=DEV)
    b = torch.as_tensor(g.source(p), device=DEV)
    kinds = [dict(), dict(method=helm.HELM_TFQMR), dict(method=helm.HELM_BICGSTABL),
             dict(precision=helm.HELM_PREC_MIXED)]
    ref, keep = {}, []
    for k in range(60):
        kw = kinds[k % 4]
        bk, x = b.clone(), torch.empty_like(b)
        keep += [bk, x]  # every solve on buffers of its own
        o = helm.default_opts(tol=1e-9, maxit=5000, launch=helm.HELM_LAUNCH_GRAPH, **kw)
        info = helm.helm_bicgstab_solve(A.handle, bk, x, o)
        assert info["status"] == "ok"
        i0, x0 = ref.setdefault(k % 4, (info, x))
        assert info == i0 and torch.equal(torch.view_as_real(x), torch.view_as_real(x0))
    A.close()
