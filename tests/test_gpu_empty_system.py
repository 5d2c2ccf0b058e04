"""Solves of a system without rows through the C ABI (a C caller's pointers are
not null): every method and loop form returns ok with nothing to do, and writes
nothing."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("use_x0", [0, 1])
@pytest.mark.parametrize("method,launch,precision,precond", [
    (m, l, helm.HELM_PREC_FP64, p)
    for m in (helm.HELM_BICGSTAB, helm.HELM_TFQMR, helm.HELM_BICGSTABL)
    for l in (helm.HELM_LAUNCH_AUTO, helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_HOST)
    for p in (helm.HELM_PRECOND_NONE, helm.HELM_PRECOND_JACOBI)
] + [(helm.HELM_BICGSTAB, helm.HELM_LAUNCH_PERSISTENT, helm.HELM_PREC_FP64, helm.HELM_PRECOND_NONE),
     (helm.HELM_BICGSTAB, helm.HELM_LAUNCH_AUTO, helm.HELM_PREC_MIXED, helm.HELM_PRECOND_NONE),
     (helm.HELM_BICGSTAB, helm.HELM_LAUNCH_GRAPH, helm.HELM_PREC_MIXED, helm.HELM_PRECOND_NONE)])
def test_empty_system(method, launch, precision, precond, use_x0):
    lib = helm.load_library()
    rowptr = torch.zeros(4, dtype=torch.int32, device=DEV)
    # a solve of another handle first: its tables are what the shared memory holds
    n = 4000
    rp = torch.arange(n + 1, dtype=torch.int32, device=DEV)
    ci = torch.arange(n, dtype=torch.int32, device=DEV)
    D = helm.CsrMatrix(rp, ci, torch.full((n,), 2.0 + 1.0j, dtype=torch.complex128, device=DEV))
    _, info = helm.solve(D, torch.ones(n, dtype=torch.complex128, device=DEV), method=method)
    assert info["status"] == "ok"

    h = helm.helm_csr_create(0, 0, rowptr.data_ptr(), None, None, helm.HELM_C128)
    b = torch.full((8,), 3.0 + 4.0j, dtype=torch.complex128, device=DEV)
    x = torch.full((8,), 5.0 + 6.0j, dtype=torch.complex128, device=DEV)
    o = helm.default_opts(method=method, launch=launch, precision=precision, precond=precond, use_x0=use_x0)
    i = helm.helm_info()
    st = lib.helm_bicgstab_solve(h, b.data_ptr(), x.data_ptr(), ctypes.byref(o), ctypes.byref(i),
                                 torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert st == helm.HELM_OK
    d = i.as_dict()
    assert (d["status"], d["iters"], d["restarts"], d["relres_true"], d["relres_recur"]) == ("ok", 0, 0, 0.0, 0.0)
    assert torch.all(b == 3.0 + 4.0j) and torch.all(x == 5.0 + 6.0j)
    helm.helm_csr_destroy(h)
    D.close()
