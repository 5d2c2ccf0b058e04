"""Default solves (cooperative kernels of every SM) from several threads at once, each
on its own handle and stream, beside other work on the GPU: no wait runs out, and each
gives the bits of the solve alone."""
import threading

import pytest

import helmgen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402

DEV = torch.device("cuda:0")
JOBS = [  # box, options: the small, mid and large shape, a sweep's worth of methods
    ((12, 12, 12), dict(tol=1e-10)),
    ((40, 30, 20), dict(tol=1e-8, method=helm.HELM_TFQMR)),
    ((40, 30, 20), dict(tol=1e-9, precision=helm.HELM_PREC_MIXED)),
    ((100, 90, 85), dict(tol=0.0, maxit=60)),
]


def test_solves_side_by_side():
    systems = []
    for dims, kw in JOBS:
        p = g.assemble(g.tiny_config(*dims, h=0.05, F=200.0, seed=1))
        A = helm.CsrMatrix.from_host(p.rowptr, p.colind, g.helmholtz_values(p, 200.0), device=DEV)
        b = torch.as_tensor(g.source(p), device=DEV)
        systems.append((A, b, dict(maxit=20000) | kw, helm.solve(A, b, **(dict(maxit=20000) | kw))))
    torch.cuda.synchronize()
    stop, errors, done = threading.Event(), [], [0] * len(systems)

    def solver(k):
        A, b, kw, (x0, i0) = systems[k]
        try:
            torch.cuda.set_device(DEV)
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(6):
                    x, info = helm.solve(A, b, stream=s, **kw)
                    assert info == i0, (k, info, i0)
                    assert torch.equal(torch.view_as_real(x), torch.view_as_real(x0)), k
                    done[k] += 1
        except BaseException as e:  # noqa: BLE001 (reported by the test's thread)
            errors.append((k, repr(e)))

    def other_work():
        torch.cuda.set_device(DEV)
        with torch.cuda.stream(torch.cuda.Stream()):
            a = torch.randn(2048, 2048, device=DEV)
            while not stop.is_set():
                for _ in range(20):
                    a = torch.tanh(a @ a * 1e-3)
                torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=solver, args=(k,)) for k in range(len(systems))]
    busy = threading.Thread(target=other_work)
    busy.start()
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    stop.set()
    busy.join(timeout=60)
    assert not errors, errors
    assert done == [6] * len(systems)
    for A, *_ in systems:
        A.close()
