"""A context that refuses the cooperative launch although the occupancy query
allows it (fewer SMs than the device reports): default solves go on with the
graph and give its result, an explicit persistent solve reports the error.  The
refusal is a fake of the launch call, in a second build of the solvers."""
import concurrent.futures as cf
import ctypes
import os
import subprocess

import pytest

import helmgen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2112_11880_gb300 as helm  # noqa: E402
from paper_2112_11880_gb300 import build as hb  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))
DEV = torch.device("cuda:0")
SMS = torch.cuda.get_device_properties(0).multi_processor_count


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = tmp_path_factory.mktemp("refused")
    srcs = [s for s in hb._sources()] + [os.path.join(HERE, "refused_launch.cpp")]

    def compile_one(src):
        obj = str(out / (os.path.basename(src) + ".o"))
        fake = [] if src.endswith(".cpp") else ["-DcudaLaunchCooperativeKernel=helm_refused_launch"]
        r = subprocess.run([hb.nvcc(), *hb.ARCH, *hb.FLAGS, *fake, "-I", hb.INCLUDE, "-c", src, "-o", obj],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return obj

    with cf.ThreadPoolExecutor(max_workers=10) as ex:
        objs = list(ex.map(compile_one, srcs))
    path = str(out / "librefused.so")
    r = subprocess.run([hb.nvcc(), *hb.ARCH, "-shared", "-o", path, *objs], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(path)
    for name, (res, args) in helm.SIGNATURES.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    return lib


@pytest.mark.parametrize("method,precision", [
    (helm.HELM_BICGSTAB, helm.HELM_PREC_FP64), (helm.HELM_TFQMR, helm.HELM_PREC_FP64),
    (helm.HELM_BICGSTABL, helm.HELM_PREC_FP64), (helm.HELM_BICGSTAB, helm.HELM_PREC_MIXED)])
@pytest.mark.parametrize("dims", [(6, 5, 4), (24, 20, 18)])
def test_default_goes_on_with_the_graph(lib, method, precision, dims):
    p = g.assemble(g.tiny_config(*dims, h=0.1, F=250.0, seed=3))
    vals = g.helmholtz_values(p, 250.0)
    rp, ci = (torch.as_tensor(a, dtype=torch.int32, device=DEV) for a in (p.rowptr, p.colind))
    v = torch.as_tensor(vals, device=DEV)
    b = torch.as_tensor(g.source(p), device=DEV)
    s = torch.cuda.current_stream().cuda_stream
    h = ctypes.c_void_p()
    assert lib.helm_csr_create(ctypes.byref(h), p.n, ci.numel(), rp.data_ptr(), ci.data_ptr(), v.data_ptr(),
                               helm.HELM_C128, 0, s) == helm.HELM_OK
    calls = ctypes.c_int.in_dll(lib, "helm_refused_launches")
    out = []
    for launch in (helm.HELM_LAUNCH_GRAPH, helm.HELM_LAUNCH_AUTO):
        before = calls.value
        x = torch.full_like(b, 7.0)
        i = helm.helm_info()
        o = helm.default_opts(tol=1e-9, maxit=20000, method=method, precision=precision, launch=launch)
        st = lib.helm_bicgstab_solve(h, b.data_ptr(), x.data_ptr(), ctypes.byref(o), ctypes.byref(i), s)
        torch.cuda.synchronize()
        assert st == helm.HELM_OK, (launch, st)
        # (mixed precision up to one slice per SM runs as a graph by default)
        tries = launch == helm.HELM_LAUNCH_AUTO and (precision == helm.HELM_PREC_FP64 or p.n > 32 * SMS)
        assert calls.value - before == int(tries)
        out.append((x, i.as_dict()))
    assert out[0][1] == out[1][1]
    assert torch.equal(torch.view_as_real(out[0][0]), torch.view_as_real(out[1][0]))
    if (method, precision) == (helm.HELM_BICGSTAB, helm.HELM_PREC_FP64):
        i, o = helm.helm_info(), helm.default_opts(launch=helm.HELM_LAUNCH_PERSISTENT)
        assert lib.helm_bicgstab_solve(h, b.data_ptr(), x.data_ptr(), ctypes.byref(o), ctypes.byref(i),
                                       s) == helm.HELM_ERR_CUDA
    lib.helm_csr_destroy(h)
