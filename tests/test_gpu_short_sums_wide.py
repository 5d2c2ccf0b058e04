"""Dot products and norms of 8,193 to 32,768 elements (one cluster of sixteen blocks,
eight up to 8,192): against FP64 sums on the host, within the roundings of a tree of
at most 32 over products of two (complex128) or over FP32 products (complex64), and the
same bits eager, in a captured graph and without scratch."""
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
@pytest.mark.parametrize("n", [8_191, 8_192, 8_193, 16_384, 16_385, 20_479, 20_481, 24_000, 32_767, 32_768])
def test_wide_dot_and_norm(n, dtype):
    x = torch.as_tensor(g.complex_vector(n, 17), device=DEV).to(dtype)
    y = torch.as_tensor(g.complex_vector(n, 18), device=DEV).to(dtype)
    out = torch.zeros(4, dtype=torch.complex128, device=DEV)
    nrm = torch.zeros(2, dtype=torch.float64, device=DEV)

    def run(k):
        helm.helm_dot(x, y, out[2 * k:2 * k + 1], True)
        helm.helm_dot_noalloc(x, y, out[2 * k + 1:2 * k + 2], True)
        helm.helm_nrm2(x, nrm[k:k + 1])

    run(0)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        run(1)
    graph.replay()
    torch.cuda.synchronize()
    d = out.cpu().numpy()
    assert d[0] == d[1] == d[2] == d[3] and nrm[0].item() == nrm[1].item()
    xe, ye = x.cpu().numpy().astype(np.complex128), y.cpu().numpy().astype(np.complex128)
    tol = 40 * 2.0 ** -53 if dtype == torch.complex128 else 4 * 2.0 ** -24
    assert abs(d[0] - np.vdot(xe, ye)) <= tol * float(np.sum(np.abs(xe) * np.abs(ye)))
    assert abs(nrm[0].item() - np.linalg.norm(xe)) <= tol * float(np.linalg.norm(xe))
