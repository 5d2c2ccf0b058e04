"""Creating a handle times the variants of the stand-alone product only where one of
them will be used (libhelm reports each timing on stderr under HELM_DEBUG)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCRIPT = """
import sys
import torch
import paper_2112_11880_gb300 as helm
n, half, dtype, sliced = int(sys.argv[1]), int(sys.argv[2]), getattr(torch, sys.argv[3]), sys.argv[4] == "1"
offs = torch.arange(-half, half + 1, device="cuda")
cols = torch.arange(n, device="cuda")[:, None] + offs
ok = (cols >= 0) & (cols < n)
rp = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
rp[1:] = ok.sum(1).cumsum(0).to(torch.int32)
A = helm.CsrMatrix(rp, cols[ok].to(torch.int32), torch.ones(int(ok.sum()), dtype=dtype, device="cuda"), sliced_only=sliced)
y = A.matvec(torch.ones(n, dtype=dtype, device="cuda"))
assert torch.equal(y, ok.sum(1).to(dtype))
A.close()
"""


@pytest.mark.parametrize("n,half,dtype,sliced,timed", [
    (20_000, 9, "complex128", 0, False),    # rows in parts
    (20_000, 20, "complex64", 0, False),    # rows in parts (no diagonal copy: 41 diagonals)
    (250_000, 1, "complex64", 0, False),    # two rows a thread on a diagonal copy
    (250_000, 1, "complex64", 1, True),
    (20_000, 9, "complex64", 0, True),      # a diagonal copy, few rows
    (100_000, 2, "complex128", 0, True),
    (10_000, 1, "complex128", 0, False),    # too few entries to time
])
def test_timed_only_where_used(n, half, dtype, sliced, timed):
    r = subprocess.run([sys.executable, "-c", SCRIPT, str(n), str(half), dtype, str(sliced)], cwd=ROOT,
                       env={**os.environ, "HELM_DEBUG": "1"}, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert ("spmv variant" in r.stderr) == timed, r.stderr
