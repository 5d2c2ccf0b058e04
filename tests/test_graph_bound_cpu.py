"""The bound on a handle's cached graphs, with the host compiler alone; and that every
place that adds one asks for room first."""
import glob
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2112_11880_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"


def test_no_more_graphs_than_the_bound(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = tmp_path / "graph_bound_check"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", CUDA_INC, "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        os.path.join(HERE, "graph_bound_check.cpp"), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=30)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr


def test_every_method_asks_for_room():
    added = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        for m in re.finditer(r"A->graphs\[\w+\] = ", text):
            before = text[:m.start()].rstrip().splitlines()[-2:]
            assert any("bound_graphs" in line or "A->graphs[" in line for line in before), (path, before)
            added += 1
    assert added == 5
