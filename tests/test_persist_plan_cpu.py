"""The plan of a persistent solver kernel (rounds, shared-memory layout),
compiled with the host compiler alone (no GPU)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    exe = tmp_path_factory.mktemp("plan") / "persist_plan_check"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2112_11880_gb300", "csrc"),
                        os.path.join(HERE, "persist_plan_check.cpp"), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(what):
        out = subprocess.run([str(exe), what], capture_output=True, text=True, timeout=30)
        assert out.returncode == 0 and out.stdout.strip().endswith("ok"), out.stdout + out.stderr
    return run


def test_a_system_without_rows_has_a_round(check):
    check("empty")


def test_every_number_of_rounds_has_a_plan(check):
    check("rounds")


def test_blocks_leave_an_sm_its_l1(check):
    check("l1")


def test_a_wait_lasts_two_seconds_of_polls(check):
    check("wait")


def test_long_rows_are_left_to_the_graph(check):
    check("long")
