"""The oracle's BiCGStab starts again from x when (r^, r) vanishes after an
iteration, as the library does."""
import os
import sys

import numpy as np

import oracle

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
from vanishing_rho import blocks  # noqa: E402


def test_oracle_restarts_when_rho_vanishes():
    rp, ci, v, b = blocks(4, pad=5)
    xs = oracle.dense_solve(rp, ci, v, b)
    x, info = oracle.bicgstab(rp, ci, v, b, tol=1e-12, maxit=100)
    assert info["status"] == "ok" and 3 <= info["iters"] <= 8
    assert np.linalg.norm(x - xs) <= 1e-11 * np.linalg.norm(xs)
    # the iteration that met the zero counts; x stands at the cap
    for maxit in (1, 2):
        x, info = oracle.bicgstab(rp, ci, v, b, tol=1e-12, maxit=maxit)
        assert info["status"] == "not_converged" and info["iters"] == maxit
        assert np.allclose(x[:12].reshape(4, 3), [[1.0, -0.3, -0.3]] * 4, atol=1e-14)


def test_oracle_still_breaks_down_in_a_first_iteration():
    rp, ci, v, b = blocks(2)
    x, info = oracle.bicgstab(rp, ci, np.zeros_like(v), b, tol=1e-12, maxit=100)
    assert info["status"] == "breakdown" and info["iters"] == 1
