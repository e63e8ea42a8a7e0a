"""Sweeps whose form is chosen by the jump rate, against the oracle and each other at the
rates where the choice changes."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2505_04328_gb300 import JdProblem, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("lamdt", [0.001, 0.0039, 0.0041, 0.2, 0.49, 0.51, 0.9])
def test_keilson_storer_sweeps_across_the_rates(prec, lamdt):
    """The short one-jump path, the general routine and the chunks take the same draws and the
    same operations: the plans agree bit for bit with parameter gradients, every 97th path's
    cost and the last state with the oracle."""
    Nt, M = 37, 12001
    p = workloads.ks_oscillator(M=M, Nt=Nt)
    p = p.replace(lam=lamdt * Nt / p.T, seed=21, dA=np.array([[0.2, -0.4], [0.7, 0.1]]))
    u = workloads.random_control(p, seed=3, scale=0.6)
    out = []
    for mode in ("stored", "recompute"):
        with JdProblem(p, prec=prec, mode=mode) as jp:
            J, g, th = jp.gradient(u, theta=True)
            X, _, c = jp.sample_paths(u, 0, 1000, lam=False)
        out.append((J, g, th, X, c))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    tol = 1e-5 if prec == "fp32" else 1e-12
    X, c = out[0][3], out[0][4]
    for m in range(0, 1000, 97):
        r = oracle.path(p, u, m)
        assert abs(c[m] - r["cost"]) <= tol * abs(r["cost"])
        assert np.max(np.abs(X[m, -1] - r["X"][-1])) <= tol * max(1.0, np.max(np.abs(r["X"][-1])))
