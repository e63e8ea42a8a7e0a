"""Steps with several jumps of the d = 32 forward (a warp per step), against the oracle: two or
more jumps, and slot layouts of fewer than 16 normal pairs (d < 31)."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2505_04328_gb300 import JdProblem, build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("law", [workloads.JUMP_NORMAL, workloads.JUMP_UNIFORM])
@pytest.mark.parametrize("d", [9, 20, 31, 32])
@pytest.mark.parametrize("lam", [3.0, 40.0, 150.0])
def test_paths_with_many_jumps(d, lam, law):
    """The pathwise FP32 bar of the other dimensions (1e-5 of the path's scale); the jump log
    of the gradient covers the same steps, so its gradient stays at the reduced bar."""
    build()
    p = workloads.linear_family(d, M=140, Nt=30, lam=lam, seed=9).replace(jump_law=law)
    u = workloads.random_control(p, seed=4, scale=0.5)
    with JdProblem(p) as jp:
        X, _, c = jp.sample_paths(u, 0, p.M, lam=False)
        J, g, _ = jp.gradient(u)
    jumps = 0
    for m in range(0, p.M, 23):
        r = oracle.path(p, u, m)
        jumps += int(r["njumps"].sum())
        rms = np.sqrt(np.mean(r["X"] ** 2))
        assert np.max(np.abs(X[m] - r["X"]) / np.maximum(np.abs(r["X"]), rms)) <= 1e-5
        assert abs(c[m] - r["cost"]) <= 1e-5 * abs(r["cost"])
    assert jumps > 0
    Jo, go, _ = oracle.gradient(p, u)
    assert abs(J - Jo) <= 1e-5 * abs(Jo)
    assert np.linalg.norm(g - go) <= 1e-5 * np.linalg.norm(go)
