"""Jump steps whose draws are kept in records, against the sweeps that take every step by
the general routine: the same FP operations in the same order, so the same bits."""
import numpy as np
import pytest

import workloads
from paper_2505_04328_gb300 import JdProblem, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


MODELS = {
    "double_well": lambda M, Nt: workloads.double_well(M=M, Nt=Nt),
    "lq_scalar": lambda M, Nt: workloads.lq_scalar(M=M, Nt=Nt),
    "ks_oscillator": lambda M, Nt: workloads.ks_oscillator(M=M, Nt=Nt),
    "ks_scalar": lambda M, Nt: workloads.lq_scalar(M=M, Nt=Nt).replace(jump_law=workloads.JUMP_KS, jump_gain=0.5),
    "linear3": lambda M, Nt: workloads.linear_family(3, M, Nt),
}


def _problem(model, M, Nt, lamdt):
    p = MODELS[model](M, Nt)
    p = p.replace(lam=lamdt * Nt / p.T, seed=11, dA=np.linspace(0.5, -1.0, p.d * p.d).reshape(p.d, p.d))
    return p, workloads.random_control(p, seed=3, scale=0.6)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("model", sorted(MODELS))
@pytest.mark.parametrize("Nt,lamdt", [(1, 0.3), (16, 0.05), (17, 0.8), (33, 0.02), (50, 2.5), (31, 0.0)])
def test_parameter_gradients_recompute_equals_stored(model, prec, Nt, lamdt):
    """The stored plan regenerates every jump step; the recompute plan keeps two one-jump
    steps per path and segment (more of them, and steps with several jumps, regenerated)."""
    p, u = _problem(model, 1000, Nt, lamdt)
    out = []
    for mode in ("stored", "recompute"):
        with JdProblem(p, prec=prec, mode=mode) as jp:
            out.append(jp.gradient(u, theta=True))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
