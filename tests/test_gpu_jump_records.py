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


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("model", ["double_well", "lq_scalar", "ks_oscillator", "ks_scalar"])
@pytest.mark.parametrize("Nt,lamdt", [(1, 0.3), (3, 0.01), (16, 0.01), (35, 0.02), (61, 0.05), (37, 0.9), (33, 0.0)])
def test_chunked_sweeps_equal_the_pre_drawn_ones(model, prec, Nt, lamdt):
    """A problem of many paths runs its sweeps in chunks; its last shard is small enough for
    the pre-drawn sweeps, which go step by step.  The path reduction is defined on units, so
    the shard's unit sums are the whole problem's last ones bit for bit."""
    p, u = _problem(model, 16384 + 4711, Nt, lamdt)
    with JdProblem(p, prec=prec, mode="stored") as jp:
        whole, cost = jp.gradient_units(u), jp.cost_units(u)
    with JdProblem(p, prec=prec, mode="recompute") as jp:
        again = jp.gradient_units(u)
    with JdProblem(p.replace(M=4711, m_offset=16384), prec=prec, mode="stored") as jp:
        part, pcost = jp.gradient_units(u), jp.cost_units(u)
    assert np.array_equal(whole[1:], part)
    assert np.array_equal(cost[1:], pcost)
    assert np.array_equal(again, whole)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("lamdt", [0.003, 0.05, 0.6])
def test_chunked_pairs_equal_single_trials(prec, lamdt):
    """Paired trials run both controls in one chunked sweep: the iterates of single trials."""
    p, u = _problem("double_well", 40001, 45, lamdt)
    out = []
    for mode in ("stored", "recompute"):
        for pairs in (True, False):
            with JdProblem(p, prec=prec, mode=mode) as jp:
                v, r, hist = jp.optimize(u0=u, max_iter=3, tol_rel_grad=0.0, pairs=pairs)
            out.append((v, hist, r["evals"]))
    for v, hist, evals in out[1:]:
        assert np.array_equal(v, out[0][0]) and np.array_equal(hist, out[0][1]) and evals == out[0][2]


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("d", [3, 4, 8])
def test_warp_wide_slot_draws_equal_single_lanes(d, prec):
    """For d > 2 the rate per step decides whether a jump step's draws are the warp's or the
    lane's, and the store and replay sweeps have different limits: across them the plans agree
    bit for bit, and the costs of the same paths (sums over the path) with the oracle."""
    import oracle
    for lamdt in (0.0002, 0.002, 0.007, 0.04, 0.09, 0.5):
        Nt, M = 37, 1001
        p = workloads.linear_family(d, M, Nt, lam=lamdt * Nt, seed=12)
        u = workloads.random_control(p, seed=3, scale=0.6)
        out = []
        for mode in ("stored", "recompute"):
            with JdProblem(p, prec=prec, mode=mode) as jp:
                J, g, _ = jp.gradient(u)
                X, _, c = jp.sample_paths(u, 0, M, lam=False)
            out.append((J, g, X, c))
        for a, b in zip(*out):
            assert np.array_equal(a, b)
        tol = 1e-5 if prec == "fp32" else 1e-12
        for m in range(0, M, 97):
            r = oracle.path(p, u, m)
            assert abs(out[0][3][m] - r["cost"]) <= tol * abs(r["cost"])
