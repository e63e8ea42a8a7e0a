"""Sweeps whose form is chosen by the jump rate, against the oracle and each other at the
rates where the choice changes."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2505_04328_gb300 import JdProblem, build, launch_count

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


def _launches(f):
    n = launch_count()
    out = f()
    return out, launch_count() - n


# a pre-drawn cost evaluation launches the draws and the combination of the paths' costs beside
# the sweep
PRE_EXTRA = 2


@pytest.mark.parametrize("d", [1, 2])
def test_form_follows_the_rate_of_an_update(d):
    """The path limit of the FP32 pre-drawn cost sweep rises with the jump rate: a problem
    between the limits moves between the forms as its rate is updated, with a fresh problem's
    bits."""
    M, Nt = 6500, 40
    p = (workloads.lq_scalar if d == 1 else workloads.double_well)(M=M, Nt=Nt)
    u = workloads.random_control(p, seed=3, scale=0.6)
    low, high = p.replace(lam=0.001 * Nt / p.T), p.replace(lam=0.1 * Nt / p.T)
    with JdProblem(low) as jp:
        J0, n0 = _launches(lambda: jp.cost(u))
        jp.update(high)
        J1, n1 = _launches(lambda: jp.cost(u))
        g1 = jp.gradient(u)[1]
        jp.update(low)
        J2, n2 = _launches(lambda: jp.cost(u))
    assert n1 == n0 + PRE_EXTRA and n2 == n0 and J2 == J0
    with JdProblem(high) as jp:
        J3, n3 = _launches(lambda: jp.cost(u))
        assert n3 == n1 and J3 == J1 and np.array_equal(jp.gradient(u)[1], g1)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("law", [workloads.JUMP_NORMAL, workloads.JUMP_UNIFORM, workloads.JUMP_KS])
@pytest.mark.parametrize("Nt,lamdt", [(33, 0.0), (61, 0.003), (40, 0.02), (35, 0.3), (17, 0.7)])
def test_pre_drawn_sweeps_equal_the_others(law, prec, Nt, lamdt):
    """The last shard of a problem is small enough for the pre-drawn sweeps at every rate, the
    whole is not: which form ran shows in the launches, and the units' sums are equal."""
    p = workloads.double_well(M=16384 + 3001, Nt=Nt).replace(lam=lamdt * Nt / 2.0, seed=11, jump_law=law, jump_gain=0.5)
    u = workloads.random_control(p, seed=3, scale=0.6)
    with JdProblem(p, prec=prec, mode="stored") as jp:
        whole, n = _launches(lambda: jp.cost_units(u))
        grads = jp.gradient_units(u)
    with JdProblem(p.replace(M=3001, m_offset=16384), prec=prec, mode="stored") as jp:
        part, npart = _launches(lambda: jp.cost_units(u))
        assert np.array_equal(grads[1:], jp.gradient_units(u))
    assert npart == n + PRE_EXTRA and np.array_equal(whole[1:], part)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("particles,lamdt", [(0, 0.24), (0, 0.27), (200, 0.12), (200, 0.14), (200, 1.5)])
def test_feedback_across_the_straight_code_limit(particles, lamdt, prec):
    """Either side of the rate that decides on a one-jump step's draws, against the oracle.
    FP32: 20 steps of 2.5 sub-steps with 4 roundings each of 2^-24 are 1.2e-5 of a path's value
    at worst, ten times that for the adjoint's weights."""
    Nt = 20
    M = oracle.ring_lanes(particles) * 2 if particles else 600
    p, fb = workloads.feedback_coupled(M=M, Nt=Nt, particles=particles) if particles else \
        workloads.feedback_centering(M=M, Nt=Nt)
    p = p.replace(lam=lamdt * Nt / p.T)
    mu = workloads.random_mu(p, fb, seed=8, scale=0.5)
    Jo, go = (oracle.fb_coupled_gradient if particles else oracle.fb_gradient)(p, fb, mu)[:2]
    with JdProblem(p, prec=prec) as jp:
        J, g = jp.fb_gradient(fb, mu)
        assert jp.fb_cost(fb, mu) == J
    tol_j, tol_g = (1e-13, 1e-12) if prec == "fp64" else (1.2e-5, 1.2e-4)
    assert abs(J - Jo) <= tol_j * abs(Jo)
    assert np.linalg.norm(g - go) <= tol_g * np.linalg.norm(go)


@pytest.mark.parametrize("nx", [4, 10, 16])
@pytest.mark.parametrize("particles", [0, 20, 200])
def test_feedback_fp64_sizes_and_rings(nx, particles):
    """Every FP64 forward's own residency: costs and gradients against the oracle."""
    Nt = 12
    M = 512 if particles else 700
    p, fb = workloads.feedback_coupled(M=M, Nt=Nt, particles=particles) if particles else \
        workloads.feedback_centering(M=M, Nt=Nt)
    p, fb = p.replace(lam=3.0), fb.replace(nx=nx, nv=nx)
    mu = workloads.random_mu(p, fb, seed=8, scale=0.5)
    Jo, go = (oracle.fb_coupled_gradient if particles else oracle.fb_gradient)(p, fb, mu)[:2]
    with JdProblem(p, prec="fp64") as jp:
        J, g = jp.fb_gradient(fb, mu)
        assert jp.fb_cost(fb, mu) == J
    assert abs(J - Jo) <= 1e-13 * abs(Jo) and np.linalg.norm(g - go) <= 1e-12 * np.linalg.norm(go)


@pytest.mark.parametrize("mode,plan", [("auto", "stored"), ("stored", "stored"), ("recompute", "recompute")])
def test_pre_pass_buffers_give_way_to_a_small_budget(mode, plan):
    """A problem that only a higher jump rate would pre-draw runs in the memory that it needs
    without the buffers, in the plan that it has without them."""
    M, Nt = 8000, 400
    p = workloads.lq_scalar(M=M, Nt=Nt)
    low, high = p.replace(lam=0.002 * Nt), p.replace(lam=0.1 * Nt)
    u = workloads.random_control(p, seed=3, scale=0.6)
    buffers = Nt * M * 4 + (Nt * 4 * M + 4 * M) * 4 + 8
    with JdProblem(low, mode=mode) as jp:
        J, g, _ = jp.gradient(u)
        full = jp.info()["device_bytes"]
    with JdProblem(low, mode=mode, mem_budget=full - buffers) as jp:
        assert jp.info()["device_bytes"] < full - buffers
        J1, g1, _ = jp.gradient(u)
        assert jp.info() == dict(device_bytes=full - buffers, mode=plan)
        jp.update(high)
        J2, n2 = _launches(lambda: jp.cost(u))
    with JdProblem(high, mode=mode) as jp:
        J3, n3 = _launches(lambda: jp.cost(u))
    assert J1 == J and np.array_equal(g1, g) and J2 == J3 and n3 == n2 + PRE_EXTRA
