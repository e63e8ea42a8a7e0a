"""The feedback sweep's optional jump log: when it is allocated, how large, and what it leaves
to others.  Results never depend on it."""
import numpy as np
import pytest

import workloads
from paper_2505_04328_gb300 import JdProblem, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def _problem(M=3000, Nt=45, **kw):
    p, fb = workloads.feedback_centering(M=M, Nt=Nt)
    p = p.replace(**kw)
    return p, fb, workloads.random_mu(p, fb, seed=5, scale=0.4)


def _bytes(jp):
    return jp.info()["device_bytes"]


def test_surrogate_adjoint_takes_no_log():
    """Its sweeps neither write nor read the log."""
    p, fb, mu = _problem()
    with JdProblem(p) as jp:
        jp.fb_gradient(fb.replace(adjoint=workloads.FB_SURROGATE, sur_rate=0.05), mu)
        without = _bytes(jp)
        J, g = jp.fb_gradient(fb, mu)
        assert _bytes(jp) > without
    with JdProblem(p, mem_budget=without + 8) as jp:
        J0, g0 = jp.fb_gradient(fb, mu)
        assert _bytes(jp) == without
    assert J == J0 and np.array_equal(g, g0)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_log_follows_an_update(prec):
    """A problem made without jumps gets its log when an update brings them, one made with few a
    larger log when they become many; the results are a fresh problem's."""
    none, fb, mu = _problem(lam=0.0)
    few, many = none.replace(lam=2.0), none.replace(lam=8.0)
    with JdProblem(none, prec=prec) as jp:
        jp.fb_gradient(fb, mu)
        sizes, out = [_bytes(jp)], []
        for p in (few, many, few):
            jp.update(p)
            out.append(jp.fb_gradient(fb, mu))
            sizes.append(_bytes(jp))
    assert sizes[0] < sizes[1] < sizes[2] == sizes[3]
    for p, (J, g) in zip((few, many, few), out):
        with JdProblem(p, prec=prec) as jp:
            J0, g0 = jp.fb_gradient(fb, mu)
            if p is many:
                assert _bytes(jp) == sizes[2]
        assert J == J0 and np.array_equal(g, g0)


def test_a_smaller_log_after_one_that_gave_way():
    """A log that made room for another allocation is tried again in the size of the present
    jumps: with fewer of them it fits beside."""
    p, fb, mu = _problem(M=4096, Nt=40, lam=8.0)
    fewer, u = p.replace(lam=0.5), np.zeros((p.Nt, 1))
    with JdProblem(p, mode="recompute") as jp:
        jp.fb_gradient(fb, mu)
        jp.gradient(u)
        both = _bytes(jp)
    with JdProblem(fewer) as jp:
        J, g = jp.fb_gradient(fb, mu)
    with JdProblem(p, mode="recompute", mem_budget=both - 8) as jp:
        jp.fb_gradient(fb, mu)
        jp.gradient(u)                      # takes the log's memory
        dropped = _bytes(jp)
        jp.fb_gradient(fb, mu)
        assert _bytes(jp) == dropped < both - 8
        jp.update(fewer)
        J1, g1 = jp.fb_gradient(fb, mu)
        assert dropped < _bytes(jp) <= both - 8
    assert J1 == J and np.array_equal(g1, g)
