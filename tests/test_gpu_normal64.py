"""The normals of the generator against extended precision."""
import numpy as np
import pytest

import workloads
from paper_2505_04328_gb300 import JdProblem, build

pytestmark = pytest.mark.gpu


def _philox(c, key):
    c = [np.asarray(v, dtype=np.uint64) for v in c]
    k = [np.uint64(key & 0xFFFFFFFF), np.uint64(key >> 32)]
    mask, s32 = np.uint64(0xFFFFFFFF), np.uint64(32)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> s32) ^ c[1] ^ k[0], p1 & mask, (p0 >> s32) ^ c[3] ^ k[1], p0 & mask]
        k = [(k[0] + np.uint64(0x9E3779B9)) & mask, (k[1] + np.uint64(0xBB67AE85)) & mask]
    return c


@pytest.mark.parametrize("prec,tol", [("fp64", 2.5 * 2.0 ** -52), ("fp32", 4 * 2.0 ** -23)])
@pytest.mark.parametrize("seed", [0, 5, (7 << 32) + 1])
def test_normals_of_one_step(seed, prec, tol):
    """One step of length 1 from 0 with unit noise and no drift is the step's normal pair.
    FP64: radius and cosine are within 0.86 and 1.0 units of the last place and the product
    rounds once: below 2.5 units, 2.5 x 2^-52 of the value.  FP32: the library's logarithm
    (1 unit, halved by the root), root (0.5), sincospi (2) and product (0.5): 4 units."""
    build()
    M = 1 << 16
    p = workloads.ks_oscillator(M=M, Nt=1).replace(
        T=1.0, A=np.zeros((2, 2)), B=np.zeros((2, 1)), sigma=np.ones(2), x0=np.zeros(2), lam=0.0,
        xd=np.zeros((2, 2)), seed=seed)
    with JdProblem(p, prec=prec) as jp:
        X, _, _ = jp.sample_paths(np.zeros((1, 1)), 0, M, lam=False)
    m = np.arange(M, dtype=np.uint64)
    w = _philox([0 * m, m, 0 * m, 0 * m], seed)
    L = np.longdouble
    u = [((v >> np.uint64(9)).astype(L) + L(0.5)) * L(2.0) ** -23 for v in (w[1], w[2])]
    # the angle reduced to the nearest quarter turn, exactly
    q = np.floor(4 * u[1] + L(0.5))
    a = (u[1] - q / 4) * 2 * (L(3.141592653589793116) + L(1.2246467991473532e-16))
    q = q.astype(int) % 4
    c, s = np.cos(a), np.sin(a)
    r = np.sqrt(-2 * np.log(u[0]))
    z = np.stack([r * np.choose(q, [c, -s, -c, s]), r * np.choose(q, [s, c, -s, -c])], axis=1)
    assert np.max(np.abs((X[:, 1, :] - z) / z)) <= tol
