"""The per-thread stack limit that a problem asks of the context."""
import subprocess
import sys

import pytest

from paper_2505_04328_gb300 import _build, build

pytestmark = pytest.mark.gpu

SCRIPT = """
import ctypes
import torch
import workloads
from paper_2505_04328_gb300 import JdProblem
torch.cuda.init()
torch.zeros(1, device="cuda")
cu = ctypes.CDLL("libcuda.so.1")
limit = ctypes.c_size_t()
def stack():
    assert cu.cuCtxGetLimit(ctypes.byref(limit), 0) == 0
    return limit.value
p = workloads.linear32(M=256, Nt=8).replace(lam=40.0)
before = stack()
for tc in (0, 1, 2, 3):
    with JdProblem(p, use_tensor_cores=tc) as jp:
        jp.gradient(workloads.random_control(p))
print(before, stack())
"""


def test_32_dimensions_ask_for_little_stack():
    """The d = 32 kernels' frames are below 1 KB (the limit holds memory for every resident
    thread: 12 KB were 3.8 GB of the device); run in a process of its own, as the limit stays."""
    build()
    r = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, timeout=600,
                       cwd=_build.ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    before, after = map(int, r.stdout.split())
    assert after <= max(before, 2048)
