"""Every argument of the generator's Box-Muller transforms: the FP32 radius' square root
against CUDA's rounding intrinsic bit for bit, the FP64 radius and angle against extended
precision.  The device functions are called from a small library built here against the
kernels' own header."""
import concurrent.futures as cf
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2505_04328_gb300 import _build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "jd_device.cuh"
using namespace jd;
// out[0]: floats of [lo, hi) (as bits) whose root differs from the rounding intrinsic;
// out[1]: radius arguments -2 log u of the 2^23 uniforms that differ, or lie outside [lo, hi)
__global__ void roots(uint32_t lo, uint32_t hi, unsigned long long *out) {
  const uint32_t n = gridDim.x * blockDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long a = 0, b = 0;
  for (uint32_t v = lo + i0; v < hi; v += n) {
    const float t = __uint_as_float(v);
    a += __float_as_uint(sqrt_radius(t)) != __float_as_uint(__fsqrt_rn(t));
  }
  for (uint32_t i = i0; i < (1u << 23); i += n) {
    const float t = Ar<float>::mul(-2.f, Ar<float>::log(Ar<float>::u01(i << 9)));
    const uint32_t v = __float_as_uint(t);
    b += v < lo || v >= hi || __float_as_uint(sqrt_radius(t)) != __float_as_uint(__fsqrt_rn(t));
  }
  atomicAdd(out, a);
  atomicAdd(out + 1, b);
}
__global__ void transforms(double *r, double *c, double *s) {
  const uint32_t i = blockIdx.x * 256 + threadIdx.x;   // the grid covers the 2^23 arguments
  r[i] = __dsqrt_rn(n64::neg2_log(i << 9));
  n64::cos_sin_2pi(i << 9, c[i], s[i]);
}
extern "C" int run_roots(uint32_t lo, uint32_t hi, unsigned long long *host) {
  unsigned long long *d = nullptr;
  if (cudaMalloc(&d, 16) != cudaSuccess || cudaMemset(d, 0, 16) != cudaSuccess) return 1;
  roots<<<1024, 256>>>(lo, hi, d);
  const cudaError_t e = cudaMemcpy(host, d, 16, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
extern "C" int run_transforms(double *r, double *c, double *s) {
  const size_t n = 1u << 23;
  double *d = nullptr;
  if (cudaMalloc(&d, 3 * n * 8) != cudaSuccess) return 1;
  transforms<<<(unsigned)(n / 256), 256>>>(d, d + n, d + 2 * n);
  cudaError_t e = cudaMemcpy(r, d, n * 8, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(c, d + n, n * 8, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(s, d + 2 * n, n * 8, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def transforms(tmp_path_factory):
    d = tmp_path_factory.mktemp("normals")
    src, lib = os.path.join(d, "normals.cu"), os.path.join(d, "normals.so")
    with open(src, "w") as f:
        f.write(SRC)
    r = subprocess.run([_build.nvcc()] + _build.NVCC_FLAGS + ["-shared", "-o", lib, src], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return ctypes.CDLL(lib)


def test_fp32_radius_root_is_correctly_rounded(transforms):
    """Every float of [3e-8, 64) and every -2 log u: the intrinsic's bits."""
    lo, hi = np.array([3e-8, 64.0], np.float32).view(np.uint32)
    out = np.zeros(2, np.uint64)
    assert transforms.run_roots(ctypes.c_uint32(int(lo)), ctypes.c_uint32(int(hi)), ctypes.c_void_p(out.ctypes.data)) == 0
    assert out.tolist() == [0, 0]


def test_fp64_radius_and_angle_of_every_argument(transforms):
    """Radius within 0.86 and cosine and sine within 1.0 units of the last place."""
    n = 1 << 23
    got = [np.empty(n) for _ in range(3)]
    assert transforms.run_transforms(*[ctypes.c_void_p(g.ctypes.data) for g in got]) == 0
    L = np.longdouble

    def ulps(x, exact):
        return float(np.max(np.abs(x.astype(L) - exact) / np.spacing(np.abs(exact.astype(np.float64))).astype(L)))

    def part(a):
        i = slice(a, a + (1 << 17))
        u = (np.arange(a, a + (1 << 17)).astype(L) + L(0.5)) * L(2.0) ** -23
        r = np.sqrt(-2 * np.log(u))
        q = np.floor(4 * u + L(0.5))             # nearest quarter turn; the rest is exact
        x = (u - q / 4) * 2 * (L(3.141592653589793116) + L(1.2246467991473532e-16))
        q = q.astype(int) % 4
        c, s = np.cos(x), np.sin(x)
        return (ulps(got[0][i], r), ulps(got[1][i], np.choose(q, [c, -s, -c, s])),
                ulps(got[2][i], np.choose(q, [s, c, -s, -c])))

    with cf.ThreadPoolExecutor(min(16, os.cpu_count() or 1)) as ex:
        worst = np.max(list(ex.map(part, range(0, n, 1 << 17))), axis=0)
    print("largest errors (radius, cosine, sine):", worst)
    assert worst[0] <= 0.86 and worst[1] <= 1.0 and worst[2] <= 1.0
