"""rcp_, rsqrt_ and sqrt_pos of the FP64 passes (lhy.cuh) against the correctly rounded
1/x, 1/sqrt(x) and sqrt(x) over the range they are used on.

One third-order step from an approximation with e < 2^-19.  rcp_: y + y (e + e^2) is
rounded once, e^3 < 2^-57, and the roundings inside (e + e^2) are 2^-53 e: half an ulp and
2^-57 beyond.  rsqrt_: e = 1 - (x y) y takes the rounding of x y, 2^-53, of which half
reaches the result: 2^-54 + half an ulp (2^-53 relative).  sqrt_pos: x times that,
rounded again."""
import ctypes as ct
import subprocess

import numpy as np
import pytest

from paper_2510_24543_gb300 import build as B

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
SRC = r"""
#include "lhy.cuh"
__global__ void k(int op, int n, const double* x, double* y) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    y[i] = op == 0 ? egpe::rcp_(x[i]) : op == 1 ? egpe::rsqrt_(x[i]) : egpe::sqrt_pos(x[i]);
}
extern "C" int apply(int op, int n, const double* x, double* y) {
  double* d = nullptr;
  if (cudaMalloc(&d, 2 * n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, x, n * sizeof(double), cudaMemcpyHostToDevice);
  k<<<152, 256>>>(op, n, d, d + n);
  const cudaError_t e = cudaMemcpy(y, d + n, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def apply(tmp_path_factory):
    d = tmp_path_factory.mktemp("recip")
    (d / "r.cu").write_text(SRC)
    cmd = [B._nvcc()] + B.ARCH + B.FLAGS + ["-I" + B.CSRC, "-shared", str(d / "r.cu"), "-o", str(d / "r.so")]
    subprocess.run(cmd, check=True, capture_output=True)
    lib = ct.CDLL(str(d / "r.so"))

    def run(op, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        assert lib.apply(op, x.size, x.ctypes.data_as(ct.c_void_p), y.ctypes.data_as(ct.c_void_p)) == 0
        return y
    return run


def _points():
    rng = np.random.default_rng(11)
    dense = 1.0 + rng.random(200000) * 3.0  # two octaves: every case of the square root's exponent
    wide = 2.0 ** rng.uniform(-980.0, 980.0, 200000)
    edges = np.ldexp(1.0, np.arange(-980, 981)) * (1.0 + np.array([[0.0], [2.0 ** -52], [-(2.0 ** -53)], [0.5]]))
    return np.concatenate([dense, wide, edges.ravel()])


def _rel(y, exact):
    return float(np.max(np.abs((y - exact) / exact)))


def test_against_correct_rounding(apply):
    x = _points()
    xl = x.astype(np.longdouble)
    assert np.finfo(np.longdouble).nmant >= 63  # extended or quadruple precision here
    assert _rel(apply(0, x), 1 / xl) < U * 1.1
    assert _rel(apply(1, x), 1 / np.sqrt(xl)) < U * 1.6
    assert _rel(apply(2, x), np.sqrt(xl)) < U * 2.7


def test_special_values(apply):
    assert np.all(apply(2, [0.0, 1e-301, 5e-324]) == 0.0)
    assert np.isnan(apply(2, [np.nan]))[0]
    for op in (0, 1):
        assert not np.any(np.isfinite(apply(op, [0.0, np.nan])))
