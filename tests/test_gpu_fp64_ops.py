"""Reciprocal and square root of the FP64 Riemann solver (csrc/teno_fp64.cuh)
against extended-precision results: within 0.51 units in the last place over the
exponents they are formed for, with significands next to powers of two and at
both ends; and the IEEE results, bit for bit, outside these (zeros, denormals,
the ends of the exponent range, infinities, NaN, roots of negative numbers)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::RuntimeWarning")]

SOURCE = r"""
#include "teno_fp64.cuh"
__global__ void k(const double* x, double* r, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = teno::rcp_f64(x[i]), s[i] = teno::sqrt_f64(x[i]);
}
extern "C" int run(const double* x, double* r, double* s, int n) {
  double* d = nullptr;
  const size_t b = sizeof(double) * n;
  if (cudaMalloc(&d, 3 * b) != cudaSuccess) return 1;
  cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
  cudaMemcpy(r, d + n, b, cudaMemcpyDeviceToHost);
  cudaMemcpy(s, d + 2 * n, b, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision")
    from paper_2105_02127_gb300 import build
    d = tmp_path_factory.mktemp("fp64")
    (d / "ops.cu").write_text(SOURCE)
    nvcc = os.path.join(build._cuda_home(), "bin", "nvcc")
    subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    f"-I{build.CSRC}", str(d / "ops.cu"), "-o", str(d / "ops.so")], check=True)
    lib = ctypes.CDLL(str(d / "ops.so"))

    def run(x):
        x = np.ascontiguousarray(x)
        r, s = np.empty_like(x), np.empty_like(x)
        assert lib.run(*(a.ctypes.data_as(ctypes.c_void_p) for a in (x, r, s)), len(x)) == 0
        return r, s

    return run


def _ulps(got, exact):
    return float((np.abs(got - exact) / np.spacing(np.abs(exact.astype(np.float64)))).max())


def test_error(ops):
    r = np.random.default_rng(1091)
    n = 1 << 20
    ends = np.concatenate([[0, 1, 2, 3], 2 ** 52 - np.arange(1, 5)])  # significand bits
    mant = np.concatenate([r.integers(0, 1 << 52, n), np.tile(ends, 1920)])
    expo = np.concatenate([r.integers(64, 1984, n), np.repeat(np.arange(64, 1984), len(ends))])
    x = (mant.astype(np.uint64) | (expo.astype(np.uint64) << np.uint64(52))).view(np.float64)
    assert x.min() == 2.0 ** -959 and x.max() < 2.0 ** 961
    rcp, root = ops(x)
    q = x.astype(np.longdouble)
    assert _ulps(rcp, 1 / q) <= 0.51
    assert _ulps(root, np.sqrt(q)) <= 0.51
    assert np.array_equal(ops(-x)[0], -rcp) and np.isnan(ops(-x)[1]).all()


def test_ieee_outside(ops):
    tiny, huge = 2.0 ** -959, 2.0 ** 961
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.2e-308, np.nextafter(tiny, 0),
                  -np.nextafter(tiny, 0), huge, -huge, 1.7e308, -1.7e308, -1.0, -4.0])
    rcp, root = ops(x)
    outside = np.abs(x) < tiny
    outside |= ~(np.abs(x) < huge)
    for got, want, which in ((rcp, 1.0 / x, outside), (root, np.sqrt(x), outside | (x < 0))):
        ok = got.view(np.int64) == want.view(np.int64)
        assert (ok | (np.isnan(got) & np.isnan(want)))[which].all()
