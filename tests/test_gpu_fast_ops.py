"""FP64 reciprocal, quotient, root and reciprocal root of the FP64 kernels (FastOps64): each within 0.51 units
in the last place of the exact value (0.5 for a correctly rounded one, and below 2^-7 for the FP32
correction), for arguments over the whole range, beside powers of two and perfect squares. The root of 0 and
of subnormals is 0, and CheckedOps64 gives special arguments what IEEE gives them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_0904_0232_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "metric.cuh"
using grpic::CheckedOps64;
using grpic::FastOps64;
__global__ void k(const double* x, const double* a, double* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double ri;
  o[i] = FastOps64::rcp(x[i]);
  o[n + i] = FastOps64::div(a[i], x[i]);
  o[2 * n + i] = FastOps64::root(x[i]);
  o[3 * n + i] = FastOps64::root_and_rsqrt(x[i], &ri);
  o[4 * n + i] = ri;
  o[5 * n + i] = CheckedOps64::div(a[i], x[i]);
  o[6 * n + i] = CheckedOps64::root(x[i]);
}
extern "C" int run(const double* x, const double* a, double* o, int n) {
  double *dx = nullptr, *da = nullptr, *d = nullptr;
  if (cudaMalloc(&dx, 8ll * n) || cudaMalloc(&da, 8ll * n) || cudaMalloc(&d, 56ll * n)) return 1;
  cudaMemcpy(dx, x, 8ll * n, cudaMemcpyHostToDevice);
  cudaMemcpy(da, a, 8ll * n, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(dx, da, d, n);
  const int e = cudaMemcpy(o, d, 56ll * n, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(da);
  cudaFree(d);
  return e;
}
"""


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("fast_ops")
    src, lib = d / "ops.cu", d / "ops.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                                                  os.path.join(build.CSRC), "-o", str(lib), str(src)], check=True)
    run = ctypes.CDLL(str(lib)).run

    def call(x, a):
        out = np.zeros((7, x.size))
        p = [v.ctypes.data_as(ctypes.c_void_p) for v in (x, a, out)]
        assert run(*p, x.size) == 0
        return out

    return call


def _arguments(kind, n, rng):
    if kind == "range":
        return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-885, 885, n))
    if kind == "ordinary":
        return np.exp(rng.uniform(-12.0, 12.0, n))
    if kind == "powers":  # within 64 units of a power of two
        p = np.ldexp(1.0, rng.integers(-60, 60, n))
        return (p.view(np.int64) + rng.integers(-64, 65, n)).view(np.float64)
    return rng.integers(1, 1 << 26, n).astype(np.float64) ** 2


@pytest.mark.parametrize("kind", ["range", "ordinary", "powers", "squares"])
def test_within_half_a_unit(ops, kind):
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("no extended precision on this host")
    rng = np.random.default_rng(5)
    n = 1 << 20
    x = _arguments(kind, n, rng)
    a = rng.normal(0.0, 1.0, n)
    out = ops(x, a)
    X, s = x.astype(np.longdouble), np.sqrt(x.astype(np.longdouble))
    for got, exact in zip(out, (1 / X, a / X, s, s, 1 / s, a / X, s)):
        e = np.floor(np.log2(np.abs(exact)))  # the binade of the exact value (log2 in the same precision)
        assert np.max(np.abs(got - exact) / np.exp2(e - 52)) <= 0.51


def test_special_arguments(ops):
    x = np.array([0.0, -0.0, 1e-310, 2.3e-308, 1e-280, 1e280, 1.7e308, np.inf, -np.inf, np.nan, -1.0, -4.0])
    for a in (1.0, 0.0, np.inf, -np.inf, np.nan):
        out = ops(x, np.full_like(x, a))
        with np.errstate(all="ignore"):
            assert np.array_equal(out[5], a / x, equal_nan=True)
            assert np.array_equal(out[6], np.sqrt(x), equal_nan=True)
        assert np.all(out[2][:3] == 0.0) and np.all(out[3][:3] == 0.0)
