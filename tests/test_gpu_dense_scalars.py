"""The reciprocal square roots and reciprocals of csrc/dense.cuh against CUDA's
own functions, over the whole range of exponents, the ends of the range where
they hand over to those functions, and next to powers of two and of four.

Bounds (units in the last place of the correctly rounded value): 2 for the
square roots and 1 for the reciprocal, as derived beside the functions, plus
the 1 that CUDA's rsqrt may be off; the approximation's own error 2^-20."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_07811_gb300", "csrc")

SOURCE = """
#include "dense.cuh"
__global__ void scalars(const double* x, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  out[i] = dense::rsqrt_nr(v);
  out[n + i] = dense::rcp_nr(v);
  out[2 * n + i] = dense::rsqrt_third_order(v, dense::rsqrt_approx(v));
  out[3 * n + i] = dense::rsqrt_approx(v);
  out[4 * n + i] = rsqrt(v);
  out[5 * n + i] = 1.0 / v;
}
extern "C" int run(const double* x, double* out, int n) {
  double *dx = nullptr, *d = nullptr;
  int st = cudaMalloc(&dx, n * sizeof(double)) || cudaMalloc(&d, 6 * (size_t)n * sizeof(double));
  if (!st) {
    st = cudaMemcpy(dx, x, n * sizeof(double), cudaMemcpyHostToDevice);
    scalars<<<(n + 255) / 256, 256>>>(dx, d, n);
    st = st || cudaMemcpy(out, d, 6 * (size_t)n * sizeof(double), cudaMemcpyDeviceToHost);
  }
  cudaFree(dx);
  cudaFree(d);
  return st;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2512_07811_gb300 import build as B
    d = tmp_path_factory.mktemp("scalars")
    src, so = d / "scalars.cu", d / "scalars.so"
    src.write_text(SOURCE)
    subprocess.run([B.nvcc()] + B.ARCH + ["-std=c++17", "-O3", "-Xcompiler", "-fPIC", "-shared", "-I", CSRC, str(src),
                                          "-o", str(so), "-lcudart"], check=True)
    return ctypes.CDLL(str(so))


def _run(lib, x):
    x = np.ascontiguousarray(x, dtype=np.float64)
    out = np.empty((6, x.size))
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    assert lib.run(p(x), p(out), x.size) == 0
    return out


def _ulps(a, b):
    return np.abs(a - b) / np.spacing(np.abs(b))


def _values(lo, hi):
    rng = np.random.default_rng(3)
    e = np.arange(lo, hi)
    m = np.concatenate([[1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0)], rng.uniform(1, 2, 400)])
    return np.ldexp(m[:, None], e[None, :]).ravel()


def test_normal_range(lib):
    x = _values(-960, 961)
    rs, rc, third, approx, rs_cuda, rc_cuda = _run(lib, x)
    assert _ulps(rs, rs_cuda).max() <= 3
    assert _ulps(third, rs_cuda).max() <= 3
    assert _ulps(rc, rc_cuda).max() <= 1
    assert np.abs(approx / rs_cuda - 1).max() <= 2.0 ** -20


def test_ends_of_the_range(lib):
    """Where the approximations' own arguments or results leave the normal range."""
    cut = np.array([1e-290, 1e290])
    x = np.concatenate([_values(-1022, -955), _values(955, 1023), cut, np.nextafter(cut, 0), np.nextafter(cut, np.inf),
                        [5e-324, 1e-310, np.finfo(float).tiny, np.finfo(float).max]])
    rs, rc, _, _, rs_cuda, rc_cuda = _run(lib, x)
    assert _ulps(rs, rs_cuda).max() <= 3
    ok = np.isfinite(rc_cuda)
    assert np.array_equal(np.isfinite(rc), ok)
    assert _ulps(rc[ok], rc_cuda[ok]).max() <= 1


def test_special_values(lib):
    x = np.array([0.0, np.inf, np.nan, -1.0])
    rs, rc, _, _, rs_cuda, rc_cuda = _run(lib, x)
    assert np.array_equal(rs, rs_cuda, equal_nan=True)
    assert np.array_equal(rc, rc_cuda, equal_nan=True)
