"""The double reciprocal, square root and order helpers of csrc/fp64.cuh against
numpy: results within 1 ulp of the rounded ones over the whole exponent range,
exact at the special values, comparisons equal to the floating-point ones."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "paper_2303_03026_gb300/csrc/fp64.cuh"
using namespace amrvac;
__global__ void k(const double* a, const double* b, double* o, int n) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s, is;
  sqrt_pair(a[i], s, is);
  const double x = fabs(a[i]), y = fabs(b[i]);
  const double r[10] = {rcp_T(a[i]), sqrt_T(a[i]), s, is, (double)gt0(a[i]), (double)ge0(a[i]),
                        min_pos(x, y), max_pos(x, y), (double)le_pos(x, y), (double)mid_range(a[i])};
  for (int c = 0; c < 10; c++) o[(size_t)c * n + i] = r[c];
}
extern "C" int run(const double* ha, const double* hb, double* ho, int n) {
  double *a, *b, *o;
  if (cudaMalloc(&a, 8ull * n) || cudaMalloc(&b, 8ull * n) || cudaMalloc(&o, 80ull * n)) return 1;
  cudaMemcpy(a, ha, 8ull * n, cudaMemcpyHostToDevice);
  cudaMemcpy(b, hb, 8ull * n, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(a, b, o, n);
  int e = cudaMemcpy(ho, o, 80ull * n, cudaMemcpyDeviceToHost);
  cudaFree(a); cudaFree(b); cudaFree(o);
  return e;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64")
    src, so = d / "m.cu", d / "m.so"
    src.write_text(SRC)
    nvcc = next((c for c in ("/usr/local/cuda/bin/nvcc",) if os.path.exists(c)), "nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I",
                    ROOT, "-shared", "-Xcompiler", "-fPIC", "-o", str(so), str(src)], check=True)
    return C.CDLL(str(so))


def _run(lib, a, b):
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    o = np.empty((10, a.size))
    p = lambda x: x.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert lib.run(p(a), p(b), p(o), C.c_int(a.size)) == 0
    return o


@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (-40.0, 40.0), (-300.0, 300.0)])
def test_within_one_ulp(lib, lo, hi):
    rng = np.random.Generator(np.random.PCG64(int(hi)))
    a = 10.0 ** rng.uniform(lo, hi, 400_000) * rng.choice([-1.0, 1.0], 400_000)
    b = 10.0 ** rng.uniform(lo, hi, 400_000) * rng.choice([-1.0, 1.0], 400_000)
    o = _run(lib, a, b)
    for got, want in ((o[0], 1.0 / a),):
        assert np.all(np.abs(got - want) <= np.spacing(np.abs(want)))
    p = a > 0
    q = a[p]
    assert np.all(np.abs(o[1][p] - np.sqrt(q)) <= np.spacing(np.sqrt(q)))
    # the product a (1/sqrt a) rounds once more; 1/sqrt a is compared with the
    # quotient of two rounded values
    assert np.all(np.abs(o[2][p] - np.sqrt(q)) <= 2 * np.spacing(np.sqrt(q)))
    assert np.all(np.abs(o[3][p] - 1 / np.sqrt(q)) <= 2 * np.spacing(1 / np.sqrt(q)))
    assert np.isnan(o[1][~p]).all()
    np.testing.assert_array_equal(o[4], (a > 0) * 1.0)
    np.testing.assert_array_equal(o[5], (a >= 0) * 1.0)
    x, y = np.abs(a), np.abs(b)
    np.testing.assert_array_equal(o[6], np.minimum(x, y))
    np.testing.assert_array_equal(o[7], np.maximum(x, y))
    np.testing.assert_array_equal(o[8], (x <= y) * 1.0)


def test_special_values(lib):
    inf, nan, tiny = np.inf, np.nan, 5e-324
    a = np.array([0.0, -0.0, inf, -inf, nan, tiny, -tiny, 2.3e-308, 1.7e308, 1.0, 4.0])
    o = _run(lib, a, np.zeros_like(a))
    np.testing.assert_array_equal(o[0][:5], [inf, -inf, 0.0, -0.0, nan])
    np.testing.assert_array_equal(o[0][-2:], [1.0, 0.25])
    np.testing.assert_array_equal(o[1][[0, 2, 4, 9, 10]], [0.0, inf, nan, 1.0, 2.0])
    assert np.isnan(o[1][3]) and abs(o[1][5]) < 1e-150
    np.testing.assert_array_equal(o[2][[0, 2, 9, 10]], [0.0, inf, 1.0, 2.0])
    with np.errstate(invalid="ignore"):
        np.testing.assert_array_equal(o[4], (a > 0) * 1.0)
        np.testing.assert_array_equal(o[5], (a >= 0) * 1.0)
