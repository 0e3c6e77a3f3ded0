"""The FP64 functions of usp_math.cuh against CUDA's own and against wider
numbers: ordinary arguments over the ranges that the per-cell forms and the FP64
collision meet, and the arguments that take CUDA's function (zeros, denormals,
negative, very large and infinite values, NaN).

Bounds, in units of the last place of the result.  Reciprocal, quotient and root end
in one rounding of a value known to 2^-60 or better: 0.51.  The logarithms round once
at the end and have at most half a unit from their parts: 1."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2508_05642_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "%s/usp_math.cuh"
using namespace usp;
__global__ void run(int f, int n, const double* a, const double* b, double* own, double* lib) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x = a[i], y = b[i];
  switch (f) {
    case 0: own[i] = d_rcp(x); lib[i] = 1.0 / x; break;
    case 1: own[i] = d_div(x, y); lib[i] = x / y; break;
    case 2: own[i] = d_sqrt(x); lib[i] = sqrt(x); break;
    case 3: own[i] = d_log1p_inv(x); lib[i] = log1p(1.0 / x); break;
    default: own[i] = d_log(x); lib[i] = log(x);
  }
}
extern "C" int math_run(int f, int n, const double* a, const double* b, double* own, double* lib) {
  double* d = nullptr;
  const size_t s = (size_t)n * sizeof(double);
  if (cudaMalloc(&d, 4 * s) != cudaSuccess) return 1;
  cudaMemcpy(d, a, s, cudaMemcpyHostToDevice);
  cudaMemcpy(d + n, b, s, cudaMemcpyHostToDevice);
  run<<<(n + 255) / 256, 256>>>(f, n, d, d + n, d + 2 * n, d + 3 * n);
  cudaMemcpy(own, d + 2 * n, s, cudaMemcpyDeviceToHost);
  cudaMemcpy(lib, d + 3 * n, s, cudaMemcpyDeviceToHost);
  const cudaError_t e = cudaDeviceSynchronize();
  cudaFree(d);
  return (int)e;
}
"""
NAMES = ["rcp", "div", "sqrt", "log1p_inv", "log"]
W = np.longdouble
WIDE = [lambda x, y: 1 / x, lambda x, y: x / y, lambda x, y: np.sqrt(x),
        lambda x, y: np.log1p(1 / x), lambda x, y: np.log(x)]
BOUND = [0.51, 0.51, 0.51, 1.0, 1.0]


@pytest.fixture(scope="module")
def math_lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("math")
    (d / "m.cu").write_text(SRC % build.CSRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", str(d / "m.cu"), "-o",
                    str(d / "libm.so"), "-cudart", "static"], check=True)
    return C.CDLL(str(d / "libm.so"))


def _run(lib, f, a, b):
    a, b = np.ascontiguousarray(a, dtype=float), np.ascontiguousarray(b, dtype=float)
    own, ref = np.full(len(a), 7.5), np.full(len(a), 7.5)
    p = lambda v: v.ctypes.data_as(C.c_void_p)
    assert lib.math_run(f, len(a), p(a), p(b), p(own), p(ref)) == 0
    return own, ref


def _arguments(f, rng, n):
    """Over the whole range, near 1, and mean levels from 10^-9 to 10^5."""
    x = 2.0 ** (rng.uniform(-300, 300, n) if f != 3 else rng.uniform(-100, 100, n))
    x[:n // 4] = rng.uniform(0.5, 2.0, n // 4)
    x[n // 4:n // 2] = 10.0 ** rng.uniform(-9, 5, n // 4)
    if f < 2:
        x *= rng.choice([-1.0, 1.0], n)
    return x, 2.0 ** rng.uniform(-300, 300, n) * rng.choice([-1.0, 1.0], n)


@pytest.mark.parametrize("f", range(5), ids=NAMES)
def test_ordinary_arguments_within_their_bounds(math_lib, f):
    x, y = _arguments(f, np.random.default_rng(f), 200000)
    own, lib = _run(math_lib, f, x, y)
    ref = WIDE[f](W(x), W(y))
    ulp = W(2.0) ** (np.floor(np.log2(np.abs(ref.astype(float)))) - 52)
    err = np.abs(W(own) - ref) / ulp
    k = int(np.argmax(err))
    rms = [float(np.sqrt(np.mean(((W(a) - ref) / ulp) ** 2))) for a in (own, lib)]
    assert err[k] <= BOUND[f], (NAMES[f], x[k], y[k], own[k], float(err[k]))
    assert rms[0] <= 1.01 * rms[1], (NAMES[f], rms)      # no less exact than CUDA's


@pytest.mark.parametrize("f", range(5), ids=NAMES)
def test_other_arguments_take_the_library_value(math_lib, f):
    v = np.array([0.0, 5e-324, 1e-310, 2.2250738585072014e-308, 1e-300, 1e-200, 1.0, 3.0, 600.0,
                  700.0, 710.0, 1e200, 1e300, 8.9e307, 1.7976931348623157e308, np.inf])
    v = np.concatenate([v, -v, [np.nan]])
    x, y = (a.ravel() for a in np.meshgrid(v, v))
    if f != 1:
        x, y = v, v
    own, lib = _run(math_lib, f, x, y)
    # where the library's value is no ordinary number, it is that value
    special = ~np.isfinite(lib) | (lib == 0) | (np.abs(lib) < 2.3e-308)
    assert special.any()
    assert np.array_equal(np.isnan(own), np.isnan(lib))
    s = special & ~np.isnan(lib)
    assert np.array_equal(own[s], lib[s]), (x[s][own[s] != lib[s]], y[s][own[s] != lib[s]])
    assert np.array_equal(np.signbit(own[s]), np.signbit(lib[s]))
    r = ~special
    assert np.all(np.abs(own[r] - lib[r]) <= 2 ** -51 * np.abs(lib[r]))
