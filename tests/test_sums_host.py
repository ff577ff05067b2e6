"""The sums that kernels carry in floats for FP32 data (csrc/sums.cuh), compiled for the host: at least
as accurate as FP64 sums of the converted values.

Bound against the exact sum: an FP64 sum of n terms may be off by n 2^-53 of the sum of their sizes, a
triple by n 2^-70 (2^-72 an addition, up to four additions a term) plus two roundings of the result."""
import ctypes
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0906_4548_gb300", "csrc")
SOURCE = """
#include <math.h>
#define __device__
#define __forceinline__ inline
static inline float rsqrtf(float x) { return (1.f / sqrtf(x)) * (1.f + 2.4e-7f); }  // two ulp off, as the device's may be
#include "sums.cuh"
using namespace dgp;
extern "C" {
double root_sum(const int* n2, const int* twice, int n) {
  ShellSum<float> s;
  for (int i = 0; i < n; ++i) s.add_root(n2[i], twice[i]);
  return s.value();
}
double norm_sum(const float* x, const float* y, int n) {
  ShellSum<float> s;
  for (int i = 0; i < n; ++i) s.add_norm(x[i], y[i]);
  return s.value();
}
double value_sum(const float* x, int n) {
  ThreadSum<float> s;
  for (int i = 0; i < n; ++i) s.add(x[i]);
  return s.value();
}
double inverse_sum(const float* x, int n) {
  ThreadSum<float> s;
  for (int i = 0; i < n; ++i) s.add_inverse(x[i]);
  return s.value();
}
double pair_sum(const float* a, const float* b, int n) {
  ProductSum<float> s;
  for (int i = 0; i < n; ++i) s.add(a[i], b[i]);
  return s.value();
}
double triple_sum(const float* a, const float* b, const float* c, int n) {
  ProductSum<float> s;
  for (int i = 0; i < n; ++i) s.add(a[i], b[i], c[i]);
  return s.value();
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("sums")
    src, out = d / "sums.cpp", d / "libsums.so"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-shared", "-fPIC",
                    "-I" + CSRC, str(src), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


def _call(lib, name, *arrays):
    fn = getattr(lib, name)
    fn.restype = ctypes.c_double
    return fn(*[ctypes.c_void_p(a.ctypes.data) for a in arrays], len(arrays[0]))


def _check(got, terms):
    exact, size = sum(terms), sum(abs(t) for t in terms)
    bound = len(terms) * size / 2 ** 70 + abs(exact) / 2 ** 52
    assert abs(Fraction(got) - exact) <= bound, float((Fraction(got) - exact) / exact) * 2.0 ** 53


def _floats(seed, n, spread):
    rng = np.random.default_rng(seed)
    return (rng.normal(size=n) * 2.0 ** rng.uniform(-spread, 0, n)).astype(np.float32)


@pytest.mark.parametrize("n", [1, 7, 900, 8000])
def test_root_sum(lib, n):
    rng = np.random.default_rng(n)
    n2 = rng.integers(1, 3 * 256 ** 2 + 1, n).astype(np.int32)
    tw = rng.integers(0, 2, n).astype(np.int32)
    # sqrt to 100 bits below the point
    terms = [(1 + int(t)) * Fraction(math.isqrt(int(v) << 200), 1 << 100) for v, t in zip(n2, tw)]
    _check(_call(lib, "root_sum", n2, tw), terms)


@pytest.mark.parametrize("n", [1, 7, 900, 8000])
@pytest.mark.parametrize("spread", [0, 12])
def test_norm_sum(lib, n, spread):
    x, y = _floats(n, n, spread), _floats(n + 1, n, spread)
    terms = [Fraction(float(a)) ** 2 + Fraction(float(b)) ** 2 for a, b in zip(x, y)]
    _check(_call(lib, "norm_sum", x, y), terms)


@pytest.mark.parametrize("n", [1, 7, 900, 8000])
@pytest.mark.parametrize("spread", [0, 12])
def test_product_sums(lib, n, spread):
    a, b, c = (_floats(n + i, n, spread) for i in range(3))
    f = [[Fraction(float(v)) for v in x] for x in (a, b, c)]
    _check(_call(lib, "pair_sum", a, b), [x * y for x, y, _ in zip(*f)])
    _check(_call(lib, "triple_sum", a, b, c), [x * y * z for x, y, z in zip(*f)])


@pytest.mark.parametrize("n", [1, 7, 900, 8000])
@pytest.mark.parametrize("spread", [0, 12])
def test_value_and_inverse_sums(lib, n, spread):
    x = _floats(n + 5, n, spread)
    _check(_call(lib, "value_sum", x), [Fraction(float(v)) for v in x])
    _check(_call(lib, "inverse_sum", x), [1 / Fraction(float(v)) for v in x])
