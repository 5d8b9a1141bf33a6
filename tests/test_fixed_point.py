"""Fixed-point sums of products of the FP64 block inverses (``csrc/fp64_util.cuh``), compiled for the host from the
kernels' own header and compared with exact rational arithmetic.

Bar of a sum of m products a_k b_k under one exponent per factor: with A, B the powers of two above the largest |a|,
|b|, each digit pair holds its value to 2^-58 of A (B), the products of the two low digits left out are at most 2^-58
A B each, the carry of the middle digits is rounded once (2^-57 A B), and the final sum and conversion are rounded to
FP64: (3 m + 2) 2^-58 A B + 2^-51 (|c| + |sum|).
"""
import ctypes
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1709_05660_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
struct int2 { int x, y; };
static inline int2 make_int2(int x, int y) { return int2{x, y}; }
static inline long long __double_as_longlong(double a) { long long b; std::memcpy(&b, &a, 8); return b; }
static inline int __double2hiint(double a) { return (int)(__double_as_longlong(a) >> 32); }
static inline double __hiloint2double(int hi, int lo) {
  const long long b = ((long long)hi << 32) | (uint32_t)lo;
  double a;
  std::memcpy(&a, &b, 8);
  return a;
}
using std::fma;
#include "fp64_util.cuh"
extern "C" double sum_of_products(int m, const double* a, const double* b, double c) {
  using namespace fsi;
  int ea = 0, eb = 0;
  for (int k = 0; k < m; ++k) {
    ea = fix_exp(a[k]) > ea ? fix_exp(a[k]) : ea;
    eb = fix_exp(b[k]) > eb ? fix_exp(b[k]) : eb;
  }
  long long hh = 0, mid = 0;
  for (int k = 0; k < m; ++k) fix_mad(hh, mid, fix_digits(a[k], ea), fix_digits(b[k], eb));
  return fix_add(c, hh, mid, ea, eb);
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fixed_point")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([gxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o",
                    str(d / "shim.so")], check=True)
    lib = ctypes.CDLL(str(d / "shim.so"))
    lib.sum_of_products.restype = ctypes.c_double
    lib.sum_of_products.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double]

    def run(a, b, c):
        a, b = np.ascontiguousarray(a, dtype=np.float64), np.ascontiguousarray(b, dtype=np.float64)
        return lib.sum_of_products(len(a), a.ctypes.data, b.ctypes.data, float(c))
    return run


@pytest.mark.parametrize("m", [1, 4, 15, 16, 32])
@pytest.mark.parametrize("spread", [0, 8, 40, 70])
def test_against_rationals(sums, m, spread):
    rng = np.random.default_rng(100 * m + spread)
    for scale in (0, -300, 300):
        for _ in range(50):
            a = rng.uniform(-1, 1, m) * 2.0 ** (rng.integers(-spread, 1, m) + scale)
            b = rng.uniform(-1, 1, m) * 2.0 ** (rng.integers(-spread, 1, m) - scale // 2)
            c = rng.uniform(-1, 1) * 2.0 ** (scale - scale // 2)
            exact = Fraction(c) + sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
            top = Fraction(2) ** (math.frexp(np.abs(a).max())[1] + math.frexp(np.abs(b).max())[1])
            bar = (3 * m + 2) * top / 2 ** 58 + (abs(Fraction(c)) + abs(exact)) / 2 ** 51
            assert abs(Fraction(sums(a, b, c)) - exact) <= bar


@pytest.mark.parametrize("a,b,c", [([2.0 ** 600], [2.0 ** 600], 1.0), ([-2.0 ** 1023], [2.0 ** 1023], 1.0),
                                   ([2.0 ** 1000, 0.0], [0.0, 2.0 ** 1000], 3.0),
                                   ([0.0, 0.0], [0.0, 0.0], 2.5), ([2.0 ** 511], [2.0 ** 511], 0.0),
                                   ([1.0, 1.0], [1.0, -1.0], -7.0)])
def test_ends_of_the_range(sums, a, b, c):
    """As FP64 products: infinite beyond the range, exact here within it, and c alone where every product is zero
    (entries far below their row's largest are not among these: they keep what the bar above says)."""
    with np.errstate(over="ignore"):
        want = float(c + np.sum(np.array(a) * np.array(b)))
    assert sums(a, b, c) == want
