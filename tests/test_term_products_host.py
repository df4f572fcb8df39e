"""Products and sums of products on the integer units (csrc/fixedpoint.cuh, the
four-multiplication form) compiled for the host with g++ and compared with
exact rational values."""
import ctypes
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1410_1764_gb300", "csrc")

HARNESS = r"""
#include "fixedpoint.cuh"
using namespace chemora;
extern "C" int mul6(double a, double b, long long* m) {
  const fx::Parts p = fx::term_product<6>(fx::term<10>(a), fx::term<7>(b));
  *m = p.m;
  return p.e;
}
template <int N> static int dotn(const double* a, const double* b, double* out) {
  constexpr int K = fx::DotGuard<N>::k;
  fx::Parts p[N];
  for (int q = 0; q < N; ++q) p[q] = fx::term_product<K>(fx::term<10>(a[q]), fx::term<K + 1>(b[q]));
  return fx::dot(p, out) ? K : 0;
}
extern "C" int dot(int n, const double* a, const double* b, double* out) {
  return n == 4 ? dotn<4>(a, b, out) : (n == 6 ? dotn<6>(a, b, out) : dotn<12>(a, b, out));
}
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("terms")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    D = ctypes.POINTER(ctypes.c_double)
    lib.mul6.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.POINTER(ctypes.c_longlong)]
    lib.dot.argtypes = [ctypes.c_int, D, D, D]
    return lib


def test_products(L):
    """Within six units of the exact product: the low words' product, two
    halved low words and three roundings down are at most one unit each (two
    units, the mean, are added back)."""
    rng, m = np.random.default_rng(0), ctypes.c_longlong()
    ends = [1.0, -1.0, 2.0 - 2.0 ** -52, -2.0 + 2.0 ** -52, 1.0 + 2.0 ** -52]
    pairs = [(a, b) for a in ends for b in ends]
    pairs += [tuple(rng.standard_normal(2) * np.exp2(rng.integers(-400, 400, 2))) for _ in range(3000)]
    for a, b in pairs:
        e = L.mul6(float(a), float(b), ctypes.byref(m))
        unit = Fraction(2) ** (e - 1075 - 6)
        assert abs(m.value * unit - Fraction(float(a)) * Fraction(float(b))) < 6 * unit
        assert 2 ** 57 - 6 <= abs(m.value) <= 2 ** 59
    assert L.mul6(0.0, 3.0, ctypes.byref(m)) == L.mul6(-3.0, -0.0, ctypes.byref(m)) == -4096
    for a, b in ((math.inf, 1.0), (0.0, math.nan), (5e-324, 1e300), (-math.inf, 0.0), (1e300, 1e300)):
        assert L.mul6(a, b, ctypes.byref(m)) > 2030


@pytest.mark.parametrize("n", [4, 6, 12])
@pytest.mark.parametrize("spread,cancel", [(0, False), (4, False), (60, False), (2, True)])
def test_sums(L, n, spread, cancel):
    """Within half an ulp of the sum and seven units (six of the product, one
    of the alignment) of the largest product's binade per term; cancel: the
    second half of the terms takes the first half away but for the last bits."""
    rng = np.random.default_rng(n + spread)
    D = ctypes.c_double * n
    for _ in range(300):
        a, b = rng.standard_normal((2, n)) * np.exp2(rng.uniform(-spread, 0, (2, n))) * 2.0 ** int(rng.integers(-200, 200))
        if cancel:
            a[n // 2:], b[n // 2:] = -a[:n // 2] * (1 + 2.0 ** -50), b[:n // 2]
        out = ctypes.c_double()
        K = L.dot(n, D(*a), D(*b), ctypes.byref(out))
        assert K
        prods = [Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b)]
        exact = sum(prods)
        # the largest e of a product is at most one above its binade
        e = max(math.frexp(float(x))[1] + math.frexp(float(y))[1] for x, y in zip(a, b))
        unit = Fraction(2) ** (e - 1 - 52 - K)
        assert abs(Fraction(out.value) - exact) <= 7 * n * unit + abs(exact) / 2 ** 53 * (1 + Fraction(1, 2 ** 20))
    z = D(*([0.0] * n))
    assert L.dot(n, z, D(*([3.0] * n)), ctypes.byref(out)) and out.value == 0.0
    for bad in (math.nan, math.inf, 1e308, 1e-300):
        x = [1.0] * n if not bad == 1e-300 else [bad] * n
        x[-1] = bad
        assert L.dot(n, D(*x), D(*([1e4 if bad == 1e308 else 1e-10] * n)), ctypes.byref(out)) == 0


@pytest.mark.parametrize("n", [4, 6, 12])
@pytest.mark.parametrize("field", ["normal", "spread", "sparse", "positive", "dominant"])
def test_sums_against_fp64(L, n, field):
    """No further from the exact sum than a chain of FP64 fmas, and without a
    bias: in ulps of the largest product, over 3000 sums."""
    rng = np.random.default_rng(n)
    D = ctypes.c_double * n
    err = np.zeros((3000, 2))
    for i in range(len(err)):
        a, b = rng.standard_normal((2, n))
        if field == "spread":
            a, b = a * np.exp2(-8 * rng.random(n)), b * np.exp2(-8 * rng.random(n))
        elif field == "sparse":
            a[max(2, n // 3):] = 0.0
        elif field == "positive":
            a, b = abs(a), abs(b)
        elif field == "dominant":
            a[1:] *= 1e-3
        out = ctypes.c_double()
        assert L.dot(n, D(*a), D(*b), ctypes.byref(out))
        prods = [Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b)]
        chain = 0.0
        for p in prods:  # a correctly rounded fma
            chain = float(Fraction(chain) + p)
        ulp = Fraction(2) ** (math.frexp(float(max(map(abs, prods))))[1] - 53)
        err[i] = [float((Fraction(v) - sum(prods)) / ulp) for v in (chain, out.value)]
    rms = np.sqrt((err ** 2).mean(0))
    # a unit's share of the ulp (what is added back is whole units), and three standard errors of the mean
    bias = 0.06 + 3 * rms[1] / len(err) ** 0.5
    assert rms[1] <= rms[0] and abs(err[:, 1].mean()) <= bias, (rms, err.mean(0))
