"""The integer stencils (csrc/fixedpoint.cuh) compiled for the host with g++
and compared with exact rational sums: the aligned values, the rounding back
to a double, and the order-4 star Laplacian as csrc/wave_point.cuh forms it."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1410_1764_gb300", "csrc")

HARNESS = r"""
#include "star_march.cuh"
using namespace chemora;
extern "C" int lap(const double* n, double c, double* out) {
  constexpr int K = Guard<2>::lap;
  int e = fx::exponent(c);
  for (int q = 0; q < 12; ++q) e = fx::emax(e, fx::exponent(n[q]));
  if (!fx::in_range(e)) return 0;
  long long s[2] = {0, 0};
  for (int q = 0; q < 12; ++q) s[q % 4 / 2] += fx::align<K>(n[q], e);
  *out = star_lap<2>(s, fx::align<K>(c, e), e);
  return 1;
}
"""


@pytest.fixture(scope="module")
def lap(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-x", "c++", "-I", CSRC, str(src), "-o", str(so)],
                   check=True)
    L = ctypes.CDLL(str(so))
    L.lap.argtypes = [ctypes.POINTER(ctypes.c_double), ctypes.c_double, ctypes.POINTER(ctypes.c_double)]

    def f(n, c):
        a = (ctypes.c_double * 12)(*n)
        o = ctypes.c_double()
        return o.value if L.lap(a, c, ctypes.byref(o)) else None
    return f


@pytest.mark.parametrize("spread,lo", [(0, 0.5), (1, 0.0), (8, 0.0), (60, 0.0), (500, 0.0)])
def test_star_laplacian_against_rationals(lap, spread, lo):
    """Values of one binade, of one sign-changing range, and spread over 2^8 ..
    2^500: the result is the exact sum to half an ulp plus the truncation of
    the smaller values, at most 192 units of 2^-58 of the largest value's
    binade (nothing is truncated within 2^6 of the largest)."""
    rng = np.random.default_rng(spread)
    for _ in range(300):
        v = rng.uniform(lo, 1.0, 13) * np.exp2(rng.uniform(-spread, 0, 13)) * np.exp2(rng.integers(-300, 300))
        if lo == 0.0:
            v *= rng.choice([-1.0, 1.0], 13)
        x = [float(q) for q in v]
        n, c = x[:12], x[12]
        exact = Fraction(0)
        for q in range(0, 12, 4):
            exact += 16 * (Fraction(n[q]) + Fraction(n[q + 1])) - (Fraction(n[q + 2]) + Fraction(n[q + 3]))
        exact -= 90 * Fraction(c)
        got = Fraction(lap(n, c))
        top = Fraction(2) ** int(np.floor(np.log2(max(abs(q) for q in x))))
        cut = 0 if spread == 0 else 192 * top / 2 ** 58
        assert abs(got - exact) <= cut + abs(exact) / 2 ** 53 * (1 + Fraction(1, 2 ** 40))


def test_special_values(lap):
    """Sums that cancel give exactly zero, zeros and subnormals beside normal
    values count as (almost) nothing, and the ends of the range are refused."""
    assert lap([3.0] * 12, 3.0) == 0.0
    assert lap([0.0] * 12, -2.0) == 180.0
    assert lap([5e-324] * 12, 1.0) == -90.0
    assert lap([-0.0, -5e-324] * 6, 1.0) == -90.0
    assert lap([0.0] * 12, 0.0) is None
    assert lap([1.0] * 12, float("nan")) is None
    assert lap([float("inf")] + [1.0] * 11, 1.0) is None
    assert lap([1e308] * 12, 1.0) is None
    assert lap([1e-290] * 12, 0.0) is None
