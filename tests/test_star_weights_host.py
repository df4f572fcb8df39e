"""The star sums of csrc/star_march.cuh (Laplacian and first differences of
orders 2 to 8, weighted in 64 or 96 bits) compiled for the host with g++ and
compared with exact rational sums."""
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
#include "star_march.cuh"
using namespace chemora;
// n[axis][k][+, -]; ns 0: Laplacian with centre c, else a sum of ns first differences
template <int R, int NS> static int star(const double* n, double c, double* out) {
  constexpr int N = 2 * R * (NS ? NS : 3), K = NS ? Guard<R>::d1 : Guard<R>::lap;
  fx::Parts p[N], pc = fx::parts_or_zero<K>(c);
  int e = NS ? fx::kZeroExp : pc.e;
  for (int q = 0; q < N; ++q) {
    p[q] = fx::parts_or_zero<K>(n[q]);
    e = fx::emax(e, p[q].e);
  }
  if (!star_ok<R>(e)) return 0;
  *out = 0.0;
  if (e == fx::kZeroExp) return 1;
  long long s[R] = {};
  for (int q = 0; q < N; ++q) s[q % (2 * R) / 2] += NS && (q & 1) ? -fx::align(p[q], e) : fx::align(p[q], e);
  if constexpr (NS == 0) *out = star_lap<R>(s, fx::align(pc, e), e);
  else *out = star_d1<R>(s, e);
  return 1;
}
template <int R> static int order(int ns, const double* n, double c, double* out) {
  return ns == 0 ? star<R, 0>(n, c, out) : (ns == 1 ? star<R, 1>(n, c, out) : star<R, 3>(n, c, out));
}
extern "C" int run(int R, int ns, const double* n, double c, double* out) {
  return R == 1 ? order<1>(ns, n, c, out) : R == 2 ? order<2>(ns, n, c, out)
       : R == 3 ? order<3>(ns, n, c, out) : order<4>(ns, n, c, out);
}
"""


@pytest.fixture(scope="module")
def star(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("star")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.run.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_double), ctypes.c_double,
                      ctypes.POINTER(ctypes.c_double)]

    def f(R, ns, n, c=0.0):
        o = ctypes.c_double()
        return o.value if L.run(R, ns, (ctypes.c_double * len(n))(*n), c, ctypes.byref(o)) else None
    return f


def _weights(R, ns):
    """Integer weights of the pairs at distance 1 .. R, from the closed form."""
    out = []
    for k in range(1, R + 1):
        w = Fraction(2 * (-1) ** (k + 1) * math.factorial(R) ** 2, math.factorial(R - k) * math.factorial(R + k))
        out.append(w / (2 * k) if ns else w / k ** 2)
    den = math.lcm(*[w.denominator for w in out])
    return [int(w * den) for w in out]


GUARD = {ns: {1: 6, 2: 4 if ns else 6, 3: 6, 4: 6} for ns in (0, 1, 3)}


@pytest.mark.parametrize("R", [1, 2, 3, 4])
@pytest.mark.parametrize("ns", [0, 1, 3])
@pytest.mark.parametrize("spread,rough", [(0, 1.0), (0, 1e-9), (0, 1e-15), (3, 1.0), (70, 1.0)])
def test_star_sums_against_rationals(star, R, ns, spread, rough):
    """Within half an ulp of the result, and of the values cut off below the
    guard bits: less than one unit of 2^(-52 - guard) of the largest value's
    binade per value, times its weight.  rough: differences between the
    values (1e-15: sums that cancel to a few units)."""
    w, rng = _weights(R, ns), np.random.default_rng(R * 100 + spread)
    naxes = ns or 3
    total = 2 * naxes * sum(abs(q) for q in w) + (abs(2 * naxes * sum(w)) if ns == 0 else 0)
    for _ in range(100):
        n = (1 + rough * rng.uniform(-1, 1, (naxes, R, 2))) * np.exp2(rng.uniform(-spread, 0, (naxes, R, 2)))
        if rough == 1.0:
            n *= rng.choice([-1.0, 1.0], n.shape)
        scale = 2.0 ** int(rng.integers(-300, 300))
        n, c = n * scale, float((1 + rough * rng.uniform(-1, 1)) * scale) if ns == 0 else 0.0
        exact = Fraction(0)
        for a in range(naxes):
            for k in range(R):
                p, m = Fraction(float(n[a, k, 0])), Fraction(float(n[a, k, 1]))
                exact += w[k] * (p - m if ns else p + m - 2 * Fraction(c))
        top = max(float(np.abs(n).max()), abs(c))
        unit = Fraction(2) ** (math.frexp(top)[1] - 1 - 52 - GUARD[ns][R])
        got = Fraction(star(R, ns, [float(q) for q in n.ravel()], c))
        cut = total * unit if spread or rough == 1.0 else 0
        assert abs(got - exact) <= cut + abs(exact) / 2 ** 53 * (1 + Fraction(1, 2 ** 20)), (got, exact)


@pytest.mark.parametrize("R", [1, 2, 3, 4])
def test_special_values(star, R):
    n3, n1 = 6 * R, 2 * R
    assert star(R, 0, [0.0, -0.0] * (n3 // 2), 0.0) == 0.0
    assert star(R, 0, [3.0] * n3, 3.0) == 0.0
    assert star(R, 0, [0.0] * n3, -1.0) == 6 * sum(_weights(R, 0))
    assert star(R, 1, [1.0, -0.0] * R) == sum(_weights(R, 1))
    assert star(R, 3, [5e-324] * n3) is None                # subnormals alone: left to FP64
    assert star(R, 1, [1.0, 5e-324] * R) == sum(_weights(R, 1))
    assert star(R, 1, [math.inf] + [1.0] * (n1 - 1)) is None
    assert star(R, 0, [1.0] * n3, math.nan) is None
    assert star(R, 0, [1.7e308] * n3, 0.0) is None
    big = 2.0 ** ((2030 if R <= 2 else 2020) - 1023)         # the largest exponent taken
    assert star(R, 0, [big] * n3, -big) == 12 * sum(_weights(R, 0)) * big
