"""Accuracy of the integer stencils (csrc/star_march.cuh) against FP64: compiled
for the host with g++, each stencil's root mean square error against exact
rational sums, in ulps of its largest term (value times weight), is no larger than that of
the generated FP64 body of the same system (gen_wave*.cuh) on pulses narrow and
wide against the spacing, long waves, a small perturbation of one, and noise."""
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
#include <cmath>
#include <cstdint>
#define __device__
#define __host__
#define __forceinline__ inline
using std::fma;
#include "generated/gen_constants.cuh"
#include "generated/gen_wave.cuh"
#include "generated/gen_wave_o2.cuh"
#include "generated/gen_wave_o6.cuh"
#include "generated/gen_wave_o8.cuh"
#include "generated/gen_wave1_o2.cuh"
#include "generated/gen_wave1_o4.cuh"
#include "generated/gen_wave1_o6.cuh"
#include "generated/gen_wave1_o8.cuh"
#include "star_march.cuh"
using namespace chemora;

struct SC {
  double i12h = 1, i12h2 = 1, ih = 1, ih2 = 1, k[CHEMORA_NK];
  SC() { for (int i = 0; i < CHEMORA_NK; ++i) k[i] = kChemoraK[i]; }
};
// f[axis][k][+, -] and the centre, of every variable
struct LD {
  const double* f;
  double c;
  int R;
  double operator()(int v, int dx, int dy, int dz) const {
    const int o = dx + dy + dz, a = dx ? 0 : (dy ? 1 : 2), k = o < 0 ? -o : o;
    return o == 0 ? c : f[(a * R + k - 1) * 2 + (o < 0)];
  }
};
struct OUT {
  double* o;
  void operator()(int v, double x) const { o[v] = x; }
};

// out: Laplacian in FP64 and in integers, divergence of (f, f, f) likewise, D_a f likewise (x, y, z)
template <int R> static void star(const double* f, double c, double* out) {
  const SC sc;
  const LD ld{f, c, R};
  double o[5];
  const OUT w{o};
  if constexpr (R == 1) chemora_wave_o2_point(ld, sc, w);
  if constexpr (R == 2) chemora_wave_point(ld, sc, w);
  if constexpr (R == 3) chemora_wave_o6_point(ld, sc, w);
  if constexpr (R == 4) chemora_wave_o8_point(ld, sc, w);
  out[0] = o[1];
  if constexpr (R == 1) chemora_wave1_o2_point(ld, sc, w);
  if constexpr (R == 2) chemora_wave1_o4_point(ld, sc, w);
  if constexpr (R == 3) chemora_wave1_o6_point(ld, sc, w);
  if constexpr (R == 4) chemora_wave1_o8_point(ld, sc, w);
  out[2] = o[1];
  for (int a = 0; a < 3; ++a) out[4 + 2 * a] = o[2 + a];
  {
    constexpr int K = Guard<R>::lap;
    const fx::Parts pc = fx::parts_or_zero<K>(c);
    int en = pc.e, e = pc.e;
    for (int q = 0; q < 6 * R; ++q) {
      const int x = fx::parts_or_zero<K>(f[q]).e;
      if (is_near<R>(1 + q % (2 * R) / 2)) en = fx::emax(en, x);
      e = fx::emax(e, x);
    }
    long long s[R] = {};
    for (int q = 0; q < 6 * R; ++q) {
      const int k = q % (2 * R) / 2;
      s[k] += fx::align(fx::parts_or_zero<K>(f[q]), is_near<R>(k + 1) ? en : e);
    }
    out[1] = star_lap<R>(s, fx::align(pc, en), en, fx::align(pc, e), e) * (R == 2 ? 1.0 : 1.0 / Central<R>::den2);
  }
  constexpr int K = Guard<R>::d1;
  for (int a = -1; a < 3; ++a) {
    const int q0 = a < 0 ? 0 : 2 * R * a, q1 = a < 0 ? 6 * R : q0 + 2 * R;
    int en = fx::kZeroExp, e = fx::kZeroExp;
    for (int q = q0; q < q1; ++q) {
      const int x = fx::parts_or_zero<K>(f[q]).e;
      if (is_near<R>(1 + q % (2 * R) / 2)) en = fx::emax(en, x);
      e = fx::emax(e, x);
    }
    long long t[R] = {};
    for (int q = q0; q < q1; ++q) {
      const int k = q % (2 * R) / 2;
      const long long m = fx::align(fx::parts_or_zero<K>(f[q]), is_near<R>(k + 1) ? en : e);
      t[k] += q & 1 ? -m : m;
    }
    out[5 + 2 * a] = star_d1<R>(t, en, e) * (1.0 / Central<R>::den1);
  }
}
// order-4 first differences with an axis of its own exponent (the variable-speed wave's): FP64 and integers, over 12 h
extern "C" void axes(const double* f, double* out) {
  constexpr int K = 5;
  for (int a = 0; a < 3; ++a) {
    const double p1 = f[4 * a], m1 = f[4 * a + 1], p2 = f[4 * a + 2], m2 = f[4 * a + 3];
    out[2 * a] = fma(8.0, p1 - m1, -(p2 - m2));
    const double v[4] = {m2, m1, p1, p2};
    long long m[4];
    int x[4], e = fx::kZeroExp;
    for (int q = 0; q < 4; ++q) {
      m[q] = fx::parts_or_zero<K>(v[q]).m;
      x[q] = fx::parts_or_zero<K>(v[q]).e;
      e = fx::emax(e, x[q]);
    }
    out[2 * a + 1] = fx::to_double<K>(Axis4(m, x, e).diff, e);
  }
}
extern "C" void run(int R, const double* f, double c, double* out) {
  R == 1 ? star<1>(f, c, out) : R == 2 ? star<2>(f, c, out) : R == 3 ? star<3>(f, c, out) : star<4>(f, c, out);
}
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("precision")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    return ctypes.CDLL(str(so))


def _weights(R, first):
    out = []
    for k in range(1, R + 1):
        w = Fraction(2 * (-1) ** (k + 1) * math.factorial(R) ** 2, math.factorial(R - k) * math.factorial(R + k))
        out.append(w / (2 * k) if first else w / k ** 2)
    return out


def stars(field, R, count, rng):
    """Values f[axis][k][+, -] and centre of `count` stars."""
    off = np.zeros((3, R, 2, 3))
    for a in range(3):
        for k in range(R):
            off[a, k, 0, a], off[a, k, 1, a] = k + 1, -k - 1
    off = np.concatenate([off.reshape(-1, 3), np.zeros((1, 3))])
    for _ in range(count):
        if field == "noise":
            v = rng.standard_normal(len(off))
        elif field.startswith("pulse"):
            r = off / float(field.split("/")[1]) + rng.uniform(-0.5, 0.5, 3)
            v = np.exp(-0.5 * ((r - np.round(r)) / 0.05) ** 2).prod(1)
        else:
            k, ph, am = rng.integers(-2, 3, (3, 3)), rng.uniform(0, 1, 3), rng.standard_normal(3)
            v = np.sin(2 * np.pi * (off @ k.T / 64 + ph)) @ am
            v = 1 + 1e-2 * v if field == "flat" else v
        yield [float(q) for q in v[:-1]], float(v[-1])


def ulp(v):
    return 2.0 ** (math.frexp(v)[1] - 53)


FIELDS = ["pulse/16", "pulse/32", "pulse/128", "wave", "flat", "noise"]


@pytest.mark.parametrize("R", [1, 2, 3, 4])
@pytest.mark.parametrize("field", FIELDS)
def test_no_further_from_exact_than_fp64(L, R, field):
    w2, w1 = _weights(R, False), _weights(R, True)
    if R == 2:
        w2 = [12 * w for w in w2]  # the order-4 Laplacian is formed over 12 h^2
    err = np.zeros((400, 5, 3))  # FP64, integers, half an ulp of the result
    for i, (f, c) in enumerate(stars(field, R, len(err), np.random.default_rng(R))):
        out = (ctypes.c_double * 10)()
        L.run(R, (ctypes.c_double * len(f))(*f), ctypes.c_double(c), out)
        F = np.array([Fraction(q) for q in f], dtype=object).reshape(3, R, 2)
        d1 = [sum(w * (F[a, k, 0] - F[a, k, 1]) for k, w in enumerate(w1)) for a in range(3)]
        lap = sum(w * (F[a, k, 0] + F[a, k, 1] - 2 * Fraction(c)) for a in range(3) for k, w in enumerate(w2))
        v = np.abs(np.array(f)).reshape(3, R, 2).max(2)  # per axis and distance
        t1 = (v * np.abs(np.array(w1, float))).max(1)
        tops = [max((v * np.abs(np.array(w2, float))).max(), abs(6 * c * float(sum(w2)))), t1.max()] + list(t1)
        for q, (exact, top) in enumerate(zip([lap, sum(d1)] + d1, tops)):
            err[i, q, 2] = ulp(float(exact)) / ulp(top) / 2
            for m in range(2):
                err[i, q, m] = float((Fraction(out[2 * q + m]) - exact) / Fraction(ulp(top)))
    sq = (err ** 2).mean(0)
    rms = np.sqrt(np.stack([sq[0], sq[1], sq[2:].mean(0)]))  # the Laplacian, the divergence, the first differences
    # 2 %: sampling (order 2's first differences are the same in both); orders 6 and 8 scale by a rounded constant
    assert (rms[:, 1] ** 2 <= (rms[:, 0] * 1.02) ** 2 + (rms[:, 2] ** 2 if R >= 3 else 0)).all(), rms


@pytest.mark.parametrize("R", [3, 4])
@pytest.mark.parametrize("shift", [0, 5, 20, 31, 32, 40, 63, 64, 95, 96, 130, 600, -5, -40])
def test_far_values(L, R, shift):
    """Values at distance 3 and 4 a power of two larger (or smaller) than the
    near ones, and near ones that are all zero: within half an ulp of the result,
    a unit of the far values' 2^-58 for the near sum, and the cut of each group's
    values below its own largest exponent."""
    w2, w1 = _weights(R, False), _weights(R, True)
    rng = np.random.default_rng(shift + 1000)
    for trial in range(60):
        v = rng.uniform(-1, 1, (3, R, 2))
        v[:, 2:] *= 2.0 ** shift
        c = float(rng.uniform(-1, 1))
        if trial % 6 == 0:
            v[:, :2], c = 0.0, 0.0
        f = [float(q) for q in v.ravel()]
        out = (ctypes.c_double * 10)()
        L.run(R, (ctypes.c_double * len(f))(*f), ctypes.c_double(c), out)
        F = np.array([Fraction(q) for q in f], dtype=object).reshape(3, R, 2)
        for name, got, exact, w, centre in (
                ("lap", out[1], sum(w * (F[a, k, 0] + F[a, k, 1] - 2 * Fraction(c)) for a in range(3)
                                    for k, w in enumerate(w2)), w2, c),
                ("div", out[3], sum(w * (F[a, k, 0] - F[a, k, 1]) for a in range(3) for k, w in enumerate(w1)), w1, 0.0)):
            near = max(float(np.abs(v[:, :2]).max()), abs(centre))
            top = max(near, float(np.abs(v[:, 2:]).max()))
            cut = sum(6 * 2 * abs(q) * Fraction(ulp(near)) for q in w[:2]) if near else 0
            cut += sum(6 * 2 * abs(q) * Fraction(ulp(top)) for q in w[2:]) + Fraction(ulp(top)) / 100
            # three roundings: the sum, one over the weights' denominator, and their product
            assert abs(Fraction(got) - exact) <= cut / 32 + abs(exact) * 3 / 2 ** 53 * (1 + Fraction(1, 2 ** 20)), (name, trial)


@pytest.mark.parametrize("field", FIELDS)
def test_axis_differences(L, field):
    """Relative to the largest value of the axis itself."""
    err = []
    for f, _ in stars(field, 2, 400, np.random.default_rng(7)):
        out = (ctypes.c_double * 6)()
        L.axes((ctypes.c_double * 12)(*f), out)
        for a in range(3):
            p1, m1, p2, m2 = (Fraction(q) for q in f[4 * a:4 * a + 4])
            exact, top = 8 * (p1 - m1) - (p2 - m2), ulp(max(map(abs, f[4 * a:4 * a + 4])))
            err.append([float(Fraction(out[2 * a + m]) - exact) / top for m in range(2)])
    rms = np.sqrt((np.array(err) ** 2).mean(0))
    assert rms[1] <= rms[0], rms


def test_order2_differences_round_as_fp64(L):
    """A difference of two doubles within six binades, correctly rounded with
    ties to even: the same bits as FP64 (differences are often ties)."""
    rng = np.random.default_rng(9)
    ties = 0
    for _ in range(500):
        f = rng.uniform(0.25, 1.0, 6) * rng.choice([-1.0, 1.0, 8.0], 6)
        out = (ctypes.c_double * 10)()
        L.run(1, (ctypes.c_double * 6)(*f), ctypes.c_double(0.5), out)
        assert out[4:10:2] == out[5:10:2]
        for a in range(3):
            d = Fraction(f[2 * a]) - Fraction(f[2 * a + 1])
            ties += 2 * abs(d - Fraction(float(d))) == Fraction(ulp(float(d)))
    assert ties > 100
