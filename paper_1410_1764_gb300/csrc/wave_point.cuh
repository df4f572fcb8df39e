// Point bodies of the scalar-wave systems with their stencils on the integer
// units (fixedpoint.cuh): the Laplacian's 24 FP64 instructions per point (16
// with x lanes and a z queue sharing differences) become one multiply and
// about 200 integer operations, which run beside the FP64 update.  GB300, one
// RK4 step: 256^3 3.21 -> 1.20 ms (0.97 on planes in shared memory,
// wave_orders.cu); 61 x 75 x 53, launch-chained: 58.5 -> 25.1 us; 32^3, the
// same: 18.7 -> 12.0 us.  Bound by the integer pipes and the latency of its
// loads (HBM alone would take 0.63 ms at 256^3).
#pragma once
#include "device_types.cuh"
#include "star_march.cuh"
#include "generated/gen_wave.cuh"

namespace chemora {

// The 12 neighbours (u+1, u-1, u+2, u-2 along x, y, z) and the centre of the
// radius-2 star stencils.
struct Star2 {
  double c, n[12];
  template <class LD>
  CHEMORA_FX void load(const LD& ld) {
    c = ld(0, 0, 0, 0);
    n[0] = ld(0, 1, 0, 0);
    n[1] = ld(0, -1, 0, 0);
    n[2] = ld(0, 2, 0, 0);
    n[3] = ld(0, -2, 0, 0);
    n[4] = ld(0, 0, 1, 0);
    n[5] = ld(0, 0, -1, 0);
    n[6] = ld(0, 0, 2, 0);
    n[7] = ld(0, 0, -2, 0);
    n[8] = ld(0, 0, 0, 1);
    n[9] = ld(0, 0, 0, -1);
    n[10] = ld(0, 0, 0, 2);
    n[11] = ld(0, 0, 0, -2);
  }
  CHEMORA_FX bool zero() const {
    unsigned b = fx::hiword(c) << 1 | fx::loword(c);
#pragma unroll
    for (int q = 0; q < 12; ++q) b |= fx::hiword(n[q]) << 1 | fx::loword(n[q]);
    return b == 0;
  }
  CHEMORA_FX int exponent() const {
    int e = fx::exponent(c);
#pragma unroll
    for (int q = 0; q < 12; ++q) e = fx::emax(e, fx::exponent(n[q]));
    return e;
  }
};

// 12 h^2 times the order-4 Laplacian: 16 sum (u+-1) - sum (u+-2) - 90 u.
CHEMORA_FX double star2_lap(const Star2& s, int e) {
  constexpr int K = Guard<2>::lap;
  long long t[2] = {0, 0};
#pragma unroll
  for (int q = 0; q < 12; q += 4) {
    t[0] += fx::align<K>(s.n[q], e) + fx::align<K>(s.n[q + 1], e);
    t[1] += fx::align<K>(s.n[q + 2], e) + fx::align<K>(s.n[q + 3], e);
  }
  return star_lap<2>(t, fx::align<K>(s.c, e), e);
}

// Loader of a point whose star is at hand, for the FP64 body.
template <class LD>
struct StarLoader {
  const Star2& s;
  const LD& ld;
  CHEMORA_FX double operator()(int v, int dx, int dy, int dz) const {
    if (v != 0) return ld(v, dx, dy, dz);
    if (dx == 0 && dy == 0 && dz == 0) return s.c;
    const int a = dx != 0 ? 0 : (dy != 0 ? 4 : 8), m = dx + dy + dz;
    return s.n[a + (m == 1 ? 0 : (m == -1 ? 1 : (m == 2 ? 2 : 3)))];
  }
};

// The order-4 scalar wave: u_t = rho, rho_t = Lap u.
template <class LD, class OUT>
CHEMORA_FX void wave_point(const LD& ld, const Scalars& sc, OUT& out) {
  Star2 s;
  s.load(ld);
  const int e = s.exponent();
  if (fx::in_range(e)) {
    out(0, ld(1, 0, 0, 0));
    out(1, fma(star2_lap(s, e), sc.i12h2, sc.k[CHEMORA_K_MZERO]));
  } else if (s.zero()) {
    out(0, ld(1, 0, 0, 0));
    out(1, 0.0);
  } else {
    const StarLoader<LD> sl{s, ld};
    chemora_wave_point(sl, sc, out);
  }
}

}  // namespace chemora
