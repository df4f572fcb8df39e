// Star stencils on the integer units (fixedpoint.cuh), a tile of columns at a
// time: a block of TX x TY threads marches through z, a point per thread and
// plane.  A value is taken apart into significand and exponent once: a thread
// keeps its column's 2R + 1 values in registers, the plane in hand lies in
// shared memory with its halo, and a tap is a shift to the largest exponent
// and an addition.
#pragma once
#include "fixedpoint.cuh"
#if defined(__CUDACC__)
#include "device_types.cuh"
#endif

namespace chemora {

// Weights of the centred differences of order 2R as integers.  kD2: pairs
// f(+k) + f(-k) - 2 f of the second difference, over kDen2 h^2; kD1: pairs
// f(+k) - f(-k) of the first, over kDen1 h.
template <int R>
struct Central;
template <>
struct Central<1> {
  static constexpr int d2[4] = {1, 0, 0, 0}, den2 = 1, d1[4] = {1, 0, 0, 0}, den1 = 2;
};
template <>
struct Central<2> {
  static constexpr int d2[4] = {16, -1, 0, 0}, den2 = 12, d1[4] = {8, -1, 0, 0}, den1 = 12;
};
template <>
struct Central<3> {
  static constexpr int d2[4] = {270, -27, 2, 0}, den2 = 180, d1[4] = {45, -9, 1, 0}, den1 = 60;
};
template <>
struct Central<4> {
  static constexpr int d2[4] = {8064, -1008, 128, -9}, den2 = 5040, d1[4] = {672, -168, 32, -3}, den1 = 840;
};

// Guard bits: with six, sums of twelve values fit in 64 bits, and the weighted
// sums of such sums take up to 96; with four, the order-4 first differences
// (weights 54 in all over three axes) stay in 64.  Root mean square errors
// against exact sums, in ulps of the star's largest value, over pulses of width
// 0.05 at 1/32 to 1/256 spacing, long waves and noise: order-4 Laplacian 0.02 to
// 16, FP64 chain 0.6 to 27 (with two guard bits 0.6 to 17, and 2 to 6 times the
// FP64 chain's on the pulses); order-4 first differences and their sums 0.06 to
// 0.5, FP64 0.09 to 0.7; the other orders no larger than FP64's either.
template <int R>
struct Guard {
  static constexpr int lap = 6, d1 = R == 2 ? 4 : 6;
};

// Exponents from which no weighted sum (orders 6 and 8: below 2^18 times the
// largest value) can leave the FP64 range.
template <int R>
CHEMORA_FX bool star_ok(int e) {
  constexpr int top = R <= 2 ? fx::kExpMax : 2020;
  return e == fx::kZeroExp || (unsigned)(e - fx::kExpMin) <= (unsigned)(top - fx::kExpMin);
}

// Values at distance 3 and 4 have weights 2^-7 and 2^-10 of the nearest ones'.
// Those of distance 1 and 2 and the centre are aligned to their own largest
// exponent, so that larger values far away do not cut them (order 8 on 33 x 40 x
// 35, pulses: with one exponent for all, 12 times FP64's error where the right-hand
// side is small).
template <int R>
constexpr bool is_near(int offset) {
  return R <= 2 || (offset >= -2 && offset <= 2);
}

// den2 h^2 times the Laplacian from the sums s[k] of the six values at
// distance k + 1 and the centre: those near and cn aligned to exponent en, the
// others and cf to e >= en.
template <int R, int K = Guard<R>::lap>
CHEMORA_FX double star_lap(const long long (&s)[R], long long cn, int en, long long cf, int e) {
  typedef Central<R> W;
  if constexpr (R == 1) {
    return fx::to_double<K>(s[0] - 6 * cn, en);
  } else if constexpr (R == 2) {
    // 16 s1 - s2 - 90 c = 16 h - r, 0 <= r < 16: 68 bits, of which the low four
    // matter only where h is small.  Every part is at most 2^(57 + K) = 2^63.
    const long long b = s[1] + 10 * cn, h = s[0] - 5 * cn - (b >> 4);
    const bool wide = (unsigned long long)(h + (1ll << 57)) >> 58 != 0;
    return fx::to_double<K>(wide ? h : 16 * h - (b & 15), wide ? en + 4 : en);
  } else {
    fx::Sum96 v;
    v.add<W::d2[0]>(s[0] - 6 * cn);
    v.add<W::d2[1]>(s[1] - 6 * cn);
    v.shift((unsigned)(e - en));
    v.add<W::d2[2]>(s[R < 3 ? 0 : 2] - 6 * cf);
    if constexpr (R == 4) v.add<W::d2[3]>(s[R - 1] - 6 * cf);
    return fx::to_double<K>(v, e);
  }
}
template <int R, int K = Guard<R>::lap>
CHEMORA_FX double star_lap(const long long (&s)[R], long long c, int e) {
  return star_lap<R, K>(s, c, e, c, e);
}

// den1 h times a sum of up to three first differences from the sums t[k] of their
// differences f(k + 1) - f(-k - 1), the near ones aligned to exponent en, the
// others to e >= en.
template <int R>
CHEMORA_FX double star_d1(const long long (&t)[R], int en, int e) {
  typedef Central<R> W;
  constexpr int K = Guard<R>::d1;
  if constexpr (R == 1) {
    return fx::to_double<K, true>(t[0], en);
  } else if constexpr (R == 2) {
    return fx::to_double<K>(8 * t[0] - t[1], en);
  } else {
    fx::Sum96 v;
    v.add<W::d1[0]>(t[0]);
    v.add<W::d1[1]>(t[1]);
    v.shift((unsigned)(e - en));
    v.add<W::d1[2]>(t[2]);
    if constexpr (R == 4) v.add<W::d1[3]>(t[R - 1]);
    return fx::to_double<K>(v, e);
  }
}
template <int R>
CHEMORA_FX double star_d1(const long long (&t)[R], int e) {
  return star_d1<R>(t, e, e);
}

// One axis of an order-4 star from its values' significands and exponents at
// offsets -2, -1, 1, 2, aligned to the largest exponent e of the four, so that a
// first difference is as close as in FP64 however large the values along the
// other axes are.
struct Axis4 {
  long long near, far;  // sums of the pairs at distance 1 and 2
  long long diff;       // 12 h D f: 8 (f(+1) - f(-1)) - (f(+2) - f(-2)), at most 18 2^(53 + K)
  CHEMORA_FX Axis4(const long long (&m)[4], const int (&x)[4], int e) {
    const long long a = fx::sar(m[0], (unsigned)(e - x[0])), b = fx::sar(m[1], (unsigned)(e - x[1]));
    const long long c = fx::sar(m[2], (unsigned)(e - x[2])), d = fx::sar(m[3], (unsigned)(e - x[3]));
    near = c + b;
    far = d + a;
    diff = 8 * (c - b) - (d - a);
  }
};

// Offset m of 2R taken in the order -R .. -1, 1 .. R.
template <int R>
CHEMORA_FX constexpr int tap(int m) { return m < R ? m - R : m - R + 1; }

#if defined(__CUDACC__)

// A thread's place in a march: tile TX x TY at (x0, y0), planes k0 .. k0 + nz - 1.
template <int TX, int TY>
struct MarchPlace {
  int x0, y0, k0, w, h, nz, lx, ly;
  bool active;
  int64_t org;  // the tile's first point in the padded layout
  __device__ __forceinline__ MarchPlace(const Dims& d, int zb) {
    x0 = blockIdx.x * TX;
    y0 = blockIdx.y * TY;
    k0 = blockIdx.z * zb;
    w = min(TX, d.nx - x0);
    h = min(TY, d.ny - y0);
    nz = min(zb, d.nz - k0);
    lx = threadIdx.x % TX;
    ly = threadIdx.x / TX;
    active = lx < w && ly < h;
    org = (int64_t)(k0 + d.g) * d.sz + (int64_t)(y0 + d.g) * d.sy + (x0 + d.g);
  }
};

// The halo cells a thread fetches: columns -R .. -1, w .. w + R - 1 of the
// tile's rows (along x), then rows -R .. -1, h .. h + R - 1 (along y).
template <int R, int TX, int TY>
struct MarchHalo {
  static constexpr int n = (2 * R * (TX + TY) + TX * TY - 1) / (TX * TY);
  int x[n], y[n];
  bool live[n], along_x[n];
  __device__ __forceinline__ MarchHalo(const MarchPlace<TX, TY>& p) {
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const int q = threadIdx.x + i * TX * TY;
      along_x[i] = q < 2 * R * p.h;
      live[i] = q < 2 * R * (p.w + p.h);
      x[i] = y[i] = 0;
      if (along_x[i]) {
        const int e = q / p.h;
        y[i] = q - e * p.h;
        x[i] = e < R ? e - R : p.w + e - R;
      } else if (live[i]) {
        const int e = (q - 2 * R * p.h) / p.w;
        x[i] = q - 2 * R * p.h - e * p.w;
        y[i] = e < R ? e - R : p.h + e - R;
      }
    }
  }
};

// The update of the wave systems (StageOutFma, same operations) with y_n and
// the accumulator loaded ahead.
template <int NV>
struct MarchUpdate {
  double yn[NV], acc[NV];
  __device__ __forceinline__ void load(const StageParams& a, int64_t c, int64_t sv) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      yn[v] = a.mode >= 1 ? a.yn[c + v * sv] : 0.0;
      acc[v] = a.mode >= 2 ? a.acc[c + v * sv] : 0.0;
    }
  }
  // A branch per mode around the stores: as selects the updates of all modes
  // would be evaluated (9 instead of 5 FP64 instructions for two variables).
  template <class ST>
  __device__ __forceinline__ void apply(const StageParams& a, int64_t c, int64_t sv, const double (&k)[NV], double one,
                                        double two, const ST& store) const {
    if (a.mode == 2 || a.mode == 3) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        a.acc[c + v * sv] = __fma_rn(two, k[v], acc[v]);
        store(c + v * sv, __fma_rn(a.c2, k[v], yn[v]));
      }
    } else if (a.mode == 1) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        a.acc[c + v * sv] = k[v];
        store(c + v * sv, __fma_rn(a.c2, k[v], yn[v]));
      }
    } else if (a.mode == 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) store(c + v * sv, k[v]);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) store(c + v * sv, __fma_rn(a.c1, __fma_rn(acc[v], one, k[v]), yn[v]));
    }
  }
};

// Planes a block marches through.  An SM (of 152) works through the planes of
// its blocks, a block's start costing about one and a half, and drains over
// about three quarters of its resident blocks.  us per stage at depths 4, 8, 16
// and 32: variable speed, 128^3 58, 60, 69, 70; order 4, 256^3 264, 253, 249,
// 256; first-order form of order 6, 117 x 90 x 131 92, 97, 114, 115.
inline int march_depth(const Dims& d, int tx, int ty, int resident) {
  const int64_t tiles = (int64_t)((d.nx + tx - 1) / tx) * ((d.ny + ty - 1) / ty);
  int best = 1;
  double cost = 1e300;
  for (int zb = 1; zb <= 64 && zb <= d.nz; ++zb) {
    const int64_t blocks = tiles * ((d.nz + zb - 1) / zb);
    const int64_t per_sm = (blocks + 151) / 152;
    const double c = ((double)per_sm + 0.75 * resident) * (zb + 1.5);
    if (c < cost) {
      cost = c;
      best = zb;
    }
  }
  const int seg = (d.nz + best - 1) / best;
  return (d.nz + seg - 1) / seg;
}

inline dim3 march_grid(const Dims& d, int tx, int ty, int zb) {
  return dim3((d.nx + tx - 1) / tx, (d.ny + ty - 1) / ty, (d.nz + zb - 1) / zb);
}

#endif

}  // namespace chemora
