// Sums of products of the BSSN algebra on the integer units.
//
// The algebra kernels are bound by FP64 issue, 16 cycles of the SM's pipe per
// warp instruction, and use little else.  Advection and dissipation of every
// variable, gt_ij's whole right-hand side, At_ij's terms in the shift and the
// traces gt^ab D_ab f are sums of products, 272 of the 1058 FP64 operations;
// on the integer units, which run beside the FP64 pipe, such a sum is closer than
// an FP64 chain (bounds and errors at fx::dot) and rounded once.  They are loops over
// variables, not straight code, to keep the kernel in the instruction cache,
// with the next variable's fields fetched an iteration ahead; results pass to
// the generated body through the thread's column in shared memory.  Values
// whose exponents leave the range are summed in FP64.
//
// GB300, algebra of 128^3 points, four blocks of 128 per SM: 4.3 ms (three
// blocks, the best without this) -> 3.6.  Without the fetch ahead 3.8.  A term
// is 35 to 55 integer instructions, so more of it does not pay: with At^ij,
// At_ij At^ij and phi's, K's and the gauge's other terms here too (374
// operations) 3.9, with advection, dissipation and traces alone (186) 3.9.
#pragma once
#include "bssn_fields.cuh"

namespace chemora {

// index of the symmetric pair (i, j) among xx, xy, xz, yy, yz, zz, and back
__device__ __forceinline__ int sym_index(int i, int j) {
  const int a = min(i, j), b = max(i, j);
  return a * (5 - a) / 2 + b;
}
__device__ __forceinline__ int sym_row(int c) { return c < 3 ? 0 : (c < 5 ? 1 : 2); }
__device__ __forceinline__ int sym_col(int c) { return c < 3 ? c : (c < 5 ? c - 2 : 2); }

// sum_q a[q] b[q]
template <int N>
__device__ __forceinline__ double dot_terms(const fx::Parts (&p)[N], const double (&a)[N], const double (&b)[N],
                                            double mzero) {
  double s;
  if (!fx::dot(p, &s)) {
    s = mzero;
#pragma unroll
    for (int q = 0; q < N; ++q) s = fma(a[q], b[q], s);
  }
  return s;
}
// Inverse conformal metric.
template <int BLK, class SC>
__device__ __forceinline__ void bssn_inverse_metric(const FieldLoader<BLK>& ld, const SC& sc) {
  const double mz = sc.k[CHEMORA_K_MZERO];
  auto mul = [&](double a, double b) { return fma(a, b, mz); };
  double g[6], c[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) g[q] = ld(1 + q, 0, 0, 0);
  c[0] = fma(-g[4], g[4], mul(g[3], g[5]));
  c[1] = fma(-g[1], g[5], mul(g[2], g[4]));
  c[2] = fma(-g[2], g[3], mul(g[1], g[4]));
  c[3] = fma(-g[2], g[2], mul(g[0], g[5]));
  c[4] = fma(-g[0], g[4], mul(g[1], g[2]));
  c[5] = fma(-g[1], g[1], mul(g[0], g[3]));
  const double idet = 1.0 / fma(g[2], c[2], fma(g[1], c[1], mul(g[0], c[0])));
#pragma unroll
  for (int q = 0; q < 6; ++q) ld.s[(kPreGu + q) * BLK] = mul(c[q], idet);
}

// The traces gt^ab D_ab f of gt_ij, alpha and beta^i.
template <int BLK, class SC>
__device__ __forceinline__ void bssn_traces(const FieldLoader<BLK>& ld, const SC& sc) {
  const double mz = sc.k[CHEMORA_K_MZERO];
  auto mul = [&](double a, double b) { return fma(a, b, mz); };
  double next[6];
  auto fetch = [&](int t) {  // an iteration ahead
    const int v = t < 6 ? t + 1 : t + 11;
    next[0] = ld.g2(v, 0);
    next[1] = ld.g11(v, 0);
    next[2] = ld.g11(v, 1);
    next[3] = ld.g2(v, 1);
    next[4] = ld.g11(v, 2);
    next[5] = ld.g2(v, 2);
  };
  fetch(0);
  const double two_i144h2 = mul(sc.i144h2, sc.k[CHEMORA_K_TWO]);
  double u[6];  // weights of the raw differences
  fx::Term<10> f[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    u[q] = mul(ld.gu(q), q == 0 || q == 3 || q == 5 ? sc.i12h2 : two_i144h2);
    f[q] = fx::term<10>(u[q]);
  }
  constexpr int K = fx::DotGuard<6>::k;
#pragma unroll 1
  for (int t = 0; t < 10; ++t) {
    double d[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) d[q] = next[q];
    if (t < 9) fetch(t + 1);
    fx::Parts p[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) p[q] = fx::term_product<K>(f[q], fx::term<K + 1>(d[q]));
    ld.s[(kPreTr + t) * BLK] = dot_terms(p, u, d, mz);
  }
}

// The inverse metric, the shift's derivatives, advection and dissipation of
// every variable; gt_ij's right-hand side, given to out; At_ij's terms in the
// shift.
template <int BLK, class SC, class OUT>
__device__ __forceinline__ void bssn_shift_terms(const FieldLoader<BLK>& ld, const SC& sc, OUT& out) {
  const double mz = sc.k[CHEMORA_K_MZERO], one = sc.k[CHEMORA_K_ONE];
  auto mul = [&](double a, double b) { return fma(a, b, mz); };
  double next[4];
  auto fetch = [&](int v) {  // an iteration ahead
    next[0] = ld.g1(v, 0);
    next[1] = ld.g1(v, 1);
    next[2] = ld.g1(v, 2);
    next[3] = ld.gko(v);
  };
  fetch(0);
  double w[4];  // weights of the raw differences
  fx::Term<10> fw[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    w[a] = a < 3 ? mul(sc.i12h, ld(18 + a, 0, 0, 0)) : sc.ko_scale;
    fw[a] = fx::term<10>(w[a]);
  }
  double div = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double d = mul(sc.i12h, ld.g1(18 + i, a));
      ld.s[(kPreDb + 3 * i + a) * BLK] = d;
      if (i == a) div = i == 0 ? d : fma(d, one, div);
    }
  const double al = ld(17, 0, 0, 0), trK = ld(7, 0, 0, 0);
  bssn_inverse_metric(ld, sc);
  const double al2 = mul(ld(17, 0, 0, 0), -sc.k[CHEMORA_K_TWO]);
  {
    constexpr int K = fx::DotGuard<4>::k;
#pragma unroll 1
    for (int t = 0; t < 12; ++t) {  // phi, K, Xt^i, alpha, beta^i, B^i
      const int v = t == 0 ? 0 : (t == 1 ? 7 : t + 12);
      double b[4];
      fx::Parts p[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = next[q];
      fetch(t == 11 ? 1 : (t == 0 ? 7 : t + 13));  // then gt_xx
#pragma unroll
      for (int q = 0; q < 4; ++q) p[q] = fx::term_product<K>(fw[q], fx::term<K + 1>(b[q]));
      ld.s[adv_index(v) * BLK] = dot_terms(p, w, b, mz);
    }
  }
  const double div23 = mul(div, -2.0 / 3.0);
  const fx::Term<10> fd = fx::term<10>(div23), fal = fx::term<10>(al2), fz = fx::term<10>(0.0);
  constexpr int K = fx::DotGuard<12>::k;
#pragma unroll 1
  for (int t = 0; t < 12; ++t) {  // gt_ij, At_ij
    const bool gt = t < 6;
    const int c = gt ? t : t - 6, base = gt ? 1 : 8, i = sym_row(c), j = sym_col(c);
    double a[12], b[12];
    fx::Parts p[12];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      a[q] = w[q];
      b[q] = next[q];
    }
    if (t < 11) fetch(t < 5 ? t + 2 : t + 3);
#pragma unroll
    for (int q = 0; q < 4; ++q) p[q] = fx::term_product<K>(fw[q], fx::term<K + 1>(b[q]));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[4 + 2 * k] = ld(base + sym_index(i, k), 0, 0, 0);
      b[4 + 2 * k] = ld.db(k, j);
      a[5 + 2 * k] = ld(base + sym_index(j, k), 0, 0, 0);
      b[5 + 2 * k] = ld.db(k, i);
    }
#pragma unroll
    for (int q = 4; q < 10; ++q) p[q] = fx::term_product<K>(fx::term<10>(a[q]), fx::term<K + 1>(b[q]));
    a[10] = div23;
    b[10] = ld(base + c, 0, 0, 0);
    p[10] = fx::term_product<K>(fd, fx::term<K + 1>(b[10]));
    a[11] = gt ? al2 : 0.0;
    b[11] = ld(8 + c, 0, 0, 0);
    p[11] = fx::term_product<K>(gt ? fal : fz, fx::term<K + 1>(b[11]));
    const double s = dot_terms(p, a, b, mz);
    if (gt)
      out(1 + c, s);
    else
      ld.s[adv_index(8 + c) * BLK] = s;
  }
}

}  // namespace chemora
