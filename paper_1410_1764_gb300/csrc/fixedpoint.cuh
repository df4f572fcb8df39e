// Finite-difference stencils on the integer units.
//
// On GB300 an FP64 fma occupies the SM's FP64 pipe for 17-19 cycles per warp
// (1.7-1.9 fmas per clock per SM, measured), a 32-bit integer operation for
// 0.4-0.8, on pipes that run beside it (measured: twelve integer operations
// per fma, or a load, do not slow a saturated fma stream).  A stencil is a
// sum of values times small integers, so it is evaluated in integers: the
// values it reads are written as multiples of one power of two, taken from
// the largest of them (align), added exactly in 64 bits, and the sum is
// rounded once to a double (to_double).  With K guard bits every value down
// to 2^-K of the largest is represented exactly and a smaller one is
// rounded down at 2^(-52-K) of the largest value's power of two.  Which values
// share an exponent, and K, are chosen so that root mean square errors against
// exact sums are no larger than an FP64 chain's (star_march.cuh; measured for
// every stencil on pulses, waves and noise).  A result depends on the values
// alone, not on the order of the sum or on the launch shape that evaluates it.
//
// A set of values whose largest exponent lies outside [128, 2030] (zeros,
// numbers near the ends of the FP64 range, Inf, NaN) is left to the caller's
// FP64 body (in_range).  Compiles for the host too (tests).
#pragma once
#if !defined(__CUDACC_RTC__)
#include <stdint.h>
#endif
#if !defined(__CUDACC__)
#include <string.h>
#endif

namespace chemora {
namespace fx {

#if defined(__CUDACC__)
#define CHEMORA_FX __device__ __forceinline__
CHEMORA_FX unsigned hiword(double v) { return (unsigned)__double2hiint(v); }
CHEMORA_FX unsigned loword(double v) { return (unsigned)__double2loint(v); }
CHEMORA_FX double from_bits(unsigned long long b) { return __longlong_as_double((long long)b); }
// PTX shifts clamp: an amount of 64 or more gives 0 (or the sign)
CHEMORA_FX unsigned long long shl(unsigned long long a, unsigned s) {
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
}
CHEMORA_FX long long sar(long long a, unsigned s) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
}
CHEMORA_FX unsigned long long shr(unsigned long long a, unsigned s) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(s));
  return r;
}
CHEMORA_FX int clz64(unsigned long long a) { return __clzll((long long)a); }
CHEMORA_FX int mulhi32(int a, int b) { return __mulhi(a, b); }
CHEMORA_FX long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
#else
#define CHEMORA_FX inline
CHEMORA_FX unsigned long long bits(double v) {
  unsigned long long b;
  memcpy(&b, &v, 8);
  return b;
}
CHEMORA_FX unsigned hiword(double v) { return (unsigned)(bits(v) >> 32); }
CHEMORA_FX unsigned loword(double v) { return (unsigned)bits(v); }
CHEMORA_FX double from_bits(unsigned long long b) {
  double v;
  memcpy(&v, &b, 8);
  return v;
}
CHEMORA_FX unsigned long long shl(unsigned long long a, unsigned s) { return s > 63 ? 0 : a << s; }
CHEMORA_FX long long sar(long long a, unsigned s) { return a >> (s > 63 ? 63 : s); }
CHEMORA_FX unsigned long long shr(unsigned long long a, unsigned s) { return s > 63 ? 0 : a >> s; }
CHEMORA_FX int clz64(unsigned long long a) { return a ? __builtin_clzll(a) : 64; }
CHEMORA_FX int mulhi32(int a, int b) { return (int)((long long)a * b >> 32); }
CHEMORA_FX long long mad_wide(int a, int b, long long c) { return (long long)a * b + c; }
#endif

constexpr int kExpMin = 128, kExpMax = 2030;
CHEMORA_FX bool in_range(int e) { return (unsigned)(e - kExpMin) <= (unsigned)(kExpMax - kExpMin); }
CHEMORA_FX int exponent(double v) { return (int)(hiword(v) >> 20) & 0x7ff; }
CHEMORA_FX int emax(int a, int b) { return a > b ? a : b; }

// A double taken apart: its exponent field e and its signed significand in
// units of 2^(e - 1075 - K).  Zeros and subnormals have e = 0 and a small
// non-negative m, which every shift to an exponent in range removes.
struct Parts {
  long long m;
  int e;
};
template <int K>
CHEMORA_FX Parts parts(double v) {
  const unsigned h = hiword(v);
  const unsigned long long m = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32 | loword(v)) << K;
  const unsigned long long s = h >= 0x80100000u ? ~0ull : 0ull;
  return Parts{(long long)((m ^ s) - s), exponent(v)};
}

// The same, with the exponent of zeros far below every other: a set of values
// whose largest exponent is kZeroExp is all zeros.
constexpr int kZeroExp = -4096;
template <int K>
CHEMORA_FX Parts parts_or_zero(double v) {
  Parts p = parts<K>(v);
  if (((hiword(v) << 1) | loword(v)) == 0) p.e = kZeroExp;
  return p;
}

// A factor of a product: its signed significand 2^S times, as the high word and
// 31 bits of the low word, and its exponent (very low for zero, very high for
// subnormals, Inf and NaN, so that the products are zero and out of every
// range).
template <int S>
struct Term {
  int hi, lo;
  int e;
};
template <int S>
CHEMORA_FX Term<S> term(double v) {
  const unsigned h = hiword(v);
  unsigned long long m = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32 | loword(v)) << S;
  const unsigned long long s = (unsigned long long)(long long)((int)h >> 31);
  m = (m ^ s) - s;
  int e = exponent(v);
  if ((unsigned)(e - 1) >= 2046u) e = ((h << 1) | loword(v)) == 0 ? -8192 : 16384;
  return Term<S>{(int)(m >> 32), (int)((unsigned)m >> 1), e};
}
// a b in units of 2^(e - 1075 - K) in four multiplications: the product of the low
// words is left out, two halved low words and the high halves of two products are
// cut, in all less than six units, of which two are added back (the mean).
template <int K>
CHEMORA_FX Parts term_product(const Term<10>& a, const Term<K + 1>& b) {
  const int x = mulhi32(a.hi, b.lo) + mulhi32(a.lo, b.hi);
  return Parts{mad_wide(x, 2, mad_wide(a.hi, b.hi, 2)), emax(a.e + b.e - 1022, kZeroExp)};
}
// The sum of N products as a double, at the guard bits k with which N of them fit
// in 64 bits (N 2^(53 + k) < 2^63); false if their exponents leave the range to
// FP64.  Within 7 N units of 2^(-52 - k) of the largest product's binade (a
// product's cut and its alignment's) and half an ulp; N / 2 units, the
// alignments' mean cut, are added back.  Root mean square errors in ulps of the
// largest product, twelve terms: 0.3 to 1.2, an FP64 fma chain 0.6 to 2.5; mean
// errors below 0.1 (0.3, all one way, with nothing added back).
template <int N>
struct DotGuard {
  static constexpr int k = N <= 7 ? 7 : 6;
};
template <int N>
CHEMORA_FX bool dot(const Parts (&p)[N], double* sum);

// In units of 2^(E - 1075 - K), E the exponent of the largest value: |result|
// <= 2^(53 + K).
CHEMORA_FX long long align(const Parts& p, int e) { return sar(p.m, (unsigned)(e - p.e)); }
template <int K>
CHEMORA_FX long long align(double v, int e) { return align(parts<K>(v), e); }

// v units of 2^(E - 1075 - K) as a double: nearest, ties away from zero, or to
// even as FP64 rounds (a difference of two doubles is often a tie, and the even
// one has a last bit less for the product with 1/h to round).
template <int K, bool EVEN = false>
CHEMORA_FX double to_double(long long v, int e) {
  const unsigned long long s = (unsigned long long)(v >> 63);
  const unsigned long long a = ((unsigned long long)v ^ s) - s;
  const int lz = clz64(a);
  const unsigned long long m = shl(a, (unsigned)lz);
  unsigned long long r = m >> 11;
  r += EVEN ? ((unsigned)m & 0x7ffu) + ((unsigned)r & 1u) > 0x400u : (m >> 10) & 1;
  r += (unsigned long long)(unsigned)(e + 10 - K - lz) << 52;
  r |= s & 0x8000000000000000ull;
  return a == 0 ? 0.0 : from_bits(r);
}

template <int N>
CHEMORA_FX bool dot(const Parts (&p)[N], double* sum) {
  int e = kZeroExp;
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int q = 0; q < N; ++q) e = emax(e, p[q].e);
  *sum = 0.0;
  if (e == kZeroExp) return true;
  if (!in_range(e)) return false;
  long long m = N / 2;
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int q = 0; q < N; ++q) m += align(p[q], e);
  *sum = to_double<DotGuard<N>::k>(m, e);
  return true;
}

// A sum of 64-bit integers with constant weights, exact in 96 bits: hi 2^32 + lo.
struct Sum96 {
  long long hi = 0, lo = 0;
  template <int W>
  CHEMORA_FX void add(long long v) {
    hi += (long long)W * (int)(v >> 32);
    if (W > 0)
      lo += (long long)((unsigned long long)(unsigned)W * (unsigned)v);
    else
      lo -= (long long)((unsigned long long)(unsigned)-W * (unsigned)v);
  }
  // rounded down to units 2^d larger
  CHEMORA_FX void shift(unsigned d) {
    const long long h = hi + (lo >> 32);
    lo = (unsigned)(d < 32 ? shr((unsigned long long)h << 32 | (unsigned)lo, d) : (unsigned long long)sar(h, d - 32));
    hi = sar(h, d);
  }
};
template <int K>
CHEMORA_FX double to_double(const Sum96& v, int e) {
  const long long h = v.hi + (v.lo >> 32);
  const unsigned s = (unsigned)(h >> 63);
  unsigned long long a = (unsigned long long)(h ^ (h >> 63));
  unsigned b = ((unsigned)v.lo ^ s) - s;
  a += (s & 1u) & (unsigned)(b == 0);
  const bool small = a == 0;
  a = small ? b : a;
  b = small ? 0u : b;
  const int lz = clz64(a);
  const unsigned long long m = shl(a, (unsigned)lz) | shr((unsigned long long)b << 32, (unsigned)(64 - lz));
  unsigned long long r = (m >> 11) + ((m >> 10) & 1);
  r += (unsigned long long)(unsigned)(e + (small ? 10 : 42) - K - lz) << 52;
  r |= (unsigned long long)(s & 0x80000000u) << 32;
  return a == 0 ? 0.0 : from_bits(r);
}

#if defined(__CUDACC__)
// to_double through the conversion instruction (nearest, ties to even), which
// takes a slot of the FP64 pipe and a few integer operations instead of some
// thirty of these.
template <int K>
CHEMORA_FX double to_double_cvt(long long v, int e) {
  const double d = __ll2double_rn(v);
  const int h = __double2hiint(d);
  return __hiloint2double(h == 0 ? 0 : h + ((e - 1075 - K) << 20), __double2loint(d));
}
#endif

}  // namespace fx
}  // namespace chemora
