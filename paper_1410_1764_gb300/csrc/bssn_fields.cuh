// Derivative fields of the BSSN variables and the algebra kernels' loader.
//
// A BSSN right-hand side is split in two kernels.  The first evaluates every
// derivative the equations read -- centred first and second differences and
// the Kreiss-Oliger term, 162 numbers per point -- almost entirely on the
// integer units (fixedpoint.cuh) and writes them to a workspace; the second
// reads them back, one number per load, and does the algebra: 1058 FP64
// instructions per point where the fused bodies issue 2039 (x/y sharing) to
// 2642 (direct).  FP64 issue is what bounds these equations on GB300, so the
// 2.6 KB per point that the workspace costs in memory traffic is the cheaper
// side.  Neither kernel needs a particular grid shape, so small and ragged
// grids, patches and refined boxes run the same code at the same rate.
#pragma once
#include "device_types.cuh"
#if !defined(__CUDACC_RTC__)
#include "fixedpoint.cuh"
#endif

namespace chemora {

constexpr int kFieldD1 = 0;                     // 12h D_a f: 3 v + a
constexpr int kFieldKo = 72;                    // 64h/eps KO f: v
constexpr int kFieldD2 = 96;                    // 6 ddi + {xx, yy, zz: 12h^2 D_aa; xy, xz, yz: 144h^2 D_ab}
constexpr int kFields = 162;
constexpr int kFieldBlock = 128;                // points per workspace block: [block][field][point]

// Index of variable v among those with second derivatives (phi, gt_ij,
// alpha, beta^i), or -1.
__host__ __device__ constexpr int dd_index(int v) { return v < 7 ? v : (v >= 17 && v <= 20 ? v - 10 : -1); }

__host__ __device__ constexpr int64_t field_base(int64_t point) {
  return (point / kFieldBlock) * (int64_t)(kFields * kFieldBlock) + point % kFieldBlock;
}

// Points whose derivatives are evaluated together: the interior of a grid or
// patch, or a range of its z planes.
struct FieldSlab {
  int64_t offset;  // first double of the slab's state in its storage
  int64_t npts;    // interior points
  int64_t w0;      // its first point in the workspace
};

// A slab with its extents and strides, and its tiles of tw x th points of one plane.
struct FieldRegion : FieldSlab {
  Dims d;
  int tw, th, tnx, tny;
};

// Loader of the algebra bodies: the state at the point and its fields.
struct FieldLoader {
  const double* __restrict__ p;  // variable 0 at the point
  int64_t sv;
  const double* __restrict__ w;  // field 0 at the point
  __device__ __forceinline__ double operator()(int v, int, int, int) const { return __ldg(p + v * sv); }
  __device__ __forceinline__ double g1(int v, int a) const {
    return __ldg(w + (kFieldD1 + 3 * v + a) * kFieldBlock);
  }
  __device__ __forceinline__ double g2(int v, int a) const {
    return __ldg(w + (kFieldD2 + 6 * dd_index(v) + a) * kFieldBlock);
  }
  __device__ __forceinline__ double g11(int v, int ab) const {
    return __ldg(w + (kFieldD2 + 6 * dd_index(v) + 3 + ab) * kFieldBlock);
  }
  __device__ __forceinline__ double gko(int v) const { return __ldg(w + (kFieldKo + v) * kFieldBlock); }
};

#if defined(__CUDACC__) && !defined(__CUDACC_RTC__)
// The radius-3 star around a point: centre and n[6 a + {+1, -1, +2, -2, +3, -3}].
struct Star3 {
  double c, n[18];
  __device__ __forceinline__ void load(const double* __restrict__ p, int64_t sy, int64_t sz) {
    const int64_t st[3] = {1, sy, sz};
    c = __ldg(p);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        n[6 * a + 2 * m] = __ldg(p + (m + 1) * st[a]);
        n[6 * a + 2 * m + 1] = __ldg(p - (m + 1) * st[a]);
      }
  }
  __device__ __forceinline__ unsigned exponent() const {
    unsigned e = fx::ebits(c);
#pragma unroll
    for (int q = 0; q < 18; ++q) e = fx::emax(e, fx::ebits(n[q]));
    return e;
  }
  __device__ __forceinline__ bool all_zero() const {
    bool z = c == 0.0;
#pragma unroll
    for (int q = 0; q < 18; ++q) z = z && n[q] == 0.0;
    return z;
  }
};

// Raw differences of a star: d1[a] = 12h D_a, d2[a] = 12h^2 D_aa (when DD)
// and ko = 64h/eps KO.  Four guard bits: the weights of each axis add up to 64
// in magnitude at most, so every axis sum fits in 64 bits; the dissipation's
// three axis sums are added a quarter each (their truncation is 2^-55 of the
// largest value, on a term of weight eps/64).
template <bool DD>
__device__ __forceinline__ void star3_differences(const Star3& s, double* d1, double* d2, double& ko) {
  const unsigned e = s.exponent();
  if (fx::in_range(e)) {
    const long long c = fx::align<4>(s.c, e);
    long long k = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const long long p1 = fx::align<4>(s.n[6 * a], e), m1 = fx::align<4>(s.n[6 * a + 1], e);
      const long long p2 = fx::align<4>(s.n[6 * a + 2], e), m2 = fx::align<4>(s.n[6 * a + 3], e);
      const long long p3 = fx::align<4>(s.n[6 * a + 4], e), m3 = fx::align<4>(s.n[6 * a + 5], e);
      const long long s1 = p1 + m1, s2 = p2 + m2;
      d1[a] = fx::to_double<4>(8 * (p1 - m1) - (p2 - m2), e);
      if (DD) d2[a] = fx::to_double<4>(16 * s1 - s2 - 30 * c, e);
      k += (15 * s1 - 6 * s2 + (p3 + m3) - 20 * c) >> 2;
    }
    ko = fx::to_double<2>(k, e);
  } else if (s.all_zero()) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      d1[a] = 0.0;
      if (DD) d2[a] = 0.0;
    }
    ko = 0.0;
  } else {  // the ends of the FP64 range, Inf, NaN: FP64 differences
    ko = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double* n = s.n + 6 * a;
      const double c1 = (n[0] - s.c) + (n[1] - s.c), c2 = (n[2] - s.c) + (n[3] - s.c);
      const double c3 = (n[4] - s.c) + (n[5] - s.c);
      d1[a] = fma(8.0, n[0] - n[1], -(n[2] - n[3]));
      if (DD) d2[a] = fma(16.0, c1, -c2);
      ko += fma(15.0, c1, fma(-6.0, c2, c3));
    }
  }
}

// 8 (f+1 - f-1) - (f+2 - f-2) along stride st, in FP64 (rows of the mixed
// derivatives past a tile's edge).
__device__ __forceinline__ double d1_row_fp64(const double* __restrict__ p, int64_t st, double one, double eight) {
  const double q1 = fma(__ldg(p - st), -one, __ldg(p + st));
  const double q2 = fma(__ldg(p - 2 * st), -one, __ldg(p + 2 * st));
  return fma(eight, q1, -q2);
}
#endif

}  // namespace chemora
