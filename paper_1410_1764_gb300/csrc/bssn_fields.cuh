// Derivative fields of the BSSN variables and the algebra kernels' loader.
//
// A BSSN right-hand side is split in two kernels.  The first evaluates every
// derivative the equations read -- centred first and second differences and
// the Kreiss-Oliger term, 162 numbers per point -- almost entirely on the
// integer units (fixedpoint.cuh) and writes them to a workspace; the second
// reads them back, one number per load, and does the algebra: 1058 FP64
// operations per point, 272 of them on the integer units (bssn_prologue.cuh),
// where the fused bodies issue 2039 (x/y sharing) to 2642 (direct).  FP64 issue is what bounds these equations on GB300, so the
// 2.6 KB per point that the workspace costs in memory traffic is the cheaper
// side.  Neither kernel needs a particular grid shape, so small and ragged
// grids, patches and refined boxes run the same code at the same rate.
#pragma once
#include "device_types.cuh"
#include "fixedpoint.cuh"

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

// A slab with its extents and strides, and its tiles: columns of tw x th
// points and zb planes.
struct FieldRegion : FieldSlab {
  Dims d;
  int tw, th, zb, tnx, tny;
};

// What the integer prologue of the algebra kernels (bssn_prologue.cuh) leaves
// in shared memory for the point's thread, kPre columns of BLK threads: sums
// adv of the variables but gt_ij, traces tr of the variables with second
// derivatives but phi, the inverse metric, the shift's derivatives.
constexpr int kPreAdv = 0, kPreTr = 18, kPreGu = 28, kPreDb = 34, kPre = 43;
__host__ __device__ constexpr int adv_index(int v) { return kPreAdv + (v == 0 ? 0 : v - 6); }
__host__ __device__ constexpr int tr_index(int v) { return kPreTr + (v < 7 ? v - 1 : v - 11); }

// Loader of the algebra bodies: the state at the point, its fields, and the
// prologue's results (unused, s NULL, by the constraints).
template <int BLK>
struct FieldLoader {
  const double* __restrict__ p;  // variable 0 at the point
  int64_t sv;
  const double* __restrict__ w;  // field 0 at the point
  double* s;                     // the thread's column of the prologue's results
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
  __device__ __forceinline__ double adv(int v) const { return s[adv_index(v) * BLK]; }
  __device__ __forceinline__ double tr(int v) const { return s[tr_index(v) * BLK]; }
  __device__ __forceinline__ double gu(int ab) const { return s[(kPreGu + ab) * BLK]; }
  __device__ __forceinline__ double db(int i, int a) const { return s[(kPreDb + 3 * i + a) * BLK]; }
};

#if defined(__CUDACC__) && !defined(__CUDACC_RTC__)
// 8 (f+1 - f-1) - (f+2 - f-2) along stride st, in FP64 (rows of the mixed
// derivatives past a tile's edge).
__device__ __forceinline__ double d1_row_fp64(const double* __restrict__ p, int64_t st, double one, double eight) {
  const double q1 = fma(__ldg(p - st), -one, __ldg(p + st));
  const double q2 = fma(__ldg(p - 2 * st), -one, __ldg(p + 2 * st));
  return fma(eight, q1, -q2);
}
#endif

}  // namespace chemora
