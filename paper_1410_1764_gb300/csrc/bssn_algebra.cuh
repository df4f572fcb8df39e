// Device body of the BSSN algebra kernels (bssn_fields.cuh): one point per
// thread, the state at the point and its derivative fields in, the fused
// Runge-Kutta update out.  The run-time compiler includes this file too.
#pragma once
#include "stage.cuh"
#include "bssn_prologue.cuh"
#include "generated/gen_bssn_alg.cuh"

namespace chemora {

// Offset of interior point `lin` (x fastest) of d in its storage.
__device__ __forceinline__ int64_t region_point(const Dims& d, int64_t lin) {
  const unsigned plane = (unsigned)d.nx * (unsigned)d.ny;
  const int k = (int)(lin / plane);
  const unsigned r = (unsigned)(lin - (int64_t)k * plane);
  const int j = (int)(r / (unsigned)d.nx), i = (int)(r - (unsigned)j * (unsigned)d.nx);
  return (int64_t)(k + d.g) * d.sz + (int64_t)(j + d.g) * d.sy + (i + d.g);
}

template <int BLK, class SC>
__device__ __forceinline__ void bssn_algebra_point(const Dims& d, const FieldSlab& R, int64_t lin, const SC& sc,
                                                   const StageParams& a, const double* __restrict__ work,
                                                   double* pre) {
  const int64_t c = R.offset + region_point(d, lin);
  const FieldLoader<BLK> ld{a.src + c, d.sv, work + field_base(R.w0 + lin), pre + threadIdx.x};
  StageOut out = CHEMORA_STAGE_OUT(a, c, d.sv, sc);
  bssn_shift_terms(ld, sc, out);
  bssn_traces(ld, sc);
  chemora_bssn_alg_point(ld, sc, out);
}

template <int BLK, class SC>
__device__ __forceinline__ void bssn_algebra(const Dims& d, const FieldSlab& R, const SC& sc, const StageParams& a,
                                             const double* __restrict__ work) {
  __shared__ double pre[kPre * BLK];
  const int64_t lin = (int64_t)blockIdx.x * BLK + threadIdx.x;
  if (lin < R.npts) bssn_algebra_point<BLK>(d, R, lin, sc, a, work, pre);
}

}  // namespace chemora
