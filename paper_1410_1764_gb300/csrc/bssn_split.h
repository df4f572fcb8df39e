// Host side of the split BSSN right-hand side, shared by its launchers.
#pragma once
#include <algorithm>

#include "bssn_fields.cuh"
#include "internal.h"

namespace chemora {

// The region of grid d (storage offset, first workspace point w0) with its tiles.
FieldRegion field_region(const Dims& d, int64_t offset, int64_t w0);
// Planes of d whose fields fit in the workspace (0: not even one).
int field_chunk_planes(const Dims& d, const FieldWork& work);
// The derivative fields of variables 0 .. nvars-1 of region R.
int launch_fields(const FieldRegion& R, int nvars, const double* src, double* work, const Scalars& sc,
                  cudaStream_t s);

// Launches the fields and then launch(R) for each range R of z planes whose
// fields fit in the workspace.
template <class F>
int for_field_chunks(const Dims& d, const Scalars& sc, const double* src, int nvars, const FieldWork& work,
                     cudaStream_t s, F launch) {
  const int planes = field_chunk_planes(d, work);
  if (planes < 1) return set_error(CHEMORA_EINVAL, "derivative workspace smaller than a plane");
  const int nchunks = (d.nz + planes - 1) / planes, each = (d.nz + nchunks - 1) / nchunks;
  int rc;
  for (int k0 = 0; k0 < d.nz; k0 += each) {
    Dims dk = d;
    dk.nz = std::min(each, d.nz - k0);
    const FieldRegion R = field_region(dk, (int64_t)k0 * d.sz, 0);
    if ((rc = launch_fields(R, nvars, src, work.w, sc, s))) return rc;
    if ((rc = launch(R))) return rc;
  }
  return CHEMORA_OK;
}

}  // namespace chemora
