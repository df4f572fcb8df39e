// Ahead-of-time BSSN stage kernels: the device bodies of bssn_kernels.cuh
// compiled for a few launch shapes with the grid and scalars as kernel
// parameters; the autotuner picks one shape per system and grid.
//
// The FP64 pipe is the bound on GB300 (two FP64 FMA per clock per SM), so
// blocks of 64-256 threads with up to 255 registers each and a few blocks per
// SM already keep it busy.
#include <atomic>

#include "internal.h"
#include "bssn_kernels.cuh"

namespace chemora {

// The direct body in one kernel without a workspace: for callers that may not
// allocate one (chemora_rk4_step_noalloc, no memory left).
__global__ void __launch_bounds__(128, 2) bssn_stage_kernel(Dims d, Scalars sc, StageParams a) {
  bssn_direct_body<32, 4>(d, sc, a);
}

static int launch_bssn_direct(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s) {
  dim3 grid((d.nx + 31) / 32, (d.ny + 3) / 4, d.nz);
  bssn_stage_kernel<<<grid, dim3(32, 4), 0, s>>>(d, sc, a);
  return launched("bssn_stage_kernel");
}

template <int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX * TY, MINB) bssn_xstage_kernel(Dims d, Scalars sc, StageParams a) {
  bssn_x_body<TX, TY>(d, sc, a);
}

template <int TX, int TY, int MINB>
static int launch_bssn_xvariant(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s) {
  if (d.nx % TX != 0 || d.g < 3)
    return set_error(CHEMORA_EUNSUPPORTED, "x-sharing BSSN kernel needs nx %% %d == 0", TX);
  dim3 grid(d.nx / TX, (d.ny + TY - 1) / TY, d.nz);
  bssn_xstage_kernel<TX, TY, MINB><<<grid, dim3(TX, TY), 0, s>>>(d, sc, a);
  return launched("bssn_xstage_kernel");
}

template <int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX * TY, MINB) bssn_xystage_kernel(Dims d, Scalars sc, StageParams a) {
  extern __shared__ double smem[];
  bssn_xy_body<TX, TY>(d, sc, a, smem);
}

template <int TX, int TY, int MINB>
static int launch_bssn_xyvariant(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s) {
  if (d.nx % TX != 0 || d.g < 3)
    return set_error(CHEMORA_EUNSUPPORTED, "xy-sharing BSSN kernel needs nx %% %d == 0", TX);
  constexpr unsigned smem = bssn_xy_smem_bytes(TX, TY);
  // the dynamic shared-memory limit is a per-device function attribute: set
  // once per device (a bit per device ordinal; thread-safe)
  static std::atomic<unsigned long long> attr_set{0};
  int dev = 0;
  CHEMORA_CUDA(cudaGetDevice(&dev));
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(attr_set.load() & bit)) {
    CHEMORA_CUDA(cudaFuncSetAttribute(bssn_xystage_kernel<TX, TY, MINB>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    attr_set.fetch_or(bit);
  }
  dim3 grid(d.nx / TX, (d.ny + TY - 1) / TY, d.nz);
  bssn_xystage_kernel<TX, TY, MINB><<<grid, dim3(TX, TY), smem, s>>>(d, sc, a);
  return launched("bssn_xystage_kernel");
}

// Launch shapes the autotuner chooses from (variant 0 is the default; bssn_shape
// says which one runs on a grid).
// Sharing 0: the split kernels, tx x ty the algebra kernel's block.
const LaunchVariant kBssnVariants[] = {
    {32, 4, 4, launch_bssn_direct},
    {32, 4, 2, launch_bssn_direct},
    {32, 4, 3, launch_bssn_direct},
    {32, 2, 5, launch_bssn_direct},
    {32, 2, 8, launch_bssn_direct},
    {64, 2, 3, launch_bssn_direct},
    {64, 2, 2, launch_bssn_direct},
    {64, 1, 5, launch_bssn_direct},
    {32, 2, 4, launch_bssn_xvariant<32, 2, 4>, 1},
    {32, 4, 2, launch_bssn_xvariant<32, 4, 2>, 1},
    {64, 2, 2, launch_bssn_xvariant<64, 2, 2>, 1},
    {32, 2, 5, launch_bssn_xvariant<32, 2, 5>, 1},
    {32, 2, 6, launch_bssn_xvariant<32, 2, 6>, 1},
    {32, 2, 8, launch_bssn_xvariant<32, 2, 8>, 1},
    {32, 8, 1, launch_bssn_xyvariant<32, 8, 1>, 2},
    {32, 8, 2, launch_bssn_xyvariant<32, 8, 2>, 2},
    {32, 16, 1, launch_bssn_xyvariant<32, 16, 1>, 2},
    // fewer rows per block: more registers per thread (168-200), fewer warps
    {32, 5, 2, launch_bssn_xyvariant<32, 5, 2>, 2},
    {32, 6, 2, launch_bssn_xyvariant<32, 6, 2>, 2},
    {32, 7, 2, launch_bssn_xyvariant<32, 7, 2>, 2},
    {32, 12, 1, launch_bssn_xyvariant<32, 12, 1>, 2},
};
const int kNumBssnVariants = sizeof(kBssnVariants) / sizeof(kBssnVariants[0]);

// The shape that runs for `variant` on d: the sharing shapes need whole warps of x
// points and three ghost layers, else the default runs, which is half a block
// (variant 4) below two waves of 128-thread blocks (four per SM), where it evens
// out the SMs' shares (37 x 29 x 23, field and algebra kernels: 122 us with 128
// threads, 106 with 64; 128^3: 4.73 and 4.83 ms).
int bssn_shape(const Dims& d, int variant) {
  if (variant < 0 || variant >= kNumBssnVariants) variant = 0;
  const LaunchVariant& v = kBssnVariants[variant];
  if (v.xshare && (d.nx % v.tx != 0 || d.g < 3)) variant = 0;
  if (variant == 0 && (int64_t)d.nx * d.ny * d.nz < 2 * 152 * 4 * 128) variant = 4;
  return variant;
}

bool bssn_shape_splits(const Dims& d, int variant) { return !kBssnVariants[bssn_shape(d, variant)].xshare; }

int launch_bssn_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s, int variant,
                      const FieldWork& work) {
  const LaunchVariant& v = kBssnVariants[bssn_shape(d, variant)];
  if (v.xshare || !work.w) return v.launch(d, sc, a, s);
  return launch_bssn_split(d, sc, a, work, v.tx * v.ty, v.minb, s);
}

}  // namespace chemora
