// Scalar wave (Sec. 3, Eq. 1, two-variable form) and variable-speed wave
// stage kernels, stencils on the integer units; a few block shapes are compiled
// for the autotuner.
#include "internal.h"
#include "stage.cuh"
#include "star_march.cuh"
#include "varc_march.cuh"
#include "wave_point.cuh"

namespace chemora {

template <int TX, int TY>
__global__ void __launch_bounds__(TX * TY) wave_stage_kernel(Dims d, Scalars sc, StageParams a) {
  const int i = blockIdx.x * TX + threadIdx.x;
  const int j = blockIdx.y * TY + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= d.nx || j >= d.ny) return;
  const int64_t c = (int64_t)(k + d.g) * d.sz + (int64_t)(j + d.g) * d.sy + (i + d.g);
  Loader<2> ld{a.src + c, nullptr, d.sy, d.sz, d.sv};
  // y_n and the accumulator are fetched with the neighbours: bound by the
  // latency of its loads otherwise
  MarchUpdate<2> up;
  up.load(a, c, d.sv);
  double kk[2];
  ArrayOut<2> out{kk};
  wave_point(ld, sc, out);
  up.apply(a, c, d.sv, kk, sc.k[CHEMORA_K_ONE], sc.k[CHEMORA_K_TWO], [&](int64_t o, double x) { a.dst[o] = x; });
}

template <int TX, int TY>
static int launch_wave_variant(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s) {
  dim3 grid((d.nx + TX - 1) / TX, (d.ny + TY - 1) / TY, d.nz);
  wave_stage_kernel<TX, TY><<<grid, dim3(TX, TY), 0, s>>>(d, sc, a);
  return launched("wave_stage_kernel");
}

template <int TX, int TY>
static int launch_varc_variant(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s) {
  return launch_varc_march<TX, TY>(d, sc, a, nullptr, s);
}

// Planes in shared memory (wave_orders.cu) win where blocks marching through
// many planes fill the GPU (256^3: 233 us per stage against 290), a point per
// thread on small grids (61 x 75 x 53: 10.3 against 11.1); the autotuner times
// both.
const LaunchVariant kWaveVariants[] = {
    {32, 8, 0, launch_wave_variant<32, 8>},   {32, 4, 0, launch_wave_variant<32, 4>},
    {64, 4, 0, launch_wave_variant<64, 4>},   {128, 2, 0, launch_wave_variant<128, 2>},
    {16, 16, 0, launch_wave_variant<16, 16>},
    {32, 8, 0, launch_wave_planes<32, 8>, 4}, {32, 4, 0, launch_wave_planes<32, 4>, 4},
    {16, 16, 0, launch_wave_planes<16, 16>, 4}, {64, 4, 0, launch_wave_planes<64, 4>, 4},
    {16, 8, 0, launch_wave_planes<16, 8>, 4},   {8, 16, 0, launch_wave_planes<8, 16>, 4},
    {32, 16, 0, launch_wave_variant<32, 16>},   {16, 8, 0, launch_wave_variant<16, 8>},
};
const int kNumWaveVariants = sizeof(kWaveVariants) / sizeof(kWaveVariants[0]);

const LaunchVariant kVarcVariants[] = {
    {32, 8, 0, launch_varc_variant<32, 8>},   {32, 4, 0, launch_varc_variant<32, 4>},
    {64, 4, 0, launch_varc_variant<64, 4>},   {16, 16, 0, launch_varc_variant<16, 16>},
    {16, 8, 0, launch_varc_variant<16, 8>},   {8, 16, 0, launch_varc_variant<8, 16>},
};
const int kNumVarcVariants = sizeof(kVarcVariants) / sizeof(kVarcVariants[0]);

int launch_wave_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s, int variant) {
  if (sc.order != 4) return launch_wave_order_stage(d, sc, a, s, variant);
  if (variant < 0 || variant >= kNumWaveVariants) variant = 0;
  const LaunchVariant& v = kWaveVariants[variant];
  return v.launch(d, sc, a, s);
}

int launch_varc_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s, int variant) {
  if (variant < 0 || variant >= kNumVarcVariants) variant = 0;
  return kVarcVariants[variant].launch(d, sc, a, s);
}

}  // namespace chemora
