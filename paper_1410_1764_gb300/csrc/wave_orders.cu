// Scalar-wave stage kernels of arbitrary finite-difference order (Sec.
// 3.2.2: "standard" operators of arbitrary order, the order fixed when the
// code is generated): the two-variable form at orders 2, 6, 8 (order 4 is in
// wave.cu) and the first-order form of Eq. 1 (u, rho, v_i) at orders 2, 4,
// 6, 8, in a few block shapes for the autotuner to choose from.  The stencils
// run on the integer units (star_march.cuh); values those cannot take go to
// the FP64 bodies generated from gen/systems.py.
//
// GB300, us per stage, FP64 bodies (49 and 42 instructions at 17.8 cycles each)
// and now: two-variable form of order 8 on 128^3 222 and 48, first-order form of
// order 6 on 117 x 90 x 131 174 and 84; order 4 on 256^3 with every point taking
// its 13 values apart itself (wave.cu) 290 and 233 here.  What bounds them now is
// the FP64 pipe (5 and 14 instructions per point, 40 to 54 % of its time) and the
// latency of the integer chains at 20 and 15 warps per SM; HBM alone takes 158 us
// of the 233.
#include "internal.h"
#include "stage.cuh"
#include "star_march.cuh"
#include "generated/gen_wave.cuh"
#include "generated/gen_wave_o2.cuh"
#include "generated/gen_wave_o6.cuh"
#include "generated/gen_wave_o8.cuh"
#include "generated/gen_wave1_o2.cuh"
#include "generated/gen_wave1_o4.cuh"
#include "generated/gen_wave1_o6.cuh"
#include "generated/gen_wave1_o8.cuh"

namespace chemora {

#define CHEMORA_BODY(NAME, NV, FN)                                                              \
  struct NAME {                                                                                 \
    static constexpr int nv = NV;                                                               \
    template <class LD, class OUT>                                                              \
    __device__ __forceinline__ static void eval(const LD& ld, const Scalars& sc, OUT& o) {      \
      FN(ld, sc, o);                                                                            \
    }                                                                                           \
  };

CHEMORA_BODY(WaveO2, 2, chemora_wave_o2_point)
CHEMORA_BODY(WaveO6, 2, chemora_wave_o6_point)
CHEMORA_BODY(WaveO8, 2, chemora_wave_o8_point)
CHEMORA_BODY(Wave1O2, 5, chemora_wave1_o2_point)
CHEMORA_BODY(Wave1O4, 5, chemora_wave1_o4_point)
CHEMORA_BODY(Wave1O6, 5, chemora_wave1_o6_point)
CHEMORA_BODY(Wave1O8, 5, chemora_wave1_o8_point)

// Threads per SM asked of the compiler, the most that leaves next to no spills
// (order 4, two guard bits: 245 us per stage of 256^3 with 768 threads, 270 with
// 1024 and 20 bytes spilled; order 8: 10 steps on 128^3 2.01 ms with 640, 2.28 with 768 and
// 48 bytes spilled; first-order form of order 6 on 117 x 90 x 131: 93 us per
// stage with 512, 141 with 640 and 160 bytes spilled).
template <int NV, int R>
constexpr int march_threads() { return NV == 2 ? (R == 1 ? 1024 : (R == 4 ? 640 : 768)) : (R == 1 ? 768 : 512); }

// Two-variable form, order 2R: one Laplacian of u per point.
template <class BODY, int R, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, march_threads<2, R>() / (TX * TY))
wave_march_order_kernel(Dims d, Scalars sc, StageParams a, int zb, double scale) {
  constexpr int P = TX + 2 * R, K = Guard<R>::lap;
  __shared__ long long pm[2][P * (TY + 2 * R)];
  __shared__ int pe[2][P * (TY + 2 * R)];
  const MarchPlace<TX, TY> p(d, zb);
  const MarchHalo<R, TX, TY> hl(p);
  const double* org = a.src + p.org;
  const int64_t own = (int64_t)p.ly * d.sy + p.lx;
  const int pc = (p.ly + R) * P + p.lx + R;
  fx::Parts z[2 * R + 1];
  double znext = 0.0, hnext[hl.n];
#pragma unroll
  for (int m = 0; m <= 2 * R; ++m) z[m] = fx::Parts{0, 0};
  if (p.active) {
#pragma unroll
    for (int m = 1; m <= 2 * R; ++m) z[m] = fx::parts_or_zero<K>(__ldg(org + own + (int64_t)(m - 1 - R) * d.sz));
    znext = __ldg(org + own + R * d.sz);
  }
#pragma unroll
  for (int q = 0; q < hl.n; ++q) hnext[q] = hl.live[q] ? __ldg(org + (int64_t)hl.y[q] * d.sy + hl.x[q]) : 0.0;
  int64_t c = p.org + own;
#pragma unroll 1
  for (int k = 0; k < p.nz; ++k, c += d.sz, org += d.sz) {
    long long* const M = pm[k & 1];
    int* const E = pe[k & 1];
    MarchUpdate<2> up;
    double rho = 0.0;
#pragma unroll
    for (int m = 0; m < 2 * R; ++m) z[m] = z[m + 1];
    z[2 * R] = fx::parts_or_zero<K>(znext);
    if (p.active) {
      M[pc] = z[R].m;
      E[pc] = z[R].e;
      rho = __ldg(a.src + d.sv + c);
      up.load(a, c, d.sv);
      if (k + 1 < p.nz) znext = __ldg(org + own + (R + 1) * d.sz);
    }
#pragma unroll
    for (int q = 0; q < hl.n; ++q)
      if (hl.live[q]) {
        const fx::Parts v = fx::parts_or_zero<K>(hnext[q]);
        const int o = (hl.y[q] + R) * P + hl.x[q] + R;
        M[o] = v.m;
        E[o] = v.e;
        if (k + 1 < p.nz) hnext[q] = __ldg(org + d.sz + (int64_t)hl.y[q] * d.sy + hl.x[q]);
      }
    __syncthreads();
    if (p.active) {
      int ex[2 * R], ey[2 * R], en = z[R].e, ef = fx::kZeroExp;
#pragma unroll
      for (int m = 0; m < 2 * R; ++m) {
        ex[m] = E[pc + tap<R>(m)];
        ey[m] = E[pc + tap<R>(m) * P];
        int& t = is_near<R>(tap<R>(m)) ? en : ef;
        t = fx::emax(t, fx::emax(fx::emax(ex[m], ey[m]), z[R + tap<R>(m)].e));
      }
      const int e = fx::emax(en, ef);
      if (star_ok<R>(e)) {
        double lap = 0.0;
        if (e != fx::kZeroExp) {
          long long s[R];
#pragma unroll
          for (int q = 0; q < R; ++q) s[q] = 0;
#pragma unroll
          for (int m = 0; m < 2 * R; ++m) {
            const int o = tap<R>(m), q = o < 0 ? -o - 1 : o - 1, to = is_near<R>(o) ? en : e;
            s[q] += fx::sar(M[pc + o], (unsigned)(to - ex[m])) + fx::sar(M[pc + o * P], (unsigned)(to - ey[m])) +
                    fx::align(z[R + o], to);
          }
          lap = star_lap<R>(s, fx::align(z[R], en), en, fx::align(z[R], e), e);
        }
        const double kk[2] = {rho, __fma_rn(lap, scale, sc.k[CHEMORA_K_MZERO])};
        up.apply(a, c, d.sv, kk, sc.k[CHEMORA_K_ONE], sc.k[CHEMORA_K_TWO], [&](int64_t o, double x) { a.dst[o] = x; });
      } else {
        Loader<2> ld{a.src + c, nullptr, d.sy, d.sz, d.sv};
        StageOutFma out = CHEMORA_STAGE_OUT_FMA(a, c, d.sv, sc);
        BODY::eval(ld, sc, out);
      }
    }
  }
}

// First-order form, order 2R: rho_t = sum_a D_a v_a, (v_a)_t = D_a rho.  rho's
// plane is in shared memory with both halos, v_x's with its x halo, v_y's
// with its y halo; rho's and v_z's columns are in registers.
template <class BODY, int R, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, march_threads<5, R>() / (TX * TY))
wave1_march_kernel(Dims d, Scalars sc, StageParams a, int zb, double scale) {
  constexpr int P = TX + 2 * R, K = Guard<R>::d1;
  constexpr int NR = P * (TY + 2 * R), NX = P * TY, NY = TX * (TY + 2 * R);
  __shared__ long long pm[2][NR + NX + NY];
  __shared__ int pe[2][NR + NX + NY];
  const MarchPlace<TX, TY> p(d, zb);
  const MarchHalo<R, TX, TY> hl(p);
  const double* org = a.src + p.org;
  const int64_t own = (int64_t)p.ly * d.sy + p.lx;
  const int pr = (p.ly + R) * P + p.lx + R;            // this point in rho's plane
  const int px = NR + p.ly * P + p.lx + R;             // in v_x's
  const int py = NR + NX + (p.ly + R) * TX + p.lx;     // in v_y's
  fx::Parts z[2 * R + 1], vz[2 * R + 1];
  double rnext = 0.0, vnext = 0.0, hr[hl.n], hv[hl.n];
#pragma unroll
  for (int m = 0; m <= 2 * R; ++m) z[m] = vz[m] = fx::Parts{0, 0};
  if (p.active) {
#pragma unroll
    for (int m = 1; m <= 2 * R; ++m) {
      z[m] = fx::parts_or_zero<K>(__ldg(org + own + d.sv + (int64_t)(m - 1 - R) * d.sz));
      vz[m] = fx::parts_or_zero<K>(__ldg(org + own + 4 * d.sv + (int64_t)(m - 1 - R) * d.sz));
    }
    rnext = __ldg(org + own + d.sv + R * d.sz);
    vnext = __ldg(org + own + 4 * d.sv + R * d.sz);
  }
#pragma unroll
  for (int q = 0; q < hl.n; ++q) {
    const double* h = org + (int64_t)hl.y[q] * d.sy + hl.x[q];
    hr[q] = hl.live[q] ? __ldg(h + d.sv) : 0.0;
    hv[q] = hl.live[q] ? __ldg(h + (hl.along_x[q] ? 2 : 3) * d.sv) : 0.0;
  }
  int64_t c = p.org + own;
#pragma unroll 1
  for (int k = 0; k < p.nz; ++k, c += d.sz, org += d.sz) {
    long long* const M = pm[k & 1];
    int* const E = pe[k & 1];
    MarchUpdate<5> up;
    double rho = 0.0;
#pragma unroll
    for (int m = 0; m < 2 * R; ++m) {
      z[m] = z[m + 1];
      vz[m] = vz[m + 1];
    }
    z[2 * R] = fx::parts_or_zero<K>(rnext);
    vz[2 * R] = fx::parts_or_zero<K>(vnext);
    if (p.active) {
      const fx::Parts vx = fx::parts_or_zero<K>(__ldg(a.src + 2 * d.sv + c));
      const fx::Parts vy = fx::parts_or_zero<K>(__ldg(a.src + 3 * d.sv + c));
      M[pr] = z[R].m;
      E[pr] = z[R].e;
      M[px] = vx.m;
      E[px] = vx.e;
      M[py] = vy.m;
      E[py] = vy.e;
      rho = __ldg(a.src + d.sv + c);
      up.load(a, c, d.sv);
      if (k + 1 < p.nz) {
        rnext = __ldg(org + own + d.sv + (R + 1) * d.sz);
        vnext = __ldg(org + own + 4 * d.sv + (R + 1) * d.sz);
      }
    }
#pragma unroll
    for (int q = 0; q < hl.n; ++q)
      if (hl.live[q]) {
        const fx::Parts r = fx::parts_or_zero<K>(hr[q]), v = fx::parts_or_zero<K>(hv[q]);
        const int o = (hl.y[q] + R) * P + hl.x[q] + R;
        const int ov = hl.along_x[q] ? NR + hl.y[q] * P + hl.x[q] + R : NR + NX + (hl.y[q] + R) * TX + hl.x[q];
        M[o] = r.m;
        E[o] = r.e;
        M[ov] = v.m;
        E[ov] = v.e;
        if (k + 1 < p.nz) {
          const double* h = org + d.sz + (int64_t)hl.y[q] * d.sy + hl.x[q];
          hr[q] = __ldg(h + d.sv);
          hv[q] = __ldg(h + (hl.along_x[q] ? 2 : 3) * d.sv);
        }
      }
    __syncthreads();
    if (p.active) {
      double kk[5];
      bool ok = true;
      {  // D_a rho, each axis to its own largest exponent
        const int st[2] = {1, P};
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          int te[2 * R], en = fx::kZeroExp, e = fx::kZeroExp;
#pragma unroll
          for (int m = 0; m < 2 * R; ++m) {
            te[m] = x < 2 ? E[pr + tap<R>(m) * st[x & 1]] : z[R + tap<R>(m)].e;
            if (is_near<R>(tap<R>(m))) en = fx::emax(en, te[m]);
            e = fx::emax(e, te[m]);
          }
          ok = ok && star_ok<R>(e);
          long long t[R];
#pragma unroll
          for (int q = 0; q < R; ++q) {
            const int up1 = R + q, dn = R - 1 - q;
            const long long f1 = x < 2 ? M[pr + (q + 1) * st[x & 1]] : z[R + q + 1].m;
            const long long f0 = x < 2 ? M[pr - (q + 1) * st[x & 1]] : z[R - q - 1].m;
            const int to = is_near<R>(q + 1) ? en : e;
            t[q] = fx::sar(f1, (unsigned)(to - te[up1])) - fx::sar(f0, (unsigned)(to - te[dn]));
          }
          kk[2 + x] = e == fx::kZeroExp ? 0.0 : star_d1<R>(t, en, e);
        }
      }
      {  // the divergence of v, one sum
        int ex[2 * R], ey[2 * R], en = fx::kZeroExp, ef = fx::kZeroExp;
#pragma unroll
        for (int m = 0; m < 2 * R; ++m) {
          ex[m] = E[px + tap<R>(m)];
          ey[m] = E[py + tap<R>(m) * TX];
          int& t = is_near<R>(tap<R>(m)) ? en : ef;
          t = fx::emax(t, fx::emax(fx::emax(ex[m], ey[m]), vz[R + tap<R>(m)].e));
        }
        const int e = fx::emax(en, ef);
        ok = ok && star_ok<R>(e);
        long long t[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int u1 = R + q, dn = R - 1 - q, to = is_near<R>(q + 1) ? en : e;
          t[q] = (fx::sar(M[px + q + 1], (unsigned)(to - ex[u1])) - fx::sar(M[px - q - 1], (unsigned)(to - ex[dn]))) +
                 (fx::sar(M[py + (q + 1) * TX], (unsigned)(to - ey[u1])) -
                  fx::sar(M[py - (q + 1) * TX], (unsigned)(to - ey[dn]))) +
                 (fx::align(vz[R + q + 1], to) - fx::align(vz[R - q - 1], to));
        }
        kk[1] = e == fx::kZeroExp ? 0.0 : star_d1<R>(t, en, e);
      }
      if (ok) {
        kk[0] = rho;
#pragma unroll
        for (int v = 1; v < 5; ++v) kk[v] = __fma_rn(kk[v], scale, sc.k[CHEMORA_K_MZERO]);
        up.apply(a, c, d.sv, kk, sc.k[CHEMORA_K_ONE], sc.k[CHEMORA_K_TWO], [&](int64_t o, double x) { a.dst[o] = x; });
      } else {
        Loader<5> ld{a.src + c, nullptr, d.sy, d.sz, d.sv};
        StageOutFma out = CHEMORA_STAGE_OUT_FMA(a, c, d.sv, sc);
        BODY::eval(ld, sc, out);
      }
    }
  }
}

template <class BODY, int R, int TX, int TY>
static int launch_order(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s) {
  const int zb = march_depth(d, TX, TY, march_threads<BODY::nv, R>() / (TX * TY));
  const dim3 grid = march_grid(d, TX, TY, zb);
  if constexpr (BODY::nv == 2)
    wave_march_order_kernel<BODY, R, TX, TY><<<grid, TX * TY, 0, s>>>(
        d, sc, a, zb, R == 2 ? sc.i12h2 : sc.ih2 / Central<R>::den2);
  else
    wave1_march_kernel<BODY, R, TX, TY><<<grid, TX * TY, 0, s>>>(d, sc, a, zb, sc.ih / Central<R>::den1);
  return launched("wave_march_order_kernel");
}

#define CHEMORA_SHAPES(BODY, R)                                                              \
  {{32, 8, 0, launch_order<BODY, R, 32, 8>},  {32, 4, 0, launch_order<BODY, R, 32, 4>},      \
   {64, 4, 0, launch_order<BODY, R, 64, 4>},  {16, 16, 0, launch_order<BODY, R, 16, 16>},    \
   {16, 8, 0, launch_order<BODY, R, 16, 8>},  {8, 16, 0, launch_order<BODY, R, 8, 16>}}

constexpr int kOrderShapes = 6;
static const LaunchVariant kWaveO2[kOrderShapes] = CHEMORA_SHAPES(WaveO2, 1);
static const LaunchVariant kWaveO6[kOrderShapes] = CHEMORA_SHAPES(WaveO6, 3);
static const LaunchVariant kWaveO8[kOrderShapes] = CHEMORA_SHAPES(WaveO8, 4);
static const LaunchVariant kWave1O2[kOrderShapes] = CHEMORA_SHAPES(Wave1O2, 1);
static const LaunchVariant kWave1O6[kOrderShapes] = CHEMORA_SHAPES(Wave1O6, 3);
static const LaunchVariant kWave1O8[kOrderShapes] = CHEMORA_SHAPES(Wave1O8, 4);
const LaunchVariant kWave1Variants[kOrderShapes] = CHEMORA_SHAPES(Wave1O4, 2);
const int kNumWave1Variants = kOrderShapes;

CHEMORA_BODY(WaveO4, 2, chemora_wave_point)

template <int TX, int TY>
int launch_wave_planes(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s) {
  return launch_order<WaveO4, 2, TX, TY>(d, sc, a, s);
}
template int launch_wave_planes<32, 8>(const Dims&, const Scalars&, const StageParams&, cudaStream_t);
template int launch_wave_planes<32, 4>(const Dims&, const Scalars&, const StageParams&, cudaStream_t);
template int launch_wave_planes<16, 16>(const Dims&, const Scalars&, const StageParams&, cudaStream_t);
template int launch_wave_planes<64, 4>(const Dims&, const Scalars&, const StageParams&, cudaStream_t);
template int launch_wave_planes<16, 8>(const Dims&, const Scalars&, const StageParams&, cudaStream_t);
template int launch_wave_planes<8, 16>(const Dims&, const Scalars&, const StageParams&, cudaStream_t);

int launch_wave_order_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s,
                            int variant) {
  if (variant < 0 || variant >= kOrderShapes) variant = 0;
  switch (sc.order) {
    case 2: return kWaveO2[variant].launch(d, sc, a, s);
    case 6: return kWaveO6[variant].launch(d, sc, a, s);
    case 8: return kWaveO8[variant].launch(d, sc, a, s);
    default: return set_error(CHEMORA_EUNSUPPORTED, "scalar wave of order %d is not compiled", sc.order);
  }
}

int launch_wave1_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s,
                       int variant) {
  if (variant < 0 || variant >= kOrderShapes) variant = 0;
  switch (sc.order) {
    case 2: return kWave1O2[variant].launch(d, sc, a, s);
    case 4: return kWave1Variants[variant].launch(d, sc, a, s);
    case 6: return kWave1O6[variant].launch(d, sc, a, s);
    case 8: return kWave1O8[variant].launch(d, sc, a, s);
    default: return set_error(CHEMORA_EUNSUPPORTED, "first-order wave of order %d is not compiled", sc.order);
  }
}

}  // namespace chemora
