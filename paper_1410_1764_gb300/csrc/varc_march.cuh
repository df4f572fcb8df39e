// Stage kernel of the variable-speed wave equation (u_t = rho, rho_t = s Lap u
// + sum_d G_d D_d u, s = c^2, G_d = D_d s) with its stencils on the integer
// units (star_march.cuh), shared by the Runge-Kutta driver and the adjoint's
// forward pass.  GB300, 128^3: 52 us per stage against 180 us in FP64 (45
// instructions); ten FP64 instructions are left (36 us), HBM alone takes 30.
// Each axis' values are aligned to their own largest exponent (to the star's, a
// first difference beside larger values along another axis lost digits: 51 us);
// one, two or three of the first differences through the conversion instruction:
// 55, 57, 59 us.
#pragma once
#include "internal.h"
#include "star_march.cuh"

namespace chemora {

// Store v at interior point (i, j, k) (offset c) of a grid function and, when
// `imaged`, also at each of its periodic images in the ghost zones (points
// within g of a face have one image per near face, and edge and corner
// images): the ghost zones are then valid without a fill pass.  Needs
// n >= g on every axis (each ghost point then has exactly one interior
// source), which the host checks before passing imaged = 1.
__device__ __forceinline__ void store_imaged(double* f, const Dims& d, int i, int j, int k, int64_t c, double v,
                                             int imaged) {
  f[c] = v;
  const int g = d.g;
  if (!imaged || (i >= g && i < d.nx - g && j >= g && j < d.ny - g && k >= g && k < d.nz - g)) return;
  // image a of an axis: 0 the point itself, 1 across the far face, 2 across the near one
  for (int e = 0; e < 3; ++e) {
    if ((e == 1 && k >= g) || (e == 2 && k < d.nz - g)) continue;
    const int64_t oz = e == 0 ? 0 : (e == 1 ? d.nz * d.sz : -(d.nz * d.sz));
    for (int b = 0; b < 3; ++b) {
      if ((b == 1 && j >= g) || (b == 2 && j < d.ny - g)) continue;
      const int64_t oy = b == 0 ? 0 : (b == 1 ? d.ny * d.sy : -(d.ny * d.sy));
      for (int a = 0; a < 3; ++a) {
        if ((a == 1 && i >= g) || (a == 2 && i < d.nx - g) || (a | b | e) == 0) continue;
        f[c + (a == 0 ? 0 : (a == 1 ? d.nx : -d.nx)) + oy + oz] = v;
      }
    }
  }
}

// What the integer units leave out: 12 h^2 Lap u and 12 h D_d u at p in FP64.
__device__ __forceinline__ void star2_fp64(const double* p, const Dims& d, double* lap, double (&t)[3]) {
  const int64_t st[3] = {1, d.sy, d.sz};
  const double c = p[0];
  *lap = 0.0;
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    const int64_t o = st[q];
    const double up1 = p[o], um1 = p[-o], up2 = p[2 * o], um2 = p[-2 * o];
    *lap += fma(16.0, (up1 - c) + (um1 - c), -((up2 - c) + (um2 - c)));
    const double v = fma(8.0, up1 - um1, -(up2 - um2));
    t[0] = q == 0 ? v : t[0];
    t[1] = q == 1 ? v : t[1];
    t[2] = q == 2 ? v : t[2];
  }
}

// One stage of the tile's columns.  coef: s and G_d, svar apart; tape (or NULL): Lap u and
// 12 h D_d u of the stage state, svar apart.
constexpr int kVarcThreads = 768;  // resident threads per SM
template <int TX, int TY>
__global__ void __launch_bounds__(TX * TY, kVarcThreads / (TX * TY))
varc_march_kernel(Dims d, double i12h, double i12h2, double one, double two, double mzero, StageParams a, int zb,
                  double* __restrict__ tape) {
  constexpr int R = 2, P = TX + 2 * R, K = 5;  // 18 x 2^58, the first differences, fits in 64 bits
  __shared__ long long pm[2][P * (TY + 2 * R)];
  __shared__ int pe[2][P * (TY + 2 * R)];
  const MarchPlace<TX, TY> p(d, zb);
  const MarchHalo<R, TX, TY> hl(p);
  const double* org = a.src + p.org;
  const int64_t own = (int64_t)p.ly * d.sy + p.lx;
  const int pc = (p.ly + R) * P + p.lx + R;
  fx::Parts z[5];
  double znext = 0.0, hnext[hl.n];
#pragma unroll
  for (int m = 0; m < 5; ++m) z[m] = fx::Parts{0, 0};
  if (p.active) {
#pragma unroll
    for (int m = 1; m < 5; ++m) z[m] = fx::parts_or_zero<K>(__ldg(org + own + (int64_t)(m - 3) * d.sz));
    znext = __ldg(org + own + 2 * d.sz);
  }
#pragma unroll
  for (int q = 0; q < hl.n; ++q) hnext[q] = hl.live[q] ? __ldg(org + (int64_t)hl.y[q] * d.sy + hl.x[q]) : 0.0;
  int64_t c = p.org + own;
#pragma unroll 1
  for (int k = 0; k < p.nz; ++k, c += d.sz, org += d.sz) {
    long long* const M = pm[k & 1];
    int* const E = pe[k & 1];
    MarchUpdate<2> up;
    double rho = 0.0, speed2 = 0.0, G[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int m = 0; m < 4; ++m) z[m] = z[m + 1];
    z[4] = fx::parts_or_zero<K>(znext);
    if (p.active) {
      M[pc] = z[2].m;
      E[pc] = z[2].e;
      rho = __ldg(a.src + d.sv + c);
      speed2 = __ldg(a.coef + c);
#pragma unroll
      for (int q = 0; q < 3; ++q) G[q] = __ldg(a.coef + (1 + q) * d.sv + c);
      up.load(a, c, d.sv);
      if (k + 1 < p.nz) znext = __ldg(org + own + 3 * d.sz);
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
    if (!p.active) continue;
    int x[3][4], ea[3], e = z[2].e;
    unsigned low = ~0u;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
#pragma unroll
      for (int q = 0; q < 4; ++q) x[ax][q] = ax == 2 ? z[2 + tap<R>(q)].e : E[pc + tap<R>(q) * (ax == 0 ? 1 : P)];
      ea[ax] = fx::emax(fx::emax(x[ax][0], x[ax][1]), fx::emax(x[ax][2], x[ax][3]));
      low = min(low, (unsigned)ea[ax]);  // (an axis of zeros, kZeroExp, is a large number)
      e = fx::emax(e, ea[ax]);
    }
    double lap = 0.0, t[3] = {0.0, 0.0, 0.0};
    if (low >= (unsigned)fx::kExpMin && star_ok<R>(e)) {
      // each axis' values to their own largest exponent, the pairs' sums then to the star's
      long long s[R] = {0, 0};
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        long long m[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) m[q] = ax == 2 ? z[2 + tap<R>(q)].m : M[pc + tap<R>(q) * (ax == 0 ? 1 : P)];
        const Axis4 f(m, x[ax], ea[ax]);
        t[ax] = fx::to_double<K>(f.diff, ea[ax]);
        s[0] += fx::sar(f.near, (unsigned)(e - ea[ax]));
        s[1] += fx::sar(f.far, (unsigned)(e - ea[ax]));
      }
      lap = star_lap<R, K>(s, fx::align(z[2], e), e);
    } else {
      star2_fp64(a.src + c, d, &lap, t);
    }
    lap = __fma_rn(lap, i12h2, mzero);
    const double adv = __fma_rn(G[2], t[2], __fma_rn(G[1], t[1], __fma_rn(G[0], t[0], mzero)));
    const double kk[2] = {rho, __fma_rn(speed2, lap, __fma_rn(adv, i12h, mzero))};
    const int i = p.x0 + p.lx, j = p.y0 + p.ly, kz = p.k0 + k;
    up.apply(a, c, d.sv, kk, one, two,
             [&](int64_t o, double x) { store_imaged(a.dst, d, i, j, kz, o, x, a.imaged); });
    if (tape) {
      tape[c] = lap;  // read at the point only
      // D_d u is read at stencil neighbours by the transposed stage
#pragma unroll
      for (int q = 0; q < 3; ++q) store_imaged(tape, d, i, j, kz, (1 + q) * d.sv + c, t[q], a.imaged);
    }
  }
}

template <int TX, int TY>
int launch_varc_march(const Dims& d, const Scalars& sc, const StageParams& a, double* tape, cudaStream_t s) {
  const int zb = march_depth(d, TX, TY, kVarcThreads / (TX * TY));
  varc_march_kernel<TX, TY><<<march_grid(d, TX, TY, zb), TX * TY, 0, s>>>(
      d, sc.i12h, sc.i12h2, sc.k[CHEMORA_K_ONE], sc.k[CHEMORA_K_TWO], sc.k[CHEMORA_K_MZERO], a, zb, tape);
  return launched("varc_march_kernel");
}

}  // namespace chemora
