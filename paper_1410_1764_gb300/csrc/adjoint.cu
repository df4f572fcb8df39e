// Discrete adjoint of the variable-speed wave equation under RK4: the exact
// transpose of the fully discrete map (the reverse-mode counterpart of the
// Jacobians Kranc generates, Sec. 3.2.1), hand-written.
//
// Forward:  u_t = rho,  rho_t = s Lap u + sum_d G_d D_d u,  G_d = D_d s,
//           s = c^2 (G_d computed once per call; periodic ghosts).
// Transpose of one right-hand side at a stage state y_q, for the cotangent
// kb = (kb_u, kb_rho) of its output, with w = kb_rho:
//   yhat_u   = Lap(s w) - sum_d D_d(G_d w)      (D_d^T = -D_d, Lap^T = Lap)
//   yhat_rho = kb_u
//   sbar    += w Lap u_q - sum_d D_d(w D_d u_q)
// Reverse RK4 step (stage 4 down to 1), from ybar' = cotangent of y_{n+1}:
//   kb_4 = dt/6 ybar';  yhat_q = J^T kb_q;  ybar_n = ybar' + sum_q yhat_q;
//   kb_3 = dt/3 ybar' + dt yhat_4;  kb_2 = dt/3 ybar' + dt/2 yhat_3;
//   kb_1 = dt/6 ybar' + dt/2 yhat_2.
// Checkpoints: y_n every ckpt_every steps.  Each segment but the newest is
// recomputed from its checkpoint with the forward kernel writing a tape
// (Lap u_q and D_d u_q for every stage), so the transpose kernel needs no
// derivatives of u; the newest segment's tape is written by the forward
// pass itself.
//
// Every product is formed at the neighbour points and then differenced, as the
// oracle's definition does; a point is written by one thread, so results are
// deterministic.
#include <math.h>
#include <string.h>

#include <vector>

#include "internal.h"
#include "varc_march.cuh"

namespace chemora {

constexpr int ATX = 32, ATY = 8;

__device__ __forceinline__ int64_t at_(const Dims& d, int i, int j, int k) {
  return (int64_t)(k + d.g) * d.sz + (int64_t)(j + d.g) * d.sy + (i + d.g);
}

// G_d = D_d s on the interior (3 grid functions).
__global__ void __launch_bounds__(ATX * ATY) varc_grad_s_kernel(Dims d, double i12h,
                                                                const double* __restrict__ s,
                                                                double* __restrict__ G) {
  const int i = blockIdx.x * ATX + threadIdx.x, j = blockIdx.y * ATY + threadIdx.y, k = blockIdx.z;
  if (i >= d.nx || j >= d.ny) return;
  const int64_t c = at_(d, i, j, k);
  const int64_t st[3] = {1, d.sy, d.sz};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const double* p = s + c;
    const double a = p[st[q]] - p[-st[q]];
    const double b = p[2 * st[q]] - p[-2 * st[q]];
    G[q * d.sv + c] = (8.0 * a - b) * i12h;
  }
}

// One transposed stage (see the file comment) on the tile's columns, marching
// through z.  The stencils act on the products s w, G_d w and w D_d u_q, formed
// once per point (and once more per halo cell) and differenced on the integer
// units (star_march.cuh): x and y neighbours come from the plane in shared
// memory, z neighbours from the thread's registers.  Six guard bits for the
// Laplacian: values cut off leave an error that adds up over the steps (with two
// bits grad_u0 of 24 steps on 64^3 was 18 % further from exact values than with
// FP64 sums).  Over 24 inputs (48 x 44 x 40, 12 steps) the errors' geometric means
// are 0.996 of FP64's for grad_u0 and 1.005 for grad_c, whose ratios scatter by 18 %.
//
// GB300, 128^3: 116 us, against 320 us when each point formed the 37 products
// of its stencils itself in FP64 (72 instructions of 17.8 cycles).  Products in
// FP64 here: 123 us.  640 threads per SM (20 bytes spilled): 7 % more.  Bound by
// the latency of its integer chains at 16 warps per SM; eleven FP64 instructions
// per point are left (40 us), HBM alone takes 47 us.
// kb: 2 grid functions with valid ghosts; coef: s and G_d (ghosts valid); tape:
// Lap u_q (interior) and 12 h D_d u_q (ghosts valid).  first: yacc = yp + yhat
// (else yacc += yhat).  kbn (if non-NULL): kbn = cq yp + aq yhat, or, after the
// step's last stage, cq yacc.
constexpr int kAdjThreads = 512;  // resident threads per SM
template <int TX, int TY>
__global__ void __launch_bounds__(TX * TY, kAdjThreads / (TX * TY))
varc_adj_march_kernel(Dims d, double i12h, double i12h2, double i144h2, const double* __restrict__ kb,
                      const double* __restrict__ coef, const double* __restrict__ tape,
                      const double* __restrict__ yp, double* __restrict__ yacc, double* __restrict__ kbn,
                      double* __restrict__ sbar, double cq, double aq, int first, int last, int zb,
                      double one, double mzero, int imaged) {
  constexpr int R = 2, P = TX + 2 * R;
  constexpr int KA = 6, KD = Guard<R>::d1;
  // s w with both halos; G_x w and w D_x u with the x halo; G_y w and w D_y u with the y halo
  constexpr int NA = P * (TY + 2 * R), NX = P * TY, NY = TX * (TY + 2 * R);
  __shared__ long long pm[2][NA + 2 * NX + 2 * NY];
  __shared__ int pe[2][NA + 2 * NX + 2 * NY];
  const MarchPlace<TX, TY> p(d, zb);
  const MarchHalo<R, TX, TY> hl(p);
  const int64_t own = (int64_t)p.ly * d.sy + p.lx;
  const int oa = (p.ly + R) * P + p.lx + R;
  const int ox = NA + p.ly * P + p.lx + R;                 // G_x w, then w D_x u NX further
  const int oy = NA + 2 * NX + (p.ly + R) * TX + p.lx;     // G_y w, then w D_y u NY further
  const double* w = kb + d.sv;                             // kb_rho
  const double* cz = coef + 3 * d.sv;                      // G_z
  const double* tz = tape + 3 * d.sv;
  auto mul = [&](double x, double y) { return __fma_rn(x, y, mzero); };
  fx::Parts za[5], zg[5], zt[5];  // s w, G_z w, w D_z u of the column
#pragma unroll
  for (int m = 0; m < 5; ++m) za[m] = zg[m] = zt[m] = fx::Parts{0, 0};
  int64_t c = p.org + own;
  if (p.active) {
#pragma unroll
    for (int m = 1; m < 5; ++m) {
      const int64_t o = c + (int64_t)(m - 3) * d.sz;
      const fx::Term<10> wv = fx::term<10>(__ldg(w + o));
      za[m] = fx::term_product<KA>(wv, fx::term<KA + 1>(__ldg(coef + o)));
      zg[m] = fx::term_product<KD>(wv, fx::term<KD + 1>(__ldg(cz + o)));
      zt[m] = fx::term_product<KD>(wv, fx::term<KD + 1>(__ldg(tz + o)));
    }
  }
#pragma unroll 1
  for (int k = 0; k < p.nz; ++k, c += d.sz) {
    long long* const M = pm[k & 1];
    int* const E = pe[k & 1];
    double wc = 0.0, kbu = 0.0, lapu = 0.0, y0 = 0.0, y1 = 0.0, a0 = 0.0, a1 = 0.0, sb = 0.0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      za[m] = za[m + 1];
      zg[m] = zg[m + 1];
      zt[m] = zt[m + 1];
    }
    auto put = [&](int o, const fx::Parts& v) {
      M[o] = v.m;
      E[o] = v.e;
    };
    if (p.active) {
      const int64_t o = c + 2 * d.sz;
      const double wz = __ldg(w + o), sz = __ldg(coef + o), gz = __ldg(cz + o), uz = __ldg(tz + o);
      wc = __ldg(w + c);
      const double gx = __ldg(coef + d.sv + c), gy = __ldg(coef + 2 * d.sv + c);
      const double ux = __ldg(tape + d.sv + c), uy = __ldg(tape + 2 * d.sv + c);
      kbu = __ldg(kb + c);
      lapu = __ldg(tape + c);
      y0 = __ldg(yp + c);
      y1 = __ldg(yp + d.sv + c);
      a0 = first ? y0 : yacc[c];
      a1 = first ? y1 : yacc[d.sv + c];
      sb = sbar[c];
      const fx::Term<10> fz = fx::term<10>(wz), fc = fx::term<10>(wc);
      za[4] = fx::term_product<KA>(fz, fx::term<KA + 1>(sz));
      zg[4] = fx::term_product<KD>(fz, fx::term<KD + 1>(gz));
      zt[4] = fx::term_product<KD>(fz, fx::term<KD + 1>(uz));
      put(oa, za[2]);
      put(ox, fx::term_product<KD>(fc, fx::term<KD + 1>(gx)));
      put(ox + NX, fx::term_product<KD>(fc, fx::term<KD + 1>(ux)));
      put(oy, fx::term_product<KD>(fc, fx::term<KD + 1>(gy)));
      put(oy + NY, fx::term_product<KD>(fc, fx::term<KD + 1>(uy)));
    }
#pragma unroll
    for (int q = 0; q < hl.n; ++q)
      if (hl.live[q]) {
        const int64_t o = p.org + k * d.sz + (int64_t)hl.y[q] * d.sy + hl.x[q];
        const int64_t ax = (hl.along_x[q] ? 1 : 2) * d.sv;
        const fx::Term<10> wv = fx::term<10>(__ldg(w + o));
        put((hl.y[q] + R) * P + hl.x[q] + R, fx::term_product<KA>(wv, fx::term<KA + 1>(__ldg(coef + o))));
        const int b = hl.along_x[q] ? NA + hl.y[q] * P + hl.x[q] + R : NA + 2 * NX + (hl.y[q] + R) * TX + hl.x[q];
        put(b, fx::term_product<KD>(wv, fx::term<KD + 1>(__ldg(coef + ax + o))));
        put(b + (hl.along_x[q] ? NX : NY), fx::term_product<KD>(wv, fx::term<KD + 1>(__ldg(tape + ax + o))));
      }
    __syncthreads();
    if (!p.active) continue;
    double lap = 0.0, div[2] = {0.0, 0.0};  // of s w; of G_d w and of w D_d u
    {
      int ex[4], ey[4], e = za[2].e;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        ex[m] = E[oa + tap<R>(m)];
        ey[m] = E[oa + tap<R>(m) * P];
        e = fx::emax(e, fx::emax(fx::emax(ex[m], ey[m]), za[2 + tap<R>(m)].e));
      }
      if (!star_ok<R>(e)) {
        const int64_t st[3] = {1, d.sy, d.sz};
        const double t0 = mul(coef[c], w[c]);
#pragma unroll 1
        for (int q = 0; q < 3; ++q)
          for (int m = 1; m <= 2; ++m) {
            const int64_t o = m * st[q];
            const double v = (coef[c + o] * w[c + o] - t0) + (coef[c - o] * w[c - o] - t0);
            lap = __fma_rn(m == 1 ? 16.0 : -1.0, v, lap);
          }
      } else if (e != fx::kZeroExp) {
        long long s2[R] = {0, 0};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int o = tap<R>(m), q = o < 0 ? -o - 1 : o - 1;
          s2[q] += fx::sar(M[oa + o], (unsigned)(e - ex[m])) + fx::sar(M[oa + o * P], (unsigned)(e - ey[m])) +
                   fx::align(za[2 + o], e);
        }
        lap = star_lap<R, KA>(s2, fx::align(za[2], e), e);
      }
    }
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const int bx = ox + f * NX, by = oy + f * NY;
      int ex[4], ey[4], e = fx::kZeroExp;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        ex[m] = E[bx + tap<R>(m)];
        ey[m] = E[by + tap<R>(m) * TX];
        e = fx::emax(e, fx::emax(fx::emax(ex[m], ey[m]), (f ? zt : zg)[2 + tap<R>(m)].e));
      }
      if (!star_ok<R>(e)) {
        const int64_t st[3] = {1, d.sy, d.sz};
        double v = 0.0;
#pragma unroll 1
        for (int q = 0; q < 3; ++q) {
          const double* g = (f ? tape : coef) + (1 + q) * d.sv + c;
          const double* wv = w + c;
          for (int m = 1; m <= 2; ++m) {
            const int64_t o = m * st[q];
            v = __fma_rn(m == 1 ? 8.0 : -1.0, g[o] * wv[o] - g[-o] * wv[-o], v);
          }
        }
        div[f] = v;
      } else if (e != fx::kZeroExp) {
        long long t[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int u1 = R + q, dn = R - 1 - q, o = q + 1;
          const fx::Parts& zu = (f ? zt : zg)[2 + o];
          const fx::Parts& zd = (f ? zt : zg)[2 - o];
          t[q] = (fx::sar(M[bx + o], (unsigned)(e - ex[u1])) - fx::sar(M[bx - o], (unsigned)(e - ex[dn]))) +
                 (fx::sar(M[by + o * TX], (unsigned)(e - ey[u1])) - fx::sar(M[by - o * TX], (unsigned)(e - ey[dn]))) +
                 (fx::align(zu, e) - fx::align(zd, e));
        }
        div[f] = star_d1<R>(t, e);
      }
    }
    const double yh = __fma_rn(div[0], -i12h, mul(lap, i12h2));
    // the terms first: one rounding per stage at the size of the sum
    sbar[c] = __fma_rn(__fma_rn(wc, lapu, mul(div[1], -i144h2)), one, sb);
    a0 = __fma_rn(yh, one, a0);
    a1 = __fma_rn(kbu, one, a1);
    yacc[c] = a0;
    yacc[d.sv + c] = a1;
    if (kbn) {  // the next transposed stage reads kb at stencil neighbours
      const int i = p.x0 + p.lx, j = p.y0 + p.ly, kz = p.k0 + k;
      double n0 = mul(cq, last ? a0 : y0), n1 = mul(cq, last ? a1 : y1);
      if (!last) {
        n0 = __fma_rn(aq, yh, n0);
        n1 = __fma_rn(aq, kbu, n1);
      }
      store_imaged(kbn, d, i, j, kz, c, n0, imaged);
      store_imaged(kbn, d, i, j, kz, d.sv + c, n1, imaged);
    }
  }
}

// kb = w ybar' (both components, interior; with its ghost images when imaged)
__global__ void scale_state_kernel(Dims d, double w, const double* __restrict__ y, double* __restrict__ out,
                                   int imaged) {
  const int i = blockIdx.x * ATX + threadIdx.x, j = blockIdx.y * ATY + threadIdx.y, k = blockIdx.z;
  if (i >= d.nx || j >= d.ny) return;
  const int64_t c = at_(d, i, j, k);
  store_imaged(out, d, i, j, k, c, __dmul_rn(w, y[c]), imaged);
  store_imaged(out, d, i, j, k, d.sv + c, __dmul_rn(w, y[d.sv + c]), imaged);
}

// Loss J = 1/2 sum (u[r] - data_r)^2 and the seed ybar_u[r] += u[r] - data_r.
// One block; a fixed tree reduction keeps the loss deterministic.
__global__ void receivers_kernel(const double* __restrict__ u, const int64_t* __restrict__ recv,
                                 const double* __restrict__ data, int nrecv, double* ybar_u,
                                 double* loss) {
  __shared__ double red[1024];
  double acc = 0.0;
  for (int r = threadIdx.x; r < nrecv; r += blockDim.x) {
    const double m = u[recv[r]] - data[r];
    acc += 0.5 * m * m;
    atomicAdd(ybar_u + recv[r], m);
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = red[0];
}

// grad_c = 2 c sbar on the interior, ghosts of grad_c zero.
__global__ void grad_c_kernel(Dims d, const double* __restrict__ c, const double* __restrict__ sbar,
                              double* __restrict__ gc) {
  const int i = blockIdx.x * ATX + threadIdx.x, j = blockIdx.y * ATY + threadIdx.y, k = blockIdx.z;
  if (i >= d.nx || j >= d.ny) return;
  const int64_t p = at_(d, i, j, k);
  gc[p] = 2.0 * c[p] * sbar[p];
}

// s = c^2 on the interior
__global__ void adj_square_kernel(Dims d, const double* __restrict__ c, double* __restrict__ s) {
  const int i = blockIdx.x * ATX + threadIdx.x, j = blockIdx.y * ATY + threadIdx.y, k = blockIdx.z;
  if (i >= d.nx || j >= d.ny) return;
  const int64_t p = at_(d, i, j, k);
  s[p] = c[p] * c[p];
}

// out = in on the interior of nv grid functions
__global__ void copy_interior_kernel(Dims d, int nv, const double* __restrict__ in, double* __restrict__ out) {
  const int i = blockIdx.x * ATX + threadIdx.x, j = blockIdx.y * ATY + threadIdx.y, k = blockIdx.z;
  if (i >= d.nx || j >= d.ny) return;
  const int64_t p = at_(d, i, j, k);
  for (int v = 0; v < nv; ++v) out[v * d.sv + p] = in[v * d.sv + p];
}

static dim3 agrid(const Dims& d) { return dim3((d.nx + ATX - 1) / ATX, (d.ny + ATY - 1) / ATY, d.nz); }

int launch_varc_grad(const Dims& d, double i12h, const double* s, double* G, cudaStream_t st) {
  varc_grad_s_kernel<<<agrid(d), dim3(ATX, ATY), 0, st>>>(d, i12h, s, G);
  return launched("varc_grad_s_kernel");
}

struct AdjBufs {
  double *s, *G,  // G right behind s
       *Y, *ck, *tape, *yp, *yacc, *kb, *kbn, *sbar, *loss;
  int64_t* recv;
  double* data;
};

// One forward RK4 step of the variable-speed wave from Y to Ynext (which may
// be Y), tape of the 4 stages written at tape (16 grid functions) when
// non-NULL.
static int fwd_step(chemora_system* sys, const AdjBufs& B, double* Y, double* Ynext, double dt, double* tape,
                    cudaStream_t s) {
  const Dims& d = sys->grid->d;
  const int im = imaged_ok(d);
  const size_t fs = sys->grid->fsize;
  double* A = sys->scratch;
  double* Sa = sys->scratch + 2 * fs;
  double* Sb = sys->scratch + 4 * fs;
  StageParams p{};
  int rc;
  double* srcs[4] = {Y, Sa, Sb, Sa};
  double* dsts[4] = {Sa, Sb, Sa, Ynext};
  const double c2[4] = {0.5 * dt, 0.5 * dt, dt, 0.0};
  for (int q = 0; q < 4; ++q) {
    if (!im && (rc = fill_ghosts(d, 2, srcs[q], s))) return rc;
    p.src = srcs[q]; p.yn = Y; p.acc = A; p.dst = dsts[q]; p.c1 = dt / 6.0; p.c2 = c2[q]; p.mode = q + 1;
    p.coef = B.s;
    p.imaged = im;
    if ((rc = launch_varc_march<32, 4>(d, sys->sc, p, tape ? tape + (size_t)q * 4 * fs : nullptr, s))) return rc;
  }
  return im ? CHEMORA_OK : fill_ghosts(d, 2, Ynext, s);
}

// One reverse RK4 step: on entry B.yp holds ybar' and, unless it is the first,
// B.kb dt/6 ybar'; on exit B.yacc holds ybar_n and, unless it is the last, B.kb
// dt/6 ybar_n.
static int rev_step(chemora_system* sys, const AdjBufs& B, const double* tape, double dt, bool first_step,
                    bool last_step, cudaStream_t s) {
  const Dims& d = sys->grid->d;
  const size_t fs = sys->grid->fsize;
  const double i12h = sys->sc.i12h, i12h2 = sys->sc.i12h2;
  constexpr int ADJX = 32, ADJY = 4;
  const int im = imaged_ok(d), zb = march_depth(d, ADJX, ADJY, kAdjThreads / (ADJX * ADJY));
  int rc;
  if (first_step) {
    scale_state_kernel<<<agrid(d), dim3(ATX, ATY), 0, s>>>(d, dt / 6.0, B.yp, B.kb, im);
    if ((rc = launched("scale_state_kernel"))) return rc;
  }
  const double cq[4] = {dt / 6.0, dt / 6.0, dt / 3.0, dt / 3.0};  // weight of ybar' in kb_{q-1} (of ybar_n: q = 0)
  const double aq[4] = {0.0, 0.5 * dt, 0.5 * dt, dt};        // a_q dt
  double* kb = B.kb;
  double* kbn = B.kbn;
  for (int q = 3; q >= 0; --q) {
    if (!im && (rc = fill_ghosts(d, 2, kb, s))) return rc;
    varc_adj_march_kernel<ADJX, ADJY><<<march_grid(d, ADJX, ADJY, zb), ADJX * ADJY, 0, s>>>(
        d, i12h, i12h2, sys->sc.i144h2, kb, B.s, tape + (size_t)q * 4 * fs, B.yp, B.yacc,
        q > 0 || !last_step ? kbn : nullptr, B.sbar, cq[q], aq[q], q == 3 ? 1 : 0, q == 0 ? 1 : 0, zb, sys->sc.k[CHEMORA_K_ONE], sys->sc.k[CHEMORA_K_MZERO], im);
    if ((rc = launched("varc_adj_march_kernel"))) return rc;
    double* t = kb;
    kb = kbn;
    kbn = t;
  }
  return CHEMORA_OK;
}

}  // namespace chemora

using namespace chemora;

extern "C" int chemora_adjoint_rk4(chemora_system* sys, const double* state0, const double* c,
                                   double dt, int nsteps, int ckpt_every, const int64_t* recv_idx,
                                   int nrecv, const double* data, double* loss, double* grad_state0,
                                   double* grad_c, void* stream) {
  if (!is_handle(sys, H_SYSTEM)) return set_error(CHEMORA_EINVAL, "not a system handle");
  if (sys->kind != CHEMORA_WAVE_VARC)
    return set_error(CHEMORA_EINVAL, "chemora_adjoint_rk4 needs a CHEMORA_WAVE_VARC system");
  if (!state0 || !c || !recv_idx || !data || !loss || !grad_state0 || !grad_c)
    return set_error(CHEMORA_EINVAL, "NULL argument");
  if (nsteps < 1 || ckpt_every < 1 || nrecv < 1 || !isfinite(dt))
    return set_error(CHEMORA_EINVAL, "need nsteps >= 1, ckpt_every >= 1, nrecv >= 1, finite dt");
  const Dims& d = sys->grid->d;
  const size_t fs = sys->grid->fsize;
  for (int r = 0; r < nrecv; ++r) {
    const int64_t p = recv_idx[r];
    if (p < 0 || p >= (int64_t)fs) return set_error(CHEMORA_EINVAL, "receiver %d outside the grid", r);
    const int64_t k = p / d.sz, j = (p % d.sz) / d.sy, i = p % d.sy;
    if (i < d.g || i >= d.g + d.nx || j < d.g || j >= d.g + d.ny || k < d.g || k >= d.g + d.nz)
      return set_error(CHEMORA_EINVAL, "receiver %d (index %lld) is not an interior point", r,
                       (long long)p);
  }
  int rc = ensure_scratch(sys);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const int K = ckpt_every < nsteps ? ckpt_every : nsteps;
  const int nck = (nsteps + K - 1) / K;
  // fields: s 1, G 3, Y 2, ck 2 nck, tape 16 K, yp 2, yacc 2, kb 2, kbn 2, sbar 1, loss
  const size_t nfields = 1 + 3 + 2 + 2 * (size_t)nck + 16 * (size_t)K + 2 + 2 + 2 + 2 + 1;
  const size_t bytes = (nfields * fs + 32) * sizeof(double) + (size_t)nrecv * (sizeof(int64_t) + sizeof(double));
  char* buf = nullptr;
  // from the device's pool: from CUDA's default one, which gives freed memory
  // back at each synchronisation, 3.4 GB cost about 10 ms a call
  const cudaError_t e = pool_alloc((void**)&buf, bytes, s);
  if (e != cudaSuccess)
    return set_error(CHEMORA_ENOMEM, "adjoint work space of %zu bytes: %s", bytes, cudaGetErrorString(e));
  AdjBufs B;
  double* q = (double*)buf;
  B.s = q; q += fs;
  B.G = q; q += 3 * fs;
  B.Y = q; q += 2 * fs;
  B.ck = q; q += 2 * (size_t)nck * fs;
  B.tape = q; q += 16 * (size_t)K * fs;
  B.yp = q; q += 2 * fs;
  B.yacc = q; q += 2 * fs;
  B.kb = q; q += 2 * fs;
  B.kbn = q; q += 2 * fs;
  B.sbar = q; q += fs;
  B.loss = q; q += 32;
  B.recv = (int64_t*)q;
  B.data = (double*)(B.recv + nrecv);

  auto run = [&]() -> int {
    int r;
    CHEMORA_CUDA(cudaMemsetAsync(B.yp, 0, 2 * fs * sizeof(double), s));
    CHEMORA_CUDA(cudaMemsetAsync(B.sbar, 0, fs * sizeof(double), s));
    CHEMORA_CUDA(cudaMemcpyAsync(B.recv, recv_idx, nrecv * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    CHEMORA_CUDA(cudaMemcpyAsync(B.data, data, nrecv * sizeof(double), cudaMemcpyHostToDevice, s));
    // s = c^2 with ghosts; G = D s with ghosts
    adj_square_kernel<<<agrid(d), dim3(ATX, ATY), 0, s>>>(d, c, B.s);
    if ((r = launched("adj_square_kernel"))) return r;
    if ((r = fill_ghosts(d, 1, B.s, s))) return r;
    if ((r = launch_varc_grad(d, sys->sc.i12h, B.s, B.G, s))) return r;
    if ((r = fill_ghosts(d, 3, B.G, s))) return r;
    // forward pass with checkpoints; the newest segment's steps write their
    // tape here (the same kernel on the same states as a recomputation), so
    // the reverse sweep recomputes only the older segments
    const int nlast = (nck - 1) * K;
    auto ckpt = [&](int q) { return B.ck + (size_t)q * 2 * fs; };
    double* y = ckpt(0);
    CHEMORA_CUDA(cudaMemcpyAsync(y, state0, 2 * fs * sizeof(double), cudaMemcpyDeviceToDevice, s));
    if ((r = fill_ghosts(d, 2, y, s))) return r;
    for (int n = 0; n < nsteps; ++n) {
      double* tp = n >= nlast ? B.tape + (size_t)(n - nlast) * 16 * fs : nullptr;
      double* next = (n + 1) % K == 0 && n + 1 < nsteps ? ckpt((n + 1) / K) : B.Y;
      if ((r = fwd_step(sys, B, y, next, dt, tp, s))) return r;
      y = next;
    }
    // loss and seed
    receivers_kernel<<<1, 1024, 0, s>>>(y, B.recv, B.data, nrecv, B.yp, B.loss);
    if ((r = launched("receivers_kernel"))) return r;
    // reverse sweep, newest segment first
    for (int sg = nck - 1; sg >= 0; --sg) {
      const int n0 = sg * K, n1 = (n0 + K < nsteps) ? n0 + K : nsteps;
      if (sg < nck - 1) {
        y = ckpt(sg);
        for (int n = n0; n < n1; ++n) {
          if ((r = fwd_step(sys, B, y, B.Y, dt, B.tape + (size_t)(n - n0) * 16 * fs, s))) return r;
          y = B.Y;
        }
      }
      // the tape's D_d u fields are read at stencil neighbours: periodic
      // ghosts (written with their images by the forward kernel when it can)
      if (!imaged_ok(d) && (r = fill_ghosts(d, 16 * (n1 - n0), B.tape, s))) return r;
      for (int n = n1 - 1; n >= n0; --n) {
        if ((r = rev_step(sys, B, B.tape + (size_t)(n - n0) * 16 * fs, dt, n == nsteps - 1, n == 0, s))) return r;
        double* t = B.yp;
        B.yp = B.yacc;
        B.yacc = t;
      }
    }
    // outputs
    CHEMORA_CUDA(cudaMemsetAsync(grad_state0, 0, 2 * fs * sizeof(double), s));
    CHEMORA_CUDA(cudaMemsetAsync(grad_c, 0, fs * sizeof(double), s));
    copy_interior_kernel<<<agrid(d), dim3(ATX, ATY), 0, s>>>(d, 2, B.yp, grad_state0);
    if ((r = launched("copy_interior_kernel"))) return r;
    grad_c_kernel<<<agrid(d), dim3(ATX, ATY), 0, s>>>(d, c, B.sbar, grad_c);
    if ((r = launched("grad_c_kernel"))) return r;
    CHEMORA_CUDA(cudaMemcpyAsync(loss, B.loss, sizeof(double), cudaMemcpyDeviceToHost, s));
    return CHEMORA_OK;
  };
  rc = run();
  pool_free(buf, s);
  cudaError_t e2 = cudaStreamSynchronize(s);
  if (rc) return rc;
  if (e2 != cudaSuccess) return cuda_error(e2, "cudaStreamSynchronize(adjoint)");
  return CHEMORA_OK;
}
