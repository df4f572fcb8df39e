// The split BSSN right-hand side (bssn_fields.cuh): the derivative-field
// kernel, the algebra kernels for one grid and for work-lists over many
// regions (batched patches, refined boxes), and the constraints.
#include <algorithm>

#include "internal.h"
#include "bssn_algebra.cuh"
#include "bssn_split.h"
#include "star_march.cuh"
#include "generated/gen_bssn_constraints_alg.cuh"

namespace chemora {

// ---------------------------------------------------------------------------
// derivative fields
// ---------------------------------------------------------------------------
constexpr int kTileThreads = 256, kTileRows = 32;
constexpr int kRowMax = 448;    // (tw + 4) x (th + 4) of every tile shape tile_shape() returns
constexpr int kPlaneMax = 532;  // (tw + 6) x (th + 6)
constexpr int kGuard = 4;       // guard bits: an axis' weights add up to 64 in magnitude, 64 x 2^57 fits

// One block: one variable (blockIdx.y) on a tile of tw x th columns, marching
// through zb planes, a point per thread and plane.  Each value is taken apart
// into integers once: a thread keeps its column's seven values in registers,
// the plane in hand lies in shared memory (significands and exponents) with
// its halo, so a tap costs a shift and an addition.  An axis' differences are
// aligned to its own largest exponent (to the star's, they lost digits beside
// larger values along another axis), the dissipation to the star's.  First differences go back to doubles through the conversion
// instruction, the others by integer operations, which shares the work
// between the two pipes.  The mixed derivatives are first-derivative stencils
// of the neighbours' first-derivative rows, in FP64 (three fmas each: fewer
// cycles than their 16 points in integers); the rows pass through shared
// memory, those past the tile's edge are computed by the block again.
//
// GB300, all 24 variables of 128 x 128 x 64 points: 578 us (the field writes
// alone take 200 us of HBM time).  With every value aligned to the star's
// largest exponent 546 us, and then: each value taken apart by each of its 19
// readers, no march: 846 us; conversion instruction for every difference 603,
// for none 572 us; two or four blocks per SM 637, 708 us; significand and
// exponent in one 16-byte cell 621 us; one kernel for both sorts of variable
// 580 us.  Bound by its FP64 pipe (70 % busy for variables with second
// derivatives) and the latency of its chains at 23 warps per SM (2.1 instructions
// per clock).
template <bool DD>
__global__ void __launch_bounds__(kTileThreads, 3)
bssn_fields_kernel(const FieldRegion* __restrict__ regions, FieldRegion one_region, const int2* __restrict__ tiles,
                   const double* __restrict__ base, double* __restrict__ work, double one, double eight) {
  __shared__ long long pm[2][kPlaneMax];
  __shared__ int pe[2][kPlaneMax];
  __shared__ double row_y[kRowMax], row_z[kRowMax];
  int tile = blockIdx.x, region = 0;
  if (tiles) {
    const int2 q = tiles[blockIdx.x];
    region = q.x;
    tile = q.y;
  }
  const FieldRegion R = regions ? regions[region] : one_region;
  const Dims& d = R.d;
  // the DD kernel takes the variables with second derivatives, the other the rest
  const int v = DD ? (blockIdx.y < 7 ? blockIdx.y : blockIdx.y + 10)
                   : (blockIdx.y < 10 ? blockIdx.y + 7 : blockIdx.y + 11);
  const int ddi = blockIdx.y;
  const int txy = tile % (R.tnx * R.tny), k0 = (tile / (R.tnx * R.tny)) * R.zb;
  const int x0 = (txy % R.tnx) * R.tw, y0 = (txy / R.tnx) * R.th;
  const int w = min(R.tw, d.nx - x0), h = min(R.th, d.ny - y0), nz = min(R.zb, d.nz - k0);
  const int t = threadIdx.x, ly = t / R.tw, lx = t - ly * R.tw;
  const bool active = lx < w && ly < h;
  const double* org = base + R.offset + v * d.sv + (int64_t)(k0 + d.g) * d.sz + (int64_t)(y0 + d.g) * d.sy + x0 + d.g;
  const double* col = org + (int64_t)ly * d.sy + lx;
  const int pp = R.tw + 6, pc = (ly + 3) * pp + lx + 3;  // plane pitch, this point
  const int rp = R.tw + 4;                               // row pitch
  // this thread's halo cell: columns -3..-1, w..w+2 of the tile's rows, then
  // rows -3..-1, h..h+2
  const bool halo = t < 6 * (w + h);
  int hx = 0, hy = 0;
  if (t < 6 * h) {
    const int e = t / h;
    hy = t - e * h;
    hx = e < 3 ? e - 3 : w + e - 3;
  } else if (halo) {
    const int e = (t - 6 * h) / w;
    hx = t - 6 * h - e * w;
    hy = e < 3 ? e - 3 : h + e - 3;
  }
  const double* hp = org + (int64_t)hy * d.sy + hx;
  const int hc = (hy + 3) * pp + hx + 3;
  fx::Parts z[7];
  double znext = 0.0, hnext = 0.0;
#pragma unroll
  for (int m = 0; m < 7; ++m) z[m] = fx::Parts{0, 0};
  if (active) {
#pragma unroll
    for (int m = 1; m < 7; ++m) z[m] = fx::parts_or_zero<kGuard>(__ldg(col + (int64_t)(m - 4) * d.sz));
    znext = __ldg(col + 3 * d.sz);
  }
  if (halo) hnext = __ldg(hp);
  int64_t point = R.w0 + ((int64_t)k0 * d.ny + y0 + ly) * d.nx + x0 + lx;
#pragma unroll 1
  for (int k = 0; k < nz; ++k) {
    long long* const M = pm[k & 1];
    int* const E = pe[k & 1];
#pragma unroll
    for (int m = 0; m < 6; ++m) z[m] = z[m + 1];
    z[6] = fx::parts_or_zero<kGuard>(znext);
    if (active) {
      M[pc] = z[3].m;
      E[pc] = z[3].e;
    }
    if (halo) {
      const fx::Parts q = fx::parts_or_zero<kGuard>(hnext);
      M[hc] = q.m;
      E[hc] = q.e;
      if (k + 1 < nz) hnext = __ldg(hp + (int64_t)(k + 1) * d.sz);
    }
    if (active && k + 1 < nz) znext = __ldg(col + (int64_t)(k + 4) * d.sz);
    __syncthreads();
    double* out = work + field_base(point);
    point += (int64_t)d.nx * d.ny;
    if (active) {
      // each axis' largest exponent over the offsets -2, -1, 1, 2, and the star's
      int x[3][6], ea[3], e = z[3].e;
      unsigned low = (unsigned)e;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int m = 0; m < 6; ++m) {
          const int o = m < 3 ? m - 3 : m - 2;
          x[a][m] = a == 2 ? z[3 + o].e : E[pc + o * (a == 0 ? 1 : pp)];
        }
        ea[a] = fx::emax(fx::emax(x[a][1], x[a][2]), fx::emax(x[a][3], x[a][4]));
        e = fx::emax(e, fx::emax(ea[a], fx::emax(x[a][0], x[a][5])));
        low = min(low, (unsigned)ea[a]);  // (zeros, kZeroExp, are a large number)
      }
      double d1[3], d2[3], ko = 0.0;
      if (low >= (unsigned)fx::kExpMin && (e == fx::kZeroExp || fx::in_range(e))) {
        long long kq = 0;  // the dissipation's weights add up to 192: its sum in quarters and their remainders
        int kr = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          long long f[6];
          int xa[4];
#pragma unroll
          for (int m = 0; m < 6; ++m) {
            const int o = m < 3 ? m - 3 : m - 2;
            f[m] = a == 2 ? z[3 + o].m : M[pc + o * (a == 0 ? 1 : pp)];
          }
          const long long g[4] = {f[1], f[2], f[3], f[4]};
#pragma unroll
          for (int m = 0; m < 4; ++m) xa[m] = x[a][m + 1];
          const Axis4 s(g, xa, ea[a]);
          d1[a] = fx::to_double_cvt<kGuard>(s.diff, ea[a]);
          if (DD) {
            const int ec = fx::emax(ea[a], z[3].e);
            d2[a] = fx::to_double<kGuard>(
                fx::sar(16 * s.near - s.far, (unsigned)(ec - ea[a])) - 30 * fx::align(z[3], ec), ec);
          }
          const long long k = fx::sar(15 * s.near - 6 * s.far, (unsigned)(e - ea[a])) +
                              fx::sar(f[0], (unsigned)(e - x[a][0])) + fx::sar(f[5], (unsigned)(e - x[a][5]));
          kq += k >> 2;
          kr += (int)k & 3;
        }
        kq += (kr >> 2) - 15 * fx::align(z[3], e);
        const bool wide = (unsigned long long)(kq + (1ll << 59)) >> 60 != 0;
        ko = fx::to_double<kGuard>(wide ? kq : 4 * kq + (kr & 3), wide ? e + 2 : e);
      } else {
        // the ends of the FP64 range, Inf, NaN
        const int64_t st[3] = {1, d.sy, d.sz};
        const double* p = col + (int64_t)k * d.sz;
        const double c = __ldg(p);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          double n[6];
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            n[2 * m] = __ldg(p + (m + 1) * st[a]);
            n[2 * m + 1] = __ldg(p - (m + 1) * st[a]);
          }
          const double c1 = (n[0] - c) + (n[1] - c), c2 = (n[2] - c) + (n[3] - c), c3 = (n[4] - c) + (n[5] - c);
          d1[a] = fma(8.0, n[0] - n[1], -(n[2] - n[3]));
          d2[a] = fma(16.0, c1, -c2);
          ko += fma(15.0, c1, fma(-6.0, c2, c3));
        }
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) out[(kFieldD1 + 3 * v + a) * kFieldBlock] = d1[a];
      out[(kFieldKo + v) * kFieldBlock] = ko;
      if (DD) {
#pragma unroll
        for (int a = 0; a < 3; ++a) out[(kFieldD2 + 6 * ddi + a) * kFieldBlock] = d2[a];
        row_y[ly * rp + lx + 2] = d1[1];
        row_z[(ly + 2) * rp + lx + 2] = d1[2];
      }
    }
    if constexpr (DD) {
      // rows past the edge: columns -2, -1, w, w+1 (y and z rows), then rows
      // -2, -1, h, h+1 (z rows)
      for (int q = t; q < 8 * h + 4 * w; q += kTileThreads) {
        const double* src = org + (int64_t)k * d.sz;
        if (q < 8 * h) {
          const int e = q / h, r = q - e * h, x = (e & 3) < 2 ? (e & 3) - 2 : w + (e & 3) - 2;
          const double* p = src + (int64_t)r * d.sy + x;
          if (e < 4)
            row_y[r * rp + x + 2] = d1_row_fp64(p, d.sy, one, eight);
          else
            row_z[(r + 2) * rp + x + 2] = d1_row_fp64(p, d.sz, one, eight);
        } else {
          const int e = (q - 8 * h) / w, x = q - 8 * h - e * w, y = e < 2 ? e - 2 : h + e - 2;
          row_z[(y + 2) * rp + x + 2] = d1_row_fp64(src + (int64_t)y * d.sy + x, d.sz, one, eight);
        }
      }
      __syncthreads();
      if (active) {
        auto mixed = [&](const double* r, int st) {
          const double q1 = fma(r[-st], -one, r[st]), q2 = fma(r[-2 * st], -one, r[2 * st]);
          return fma(eight, q1, -q2);
        };
        const double* ry = row_y + ly * rp + lx + 2;
        const double* rz = row_z + (ly + 2) * rp + lx + 2;
        out[(kFieldD2 + 6 * ddi + 3) * kFieldBlock] = mixed(ry, 1);
        out[(kFieldD2 + 6 * ddi + 4) * kFieldBlock] = mixed(rz, 1);
        out[(kFieldD2 + 6 * ddi + 5) * kFieldBlock] = mixed(rz, rp);
      }
    }
  }
}

// Tiles of nearly equal shape, at most 32 wide, at most 256 points, so that
// ragged grids leave few threads idle; 16 planes deep where that leaves enough
// blocks to fill the GPU, else fewer.
static void tile_shape(FieldRegion* R) {
  const Dims& d = R->d;
  R->tnx = (d.nx + 31) / 32;
  R->tw = (d.nx + R->tnx - 1) / R->tnx;
  const int rows = std::min(kTileRows, kTileThreads / R->tw);
  R->tny = (d.ny + rows - 1) / rows;
  R->th = (d.ny + R->tny - 1) / R->tny;
  int zb = 16;
  while (zb > 4 && (int64_t)R->tnx * R->tny * ((d.nz + zb - 1) / zb) * 24 < 4 * 152) zb /= 2;
  const int nseg = (d.nz + zb - 1) / zb;
  R->zb = (d.nz + nseg - 1) / nseg;
}

static int64_t region_tiles(const FieldRegion& R) { return (int64_t)R.tnx * R.tny * ((R.d.nz + R.zb - 1) / R.zb); }

FieldRegion field_region(const Dims& d, int64_t offset, int64_t w0) {
  FieldRegion R;
  R.d = d;
  R.offset = offset;
  R.npts = (int64_t)d.nx * d.ny * d.nz;
  R.w0 = w0;
  tile_shape(&R);
  return R;
}

// Planes of d that fit in `cap` workspace points (at least one).
static int chunk_planes(const Dims& d, int64_t cap) {
  const int64_t plane = (int64_t)d.nx * d.ny;
  return (int)std::min<int64_t>(d.nz, std::max<int64_t>(1, cap / plane));
}

int64_t field_work_points(const Dims& d, int64_t cap) { return (int64_t)d.nx * d.ny * chunk_planes(d, cap); }

int field_chunk_planes(const Dims& d, const FieldWork& work) {
  const int planes = chunk_planes(d, work.points);
  return (int64_t)d.nx * d.ny * planes <= work.points ? planes : 0;
}

size_t field_work_bytes(int64_t points) {
  return (size_t)((points + kFieldBlock - 1) / kFieldBlock) * kFields * kFieldBlock * sizeof(double);
}

// FP64 instructions of the field kernels per point of d: a conversion per first
// difference, three fmas per mixed derivative and per row past a tile's edge.
double field_fp64_instr(const Dims& d) {
  const FieldRegion R = field_region(d, 0, 0);
  return 24 * 3 + 11 * 3 * (3.0 + (8.0 * R.th + 4.0 * R.tw) / ((double)R.tw * R.th));
}

static int launch_field_kernels(const FieldRegion* regions, const FieldRegion& R, const int2* tiles, unsigned ntiles,
                                int nvars, const double* src, double* work, const Scalars& sc, cudaStream_t s) {
  // 24 variables: 11 with second derivatives, 13 without; the constraints' 17: 7 and 10
  const unsigned ndd = nvars == 24 ? 11 : 7, nd = nvars - ndd;
  bssn_fields_kernel<true><<<dim3(ntiles, ndd), kTileThreads, 0, s>>>(regions, R, tiles, src, work,
                                                                     sc.k[CHEMORA_K_ONE], sc.k[CHEMORA_K_EIGHT]);
  bssn_fields_kernel<false><<<dim3(ntiles, nd), kTileThreads, 0, s>>>(regions, R, tiles, src, work,
                                                                     sc.k[CHEMORA_K_ONE], sc.k[CHEMORA_K_EIGHT]);
  return launched("bssn_fields_kernel", 2);
}

int launch_fields(const FieldRegion& R, int nvars, const double* src, double* work, const Scalars& sc,
                         cudaStream_t s) {
  const unsigned n = (unsigned)region_tiles(R);
  return launch_field_kernels(nullptr, R, nullptr, n, nvars, src, work, sc, s);
}

// ---------------------------------------------------------------------------
// algebra, one region
// ---------------------------------------------------------------------------
// MODE: the RK stage mode, compiled in (modes 2 and 3 are the same update).
template <int BLK, int MINB, int MODE>
__global__ void __launch_bounds__(BLK, MINB)
bssn_algebra_kernel(FieldRegion R, Scalars sc, StageParams a_in, const double* __restrict__ work) {
  StageParams a = a_in;
  a.mode = MODE;
  bssn_algebra<BLK>(R.d, R, sc, a, work);
}

template <int BLK, int MINB, int MODE>
static void launch_algebra_mode(const FieldRegion& R, const Scalars& sc, const StageParams& a, const double* work,
                                cudaStream_t s) {
  bssn_algebra_kernel<BLK, MINB, MODE><<<(unsigned)((R.npts + BLK - 1) / BLK), BLK, 0, s>>>(R, sc, a, work);
}

template <int BLK, int MINB>
static int launch_algebra(const FieldRegion& R, const Scalars& sc, const StageParams& a, const double* work,
                          cudaStream_t s) {
  switch (a.mode) {
    case 0: launch_algebra_mode<BLK, MINB, 0>(R, sc, a, work, s); break;
    case 1: launch_algebra_mode<BLK, MINB, 1>(R, sc, a, work, s); break;
    case 2:
    case 3: launch_algebra_mode<BLK, MINB, 2>(R, sc, a, work, s); break;
    default: launch_algebra_mode<BLK, MINB, 4>(R, sc, a, work, s); break;
  }
  return launched("bssn_algebra_kernel");
}

int launch_bssn_split(const Dims& d, const Scalars& sc, const StageParams& a, const FieldWork& work, int block,
                      int minb, cudaStream_t s) {
  return for_field_chunks(d, sc, a.src, 24, work, s, [&](const FieldRegion& R) {
    if (block == 64) return minb >= 8 ? launch_algebra<64, 8>(R, sc, a, work.w, s) : launch_algebra<64, 5>(R, sc, a, work.w, s);
    if (minb == 2) return launch_algebra<128, 2>(R, sc, a, work.w, s);
    return minb == 4 ? launch_algebra<128, 4>(R, sc, a, work.w, s) : launch_algebra<128, 3>(R, sc, a, work.w, s);
  });
}

// ---------------------------------------------------------------------------
// algebra over many regions
// ---------------------------------------------------------------------------
// Persistent blocks pull work items -- 128 consecutive interior points of one
// region -- from the list with an atomic counter, so uneven regions keep every
// SM busy.  The loop is bounded by the item count (the counter only grows), an
// item naming a region outside the table sets bit 0 of the error word instead
// of touching memory, and a block past the time limit takes no more items and
// sets bit 1.
template <int MODE>
__global__ void __launch_bounds__(kItemPoints, 4)
batch_algebra_kernel(const FieldRegion* __restrict__ regions, int nregions, const WorkItem* __restrict__ items,
                     int nitems, unsigned int* counter, int* err, long long limit, Scalars sc, StageParams a_in,
                     const double* __restrict__ work) {
  StageParams a = a_in;
  a.mode = MODE;
  __shared__ unsigned int s_item;
  __shared__ double pre[kPre * kItemPoints];
  const long long t0 = clock64();
  for (int iter = 0; iter <= nitems; ++iter) {
    if (threadIdx.x == 0) {
      if (limit > 0 && clock64() - t0 > limit) {
        atomicOr(err, 2);
        s_item = (unsigned)nitems;
      } else {
        s_item = atomicAdd(counter, 1u);
      }
    }
    __syncthreads();
    const unsigned int it = s_item;
    __syncthreads();
    if (it >= (unsigned)nitems) break;
    const WorkItem q = items[it];
    if (q.patch < 0 || q.patch >= nregions) {
      if (threadIdx.x == 0) atomicOr(err, 1);
      continue;
    }
    const FieldRegion& R = regions[q.patch];
    const int64_t lin = (int64_t)q.start + threadIdx.x;
    if (q.start < 0 || lin >= R.npts) continue;
    bssn_algebra_point<kItemPoints>(R.d, R, lin, sc, a, work, pre);
  }
}

// Chunks of nearly equal size, each at most `cap` points (or one plane).
static int field_plan_create(const std::vector<PatchDesc>& patches, int64_t cap, FieldPlan* plan) {
  int64_t total = 0;
  for (const PatchDesc& P : patches) total += P.npts;
  const int64_t nchunks = (total + cap - 1) / cap;
  const int64_t target = std::max<int64_t>(1, (total + nchunks - 1) / std::max<int64_t>(1, nchunks));
  std::vector<FieldRegion> regions;
  std::vector<WorkItem> items;
  std::vector<int2> tiles;
  plan->chunks.clear();
  plan->points = 0;
  int64_t cur = 0;
  FieldPlan::Chunk ch{0, 0, 0, 0};
  auto close = [&]() {
    if (cur == 0) return;
    ch.item1 = (int)items.size();
    ch.tile1 = (int)tiles.size();
    plan->chunks.push_back(ch);
    plan->points = std::max(plan->points, cur);
    ch = FieldPlan::Chunk{ch.item1, 0, ch.tile1, 0};
    cur = 0;
  };
  for (const PatchDesc& P : patches) {
    const int64_t plane = (int64_t)P.d.nx * P.d.ny;
    for (int k0 = 0; k0 < P.d.nz;) {
      if (cur > 0 && cur + plane > target) close();
      Dims dk = P.d;
      dk.nz = (int)std::min<int64_t>(P.d.nz - k0, std::max<int64_t>(1, (target - cur) / plane));
      const FieldRegion R = field_region(dk, P.offset + (int64_t)k0 * P.d.sz, cur);
      const int q = (int)regions.size();
      regions.push_back(R);
      append_items(items, q, R.npts);
      const int64_t nt = region_tiles(R);
      for (int64_t t = 0; t < nt; ++t) tiles.push_back(int2{q, (int)t});
      cur += R.npts;
      k0 += dk.nz;
    }
  }
  close();
  if (items.size() > (size_t)0x7fffffff || tiles.size() > (size_t)0x7fffffff)
    return set_error(CHEMORA_EINVAL, "too many work items");
  plan->nregions = (int)regions.size();
  plan->nitems = (int)items.size();
  cudaError_t e = device_alloc(&plan->regions, regions.size() * sizeof(FieldRegion));
  if (e == cudaSuccess) e = device_alloc(&plan->items, items.size() * sizeof(WorkItem));
  if (e == cudaSuccess) e = device_alloc(&plan->tiles, tiles.size() * sizeof(int2));
  if (e == cudaSuccess)
    e = cudaMemcpy(plan->regions, regions.data(), regions.size() * sizeof(FieldRegion), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(plan->items, items.data(), items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(plan->tiles, tiles.data(), tiles.size() * sizeof(int2), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cudaGetLastError();
    field_plan_free(plan);
    return set_error(e == cudaErrorMemoryAllocation ? CHEMORA_ENOMEM : CHEMORA_ECUDA, "work-list storage: %s",
                     cudaGetErrorString(e));
  }
  return CHEMORA_OK;
}

int field_plans_create(const std::vector<PatchDesc>* tables, int n, const Dims* grid, FieldPlan* plans, double** work,
                       int64_t* points) {
  int64_t cap = kFieldWorkPoints, tried = 0;
  for (;;) {
    int rc = CHEMORA_OK;
    *points = grid ? field_work_points(*grid, cap) : 0;
    for (int t = 0; t < n && !rc; ++t) {
      rc = field_plan_create(tables[t], cap, &plans[t]);
      *points = std::max(*points, plans[t].points);
    }
    if (!rc && *points == tried) {
      rc = set_error(CHEMORA_ENOMEM, "derivative workspace of %zu bytes", field_work_bytes(*points));
    } else if (!rc) {
      const cudaError_t e = device_alloc(work, field_work_bytes(*points));
      if (e == cudaSuccess) return CHEMORA_OK;
      cudaGetLastError();
      *work = nullptr;
      if (e != cudaErrorMemoryAllocation) rc = cuda_error(e, "derivative workspace");
    }
    for (int t = 0; t < n; ++t) field_plan_free(&plans[t]);
    if (rc) return rc;
    tried = *points;
    cap = std::max<int64_t>(1, std::min(cap, tried) / 2);
  }
}

void field_plan_free(FieldPlan* plan) {
  cudaFree(plan->regions);
  cudaFree(plan->items);
  cudaFree(plan->tiles);
  plan->regions = nullptr;
  plan->items = nullptr;
  plan->tiles = nullptr;
}

static int persistent_algebra_blocks() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
    sms = 152;
  return 4 * sms;
}

int launch_field_plan(const FieldPlan& plan, unsigned int* counters, int* err, long long limit, const Scalars& sc,
                      const StageParams& p, double* work, cudaStream_t s) {
  const int blocks = persistent_algebra_blocks();
  int rc;
  for (size_t q = 0; q < plan.chunks.size(); ++q) {
    const FieldPlan::Chunk& c = plan.chunks[q];
    if ((rc = launch_field_kernels(plan.regions, FieldRegion{}, plan.tiles + c.tile0,
                                   (unsigned)(c.tile1 - c.tile0), 24, p.src, work, sc, s)))
      return rc;
    const WorkItem* items = plan.items + c.item0;
    const int n = c.item1 - c.item0;
    switch (p.mode) {
#define CHEMORA_BATCH_ALGEBRA(MODE)                                                                             \
  batch_algebra_kernel<MODE><<<blocks, kItemPoints, 0, s>>>(plan.regions, plan.nregions, items, n, counters + q, \
                                                            err, limit, sc, p, work)
      case 1: CHEMORA_BATCH_ALGEBRA(1); break;
      case 2:
      case 3: CHEMORA_BATCH_ALGEBRA(2); break;
      case 4: CHEMORA_BATCH_ALGEBRA(4); break;
      default: return set_error(CHEMORA_EINVAL, "batched stage mode %d", p.mode);
#undef CHEMORA_BATCH_ALGEBRA
    }
    if ((rc = launched("batch_algebra_kernel"))) return rc;
  }
  return CHEMORA_OK;
}

// ---------------------------------------------------------------------------
// constraints
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128, 3)
bssn_constraints_algebra_kernel(FieldRegion R, Scalars sc, const double* __restrict__ st, double* __restrict__ out,
                                const double* __restrict__ work) {
  const int64_t lin = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (lin >= R.npts) return;
  const int64_t c = R.offset + region_point(R.d, lin);
  const FieldLoader<128> ld{st + c, R.d.sv, work + field_base(R.w0 + lin), nullptr};
  auto o = [&](int v, double x) { out[c + v * R.d.sv] = x; };
  chemora_bssn_constraints_alg_point(ld, sc, o);
}

int launch_constraints_split(const Dims& d, const Scalars& sc, const double* state, double* out,
                             const FieldWork& work, cudaStream_t s) {
  // the constraints read no derivative of the lapse, the shift and B
  return for_field_chunks(d, sc, state, 17, work, s, [&](const FieldRegion& R) {
    bssn_constraints_algebra_kernel<<<(unsigned)((R.npts + 127) / 128), 128, 0, s>>>(R, sc, state, out, work.w);
    return launched("bssn_constraints_algebra_kernel");
  });
}

}  // namespace chemora
