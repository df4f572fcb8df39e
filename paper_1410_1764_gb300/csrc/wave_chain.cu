// RK4 steps of the order-4 scalar wave (Sec. 3, Eq. 1, two-variable form)
// on small grids as a chain of stage kernels joined by programmatic
// dependent launches.
//
// On a 32^3 grid (32,768 points) a graph-replayed RK4 step of the per-stage
// kernels is 8 nodes -- 4 ghost fills, 4 stages -- of about 3 us each, set by
// launch latency rather than by arithmetic.  Here the stage kernel reads
// every neighbour at its periodic image (so no ghost fill is needed between
// stages; the ghosts are filled once per call), and each stage is launched
// as a programmatic dependent launch: the next stage's grid is scheduled
// while the current one runs, and waits in hardware (griddepcontrol.wait)
// until its predecessor has completed and its writes are visible.  Steps are
// captured K at a time in a CUDA graph.  The arithmetic is the generated
// point body and the RK update of the per-stage kernels, so both paths give
// the same bits.  No kernel here spins on memory.
#include <math.h>

#include <new>
#include <vector>

#include "internal.h"
#include "wave_point.cuh"

namespace chemora {

// The star's points of u at their periodic images, in Star2's order and the
// centre, read through L2 (the grid may start while its predecessor still runs,
// so nothing is read before the dependency wait and nothing is served from the
// SM's L1).
struct WrapLoader {
  const double* q[13];
  int64_t sv;
  __device__ __forceinline__ double operator()(int v, int dx, int dy, int dz) const {
    const int a = dx != 0 ? 0 : (dy != 0 ? 4 : 8), m = dx + dy + dz;
    return __ldcg(q[m == 0 ? 12 : a + (m == 1 ? 0 : (m == -1 ? 1 : (m == 2 ? 2 : 3)))] + v * sv);
  }
};

// The scalar wave's fused RK update of StageOutFma (same operations in the
// same order) with y_n and the accumulator of both variables loaded up
// front, together with the neighbours, and the results stored to L2.
struct ChainStageOut {
  const StageParams& a;
  int64_t c, sv;
  double one, two;
  double yn[2], acc[2];
  __device__ __forceinline__ void operator()(int v, double k) const {
    const int64_t cv = c + v * sv;
    switch (a.mode) {
      case 1:
        __stcg(a.acc + cv, k);
        __stcg(a.dst + cv, __fma_rn(a.c2, k, yn[v]));
        break;
      case 2:
      case 3:
        __stcg(a.acc + cv, __fma_rn(two, k, acc[v]));
        __stcg(a.dst + cv, __fma_rn(a.c2, k, yn[v]));
        break;
      default:
        __stcg(a.dst + cv, __fma_rn(a.c1, __fma_rn(acc[v], one, k), yn[v]));
        break;
    }
  }
};

__device__ __forceinline__ int wrap_index(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// One stage (mode 1..4) of the order-4 scalar wave on the interior, one
// point per thread (thread t of block b: interior point 128 b + t, x
// fastest).
__global__ void __launch_bounds__(128) wave_chain_stage_kernel(Dims d, Scalars sc, StageParams a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // 32-bit indices (chain_available): 64-bit divisions for the point's place
  // took a third of the instructions.  The addresses are pinned here, before the
  // wait, where they cost nothing: left to the compiler, 32-bit ones are formed
  // after it (61 x 75 x 53 x 20 steps 525 us, 32^3 x 100 steps 1247; pinned 491
  // and 1162; with 64-bit indices 530 and 1205; order-4 Laplacian with two guard bits
  // then, 503 and 1188 now).
  const unsigned t = blockIdx.x * 128 + threadIdx.x;
  const unsigned npts = (unsigned)d.nx * d.ny * d.nz;
  const unsigned row = t / (unsigned)d.nx;
  const int k = (int)(row / (unsigned)d.ny);
  const int j = (int)(row - (unsigned)k * d.ny), i = (int)(t - row * d.nx);
  const int64_t c = (int64_t)(k + d.g) * d.sz + (int64_t)(j + d.g) * d.sy + (i + d.g);
  WrapLoader ld;
  ld.sv = d.sv;
  ld.q[12] = a.src + c;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int o = m == 0 ? 1 : (m == 1 ? -1 : (m == 2 ? 2 : -2));
    ld.q[m] = ld.q[12] + (wrap_index(i + o, d.nx) - i);
    ld.q[4 + m] = ld.q[12] + (wrap_index(j + o, d.ny) - j) * (int)d.sy;
    ld.q[8 + m] = ld.q[12] + (wrap_index(k + o, d.nz) - k) * (int)d.sz;
  }
#pragma unroll
  for (int m = 0; m < 13; ++m) asm volatile("" : "+l"(ld.q[m]));
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (t >= npts) return;
  ChainStageOut out{a, c, d.sv, sc.k[CHEMORA_K_ONE], sc.k[CHEMORA_K_TWO], {0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    out.yn[v] = __ldcg(a.yn + c + v * d.sv);
    if (a.mode >= 2) out.acc[v] = __ldcg(a.acc + c + v * d.sv);
  }
  wave_point(ld, sc, out);
}

struct ChainGraph {
  cudaGraphExec_t exec = nullptr;
  double* state = nullptr;
  double dt = 0.0;
  int steps = 0;
  int launches = 0;
};

// Per-system state: graphs of K steps and of the remainder.
struct ChainState {
  ChainGraph graph[2];
};

constexpr int kChainGraphSteps = 8;

static int chain_stage(const chemora_system* sys, const StageParams& p, cudaStream_t s) {
  const Dims& d = sys->grid->d;
  const int64_t npts = (int64_t)d.nx * d.ny * d.nz;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((npts + 127) / 128));
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  CHEMORA_CUDA(cudaLaunchKernelEx(&cfg, wave_chain_stage_kernel, d, sys->sc, p));
  return launched("wave_chain_stage_kernel");
}

static int chain_steps(const chemora_system* sys, double* Y, double dt, int nsteps, cudaStream_t s) {
  const size_t n = (size_t)sys->nvars * sys->grid->fsize;
  double* acc = sys->scratch;
  double* Sa = sys->scratch + n;
  double* Sb = sys->scratch + 2 * n;
  double* srcs[4] = {Y, Sa, Sb, Sa};
  double* dsts[4] = {Sa, Sb, Sa, Y};
  const double c2[4] = {0.5 * dt, 0.5 * dt, dt, 0.0};
  int rc;
  for (int step = 0; step < nsteps; ++step)
    for (int q = 0; q < 4; ++q) {
      StageParams p{};
      p.src = srcs[q]; p.yn = Y; p.acc = acc; p.dst = dsts[q];
      p.c1 = dt / 6.0; p.c2 = c2[q]; p.mode = q + 1;
      if ((rc = chain_stage(sys, p, s))) return rc;
    }
  return CHEMORA_OK;
}

static int chain_graph(chemora_system* sys, ChainGraph& g, double* Y, double dt, int steps) {
  if (g.exec && g.state == Y && g.dt == dt && g.steps == steps) return CHEMORA_OK;
  if (g.exec) cudaGraphExecDestroy(g.exec);
  g.exec = nullptr;
  if (!sys->cap_stream) CHEMORA_CUDA(cudaStreamCreateWithFlags(&sys->cap_stream, cudaStreamNonBlocking));
  CHEMORA_CUDA(cudaStreamBeginCapture(sys->cap_stream, cudaStreamCaptureModeThreadLocal));
  const CaptureTally tally;
  int rc = chain_steps(sys, Y, dt, steps, sys->cap_stream);
  g.launches = tally.take();
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(sys->cap_stream, &graph);
  if (rc) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return cuda_error(e, "cudaStreamEndCapture");
  e = cudaGraphInstantiate(&g.exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return cuda_error(e, "cudaGraphInstantiate");
  g.state = Y;
  g.dt = dt;
  g.steps = steps;
  return CHEMORA_OK;
}

bool chain_available(const chemora_system* sys) {
  const Dims& d = sys->grid->d;
  // one point per thread in one grid; int offsets
  return sys->kind == CHEMORA_WAVE && sys->sc.order == 4 && d.g >= 2 && d.nx >= 2 && d.ny >= 2 && d.nz >= 2 &&
         (double)d.sv * sys->nvars < 2.0e9 && (double)d.nx * d.ny * d.nz <= 128.0 * 2147483647.0;
}

int chain_rk4(chemora_system* sys, double* state, double dt, int nsteps, cudaStream_t s) {
  if (!chain_available(sys)) return set_error(CHEMORA_EUNSUPPORTED, "no launch-chained step for this system");
  if (!sys->chain) {
    ChainState* cs = new (std::nothrow) ChainState();
    if (!cs) return set_error(CHEMORA_ENOMEM, "host allocation");
    sys->chain = cs;
  }
  ChainState* cs = static_cast<ChainState*>(sys->chain);
  int rc;
  const int full = nsteps / kChainGraphSteps, rest = nsteps % kChainGraphSteps;
  if (full) {
    if ((rc = chain_graph(sys, cs->graph[0], state, dt, kChainGraphSteps))) return rc;
    for (int q = 0; q < full; ++q) {
      CHEMORA_CUDA(cudaGraphLaunch(cs->graph[0].exec, s));
      if ((rc = launched("cudaGraphLaunch(chained RK4 steps)", cs->graph[0].launches))) return rc;
    }
  }
  if (rest) {
    if ((rc = chain_graph(sys, cs->graph[1], state, dt, rest))) return rc;
    CHEMORA_CUDA(cudaGraphLaunch(cs->graph[1].exec, s));
    if ((rc = launched("cudaGraphLaunch(chained RK4 steps)", cs->graph[1].launches))) return rc;
  }
  return fill_ghosts(sys->grid->d, sys->nvars, state, s);
}

void chain_free(chemora_system* sys) {
  if (!sys->chain) return;
  ChainState* cs = static_cast<ChainState*>(sys->chain);
  for (ChainGraph& g : cs->graph)
    if (g.exec) cudaGraphExecDestroy(g.exec);
  delete cs;
  sys->chain = nullptr;
}

}  // namespace chemora
