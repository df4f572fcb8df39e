// Internal declarations of libchemora (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "chemora.h"
#include "device_types.cuh"

namespace chemora {

// ---------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------
int set_error(int code, const char* fmt, ...);
int cuda_error(cudaError_t e, const char* what);
#define CHEMORA_CUDA(call)                                  \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return ::chemora::cuda_error(e_, #call); \
  } while (0)
// after a kernel launch: count it and check the launch status
int launched(const char* name, int n = 1);
// Launches of this thread since the tally began, taken out of the count: they
// were captured, and count when their graph is launched.
class CaptureTally {
 public:
  CaptureTally();
  int take() const;

 private:
  int64_t start_;
};

// ---------------------------------------------------------------------------
// handles
// ---------------------------------------------------------------------------
enum HandleType : uint32_t {
  H_GRID = 0x47524944u,
  H_SYSTEM = 0x53595354u,
  H_BATCH = 0x42415443u,
  H_AMR = 0x414d5246u
};

struct chemora_grid_impl;
struct JitModule;  // run-time specialised stage kernels of one system

}  // namespace chemora

struct chemora_grid {
  uint32_t type;
  chemora::Dims d;
  int nvars;
  double dx;
  int64_t fsize;  // doubles per grid function
};

namespace chemora {
// The workspace of a system's last call on a stream that is being captured
// (capture.cu): capture, stream, last node of the call.
struct CaptureWork {
  double* w = nullptr;
  int64_t points = 0;
  unsigned long long id = 0;
  cudaStream_t stream = nullptr;
  cudaGraphNode_t last = nullptr;
};
}  // namespace chemora

struct chemora_system {
  uint32_t type;
  chemora_grid* grid;
  int kind;
  int nvars;
  chemora_params params;
  chemora::Scalars sc;
  // RK4 scratch: acc, stage a, stage b (library-owned)
  double* scratch;
  // variable-speed coefficients (library-owned, 4 grid functions svar apart):
  // s = c^2 with ghosts, then G_d = D_d s on the interior
  double* coef;
  // device copy of a host state for chemora_rk4_step_host (library-owned)
  double* dev_state;
  // derivative fields of the split BSSN right-hand side for the RK4 driver
  // (allocated on first use); calls that may run on several streams at once
  // (chemora_rhs, chemora_stage, chemora_constraints) take theirs from the
  // device's pool
  double* field_work;
  int64_t field_points;
  chemora::CaptureWork capture_work;
  // launch shape chosen by the autotuner (index into the kind's variants)
  int variant;
  // CUDA graph of one RK4 step (captured on cap_stream, replayed on the
  // caller's stream); key: state pointer, dt, variant
  cudaStream_t cap_stream;
  cudaGraph_t graph;
  cudaGraphExec_t graph_exec;
  double* graph_state;
  double graph_dt;
  int graph_variant;
  int graph_launches;  // kernels of the step
  // run-time specialised stage kernels (NULL until chemora_system_specialize)
  chemora::JitModule* jit;
  int jit_on;
  // launch-chained RK4 steps of the order-4 scalar wave (wave_chain.cu):
  // its captured graphs, and whether chemora_rk4_step uses it
  void* chain;
  int chain_on;
  // profiling
  int profile_on;
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used;
  double prof_ms;
  int64_t prof_launches;
};

namespace chemora {

Scalars make_scalars(double dx, const chemora_params& p);
int validate_system(int kind, int nvars, int nghost, int order);
int effective_order(int kind, const chemora_params& p);

// ghost fill of nvars grid functions (periodic image of the interior)
int fill_ghosts(const Dims& d, int nvars, double* state, cudaStream_t s);
// Every axis has at least g points: each ghost point lies within one period of
// the interior, and stages of the variable-speed wave write their outputs'
// ghost images themselves, with no fill passes between them.
inline int imaged_ok(const Dims& d) { return d.nx >= d.g && d.ny >= d.g && d.nz >= d.g ? 1 : 0; }
int fill_ghosts_axes(const Dims& d, int nvars, double* state, int mask, cudaStream_t s);

// Workspace of the split BSSN right-hand side (bssn_split.cu): derivative
// fields of up to `points` grid points; w NULL: none, the direct kernel runs.
struct FieldWork {
  double* w = nullptr;
  int64_t points = 0;
  bool captured = false;  // belongs to the graph the stream is captured into
};
constexpr int64_t kFieldWorkPoints = 1 << 20;  // points whose fields are held at once (1.36 GB)
int64_t field_work_points(const Dims& d, int64_t cap = kFieldWorkPoints);  // workspace points a stage on d uses
size_t field_work_bytes(int64_t points);
double field_fp64_instr(const Dims& d);
int launch_bssn_split(const Dims& d, const Scalars& sc, const StageParams& a, const FieldWork& work, int block,
                      int minb, cudaStream_t s);
int launch_constraints_split(const Dims& d, const Scalars& sc, const double* state, double* out,
                             const FieldWork& work, cudaStream_t s);
// The launch shape that runs for `variant` on d, and whether it runs the split
// kernels when it has a workspace.
int bssn_shape(const Dims& d, int variant);
bool bssn_shape_splits(const Dims& d, int variant);
// The RK4 driver's workspace (none if there is no memory for one), and one for a
// call on s: taken from and given back to the device's pool in stream order, or,
// while s is being captured, the graph's (capture.cu).
FieldWork system_field_work(chemora_system* sys);
FieldWork take_field_work(chemora_system* sys, cudaStream_t s);
void give_field_work(chemora_system* sys, const FieldWork& w, cudaStream_t s);
FieldWork capture_field_work(chemora_system* sys, int64_t points, cudaStream_t s);
void capture_work_used(chemora_system* sys, const FieldWork& w, cudaStream_t s);
void free_orphans();  // workspaces of graphs that are gone
cudaError_t device_alloc_relaxed(void** p, size_t bytes);  // also while a stream is being captured

// device memory in stream order from the device's pool (pool.cu), and for good
// (cudaMalloc; the pool's unused memory makes room)
cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s);
void pool_free(void* p, cudaStream_t s);
void pool_count_systems(int by);  // a system was made (+1) or destroyed (-1)
cudaError_t device_alloc(void** p, size_t bytes);
template <class T>
cudaError_t device_alloc(T** p, size_t bytes) {
  return device_alloc(reinterpret_cast<void**>(p), bytes);
}

int launch_stage(int kind, const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s,
                 int variant = 0, const FieldWork& work = FieldWork());
int launch_wave_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s, int variant);
int launch_varc_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s, int variant);
// G_d = D_d s (4th-order centred) on the interior of 3 grid functions at G,
// svar apart; s with valid ghosts.
int launch_varc_grad(const Dims& d, double i12h, const double* s, double* G, cudaStream_t st);
int launch_bssn_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s, int variant,
                      const FieldWork& work);
int launch_wave_order_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s,
                            int variant);
// Order-4 wave on planes in shared memory (wave_orders.cu).
template <int TX, int TY>
int launch_wave_planes(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s);
int launch_wave1_stage(const Dims& d, const Scalars& sc, const StageParams& a, cudaStream_t s, int variant);

// A compiled launch shape of a stage kernel (tx x ty threads, min blocks/SM).
typedef int (*StageLaunchFn)(const Dims&, const Scalars&, const StageParams&, cudaStream_t);
struct LaunchVariant {
  int tx, ty, minb;
  StageLaunchFn launch;
  int xshare;  // 1: lanes share x-direction work (nx % tx == 0); 2: and y via
               // shared memory; 4: z-march, the column in registers,
               // the plane in hand in shared memory (order-4 wave)
};
extern const LaunchVariant kBssnVariants[];
extern const int kNumBssnVariants;
extern const LaunchVariant kWaveVariants[];
extern const int kNumWaveVariants;
extern const LaunchVariant kVarcVariants[];
extern const int kNumVarcVariants;
extern const LaunchVariant kWave1Variants[];
extern const int kNumWave1Variants;
int num_variants(int kind);
const LaunchVariant* variant_info(int kind, int v);

// Time the plausible launch shapes of kind's stage kernel on grid d (stage
// arguments p, written into p.acc / p.dst) and return the fastest in *best
// (left alone if none ran) and its time.  Synchronous.
int autotune_stage(int kind, const Dims& d, const Scalars& sc, const StageParams& p, cudaStream_t s, int* best,
                   float* best_ms, const FieldWork& work = FieldWork());

// timing helpers for systems with profiling enabled
int prof_begin(chemora_system* sys, cudaStream_t s, cudaEvent_t* e0);
int prof_end(chemora_system* sys, cudaStream_t s, cudaEvent_t e0);

int ensure_scratch(chemora_system* sys);
void free_step_graph(chemora_system* sys);

// launch-chained RK4 steps of the order-4 scalar wave (wave_chain.cu)
bool chain_available(const chemora_system* sys);
int chain_rk4(chemora_system* sys, double* state, double dt, int nsteps, cudaStream_t s);
void chain_free(chemora_system* sys);

// run-time specialisation (jit.cu)
bool jit_active(const chemora_system* sys, const FieldWork& work);
int jit_launch(chemora_system* sys, const StageParams& a, const FieldWork& work, cudaStream_t s);
void jit_free(chemora_system* sys);

// Batched work-lists (patches.cu): a table of patches (grids inside one
// storage, each with its own extents and strides; the stage kernels compute
// the patch interior [g, n + g) per axis) and work items of up to 128
// consecutive interior points of one patch, x fastest.
struct PatchDesc {
  Dims d;
  int64_t offset;  // first double of the patch's state in the storage
  int64_t npts;    // interior points
};
struct WorkItem {
  int patch;
  int start;  // first interior point (linear, x fastest)
};
constexpr int kItemPoints = 128;
// Append the work items of patch q (npts interior points) to `items`.
void append_items(std::vector<WorkItem>& items, int q, int64_t npts);
// One persistent batched stage launch of the scalar wave over the device
// work-list `items` of the device patch table `pd`; `counter` (device, zero before the launch) hands out the items; bit
// 0 of *err is set for an item naming a patch outside the table, bit 1 when
// a block passed `limit` SM cycles (0: no limit).  src, yn, acc and dst of
// `p` are the storage bases; each patch's offset is added per item.
int launch_batch_stage(const PatchDesc* pd, int npatch, const WorkItem* items, int nitems,
                       unsigned int* counter, int* err, long long limit, const Scalars& sc,
                       const StageParams& p, cudaStream_t s);

// The split BSSN right-hand side over many regions: their z ranges, grouped
// into chunks whose derivative fields fit in one workspace.  Per chunk one
// field launch and one persistent algebra launch over a work-list.
struct FieldRegion;
struct FieldPlan {
  struct Chunk {
    int item0, item1, tile0, tile1;
  };
  std::vector<Chunk> chunks;
  int nregions = 0, nitems = 0;
  int64_t points = 0;  // workspace points
  FieldRegion* regions = nullptr;  // device
  WorkItem* items = nullptr;       // device: region and first point
  int2* tiles = nullptr;           // device: region and tile
};
// The plans of n tables of regions and the workspace that they (and the stages of
// *grid, if given) share: for kFieldWorkPoints points, or, where there is no memory
// for it, for as many halvings fewer as it takes, down to a plane at a time.
int field_plans_create(const std::vector<PatchDesc>* tables, int n, const Dims* grid, FieldPlan* plans, double** work,
                       int64_t* points);
void field_plan_free(FieldPlan* plan);
// One stage; counters: one per chunk, zero before the launch.
int launch_field_plan(const FieldPlan& plan, unsigned int* counters, int* err, long long limit, const Scalars& sc,
                      const StageParams& p, double* work, cudaStream_t s);

inline bool is_handle(const void* h, uint32_t t) {
  return h != nullptr && *reinterpret_cast<const uint32_t*>(h) == t;
}

}  // namespace chemora
