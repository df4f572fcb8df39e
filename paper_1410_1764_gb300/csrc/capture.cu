// Derivative-field workspaces of BSSN right-hand sides, stages and constraints on
// a stream that is being captured.  Memory taken in stream order would become a
// node of the caller's graph, which such a graph may not have everywhere (bodies
// of conditional nodes) and which bars a second instance of it.  So the workspace
// is allocated at once and given to the graph as a user object: it lives as long
// as the graph and its instances.  Calls in a row of one capture share it.  (Without
// one, the kernel that needs no workspace ran: 128^3 right-hand side 10.4 ms in a
// graph, 4.4 outside.)
#include <mutex>
#include <vector>

#include "internal.h"

namespace chemora {

// Not held over a CUDA call: the destructors below run on a thread of CUDA's.
static std::mutex g_capture_mu;
// workspaces whose graphs are gone (a destructor may not free them: that is a CUDA
// call); never destroyed, since graphs may outlive static objects
static std::vector<double*>& g_orphans = *new std::vector<double*>();

static void orphan(void* p) {
  const std::lock_guard<std::mutex> lock(g_capture_mu);
  g_orphans.push_back(static_cast<double*>(p));
}

// Calls that are refused while a stream is being captured are allowed to this
// thread while one of these lives.
class Relaxed {
 public:
  Relaxed() { cudaThreadExchangeStreamCaptureMode(&mode_); }
  ~Relaxed() { cudaThreadExchangeStreamCaptureMode(&mode_); }

 private:
  cudaStreamCaptureMode mode_ = cudaStreamCaptureModeRelaxed;
};

cudaError_t device_alloc_relaxed(void** p, size_t bytes) {
  const Relaxed relaxed;
  return device_alloc(p, bytes);
}

void free_orphans() {
  std::vector<double*> gone;
  {
    const std::lock_guard<std::mutex> lock(g_capture_mu);
    gone.swap(g_orphans);
  }
  if (gone.empty()) return;
  const Relaxed relaxed;
  for (double* p : gone) cudaFree(p);
}

// Does the capture's present end come after node `from`, as far as following one
// predecessor each shows?  (Calls in a row on a stream do; not on a stream whose
// dependencies were set back.)
static bool follows(const cudaGraphNode_t* ends, size_t n, cudaGraphNode_t from) {
  if (n != 1) return false;
  cudaGraphNode_t node = ends[0];
  for (int step = 0; step < 4096; ++step) {
    if (node == from) return true;
    cudaGraphNode_t before[8];
    cudaGraphEdgeData edges[8];
    size_t m = 8;
    if (cudaGraphNodeGetDependencies(node, before, edges, &m) != cudaSuccess || m == 0) {
      cudaGetLastError();
      return false;
    }
    for (size_t q = 1; q < m && q < 8; ++q)
      if (before[q] == from) return true;
    node = before[0];
  }
  return false;
}

struct CaptureInfo {
  unsigned long long id = 0;
  cudaGraph_t graph = nullptr;
  const cudaGraphNode_t* ends = nullptr;
  size_t n = 0;
  bool get(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    const cudaGraphEdgeData* edges = nullptr;
    if (cudaStreamGetCaptureInfo(s, &st, &id, &graph, &ends, &edges, &n) == cudaSuccess)
      return st == cudaStreamCaptureStatusActive;
    cudaGetLastError();
    return false;
  }
};

FieldWork capture_field_work(chemora_system* sys, int64_t points, cudaStream_t s) {
  FieldWork w;
  w.captured = true;
  CaptureInfo c;
  if (!c.get(s)) return w;
  CaptureWork k;
  {
    const std::lock_guard<std::mutex> lock(g_capture_mu);
    k = sys->capture_work;
  }
  if (k.w && k.id == c.id && k.stream == s && k.points == points && follows(c.ends, c.n, k.last)) {
    w.w = k.w;
    w.points = points;
    return w;
  }
  free_orphans();
  double* p = nullptr;
  if (device_alloc_relaxed((void**)&p, field_work_bytes(points)) != cudaSuccess) {
    cudaGetLastError();
    return w;
  }
  cudaUserObject_t owner = nullptr;
  if (cudaUserObjectCreate(&owner, p, orphan, 1, cudaUserObjectNoDestructorSync) != cudaSuccess) {
    cudaGetLastError();
    orphan(p);
    return w;
  }
  if (cudaGraphRetainUserObject(c.graph, owner, 1, cudaGraphUserObjectMove) != cudaSuccess) {
    cudaGetLastError();
    cudaUserObjectRelease(owner, 1);
    return w;
  }
  w.w = p;
  w.points = points;
  return w;
}

void capture_work_used(chemora_system* sys, const FieldWork& w, cudaStream_t s) {
  CaptureInfo c;
  const bool ok = w.w && c.get(s) && c.n == 1;
  const std::lock_guard<std::mutex> lock(g_capture_mu);
  CaptureWork& k = sys->capture_work;
  k = CaptureWork();
  if (!ok) return;
  k.w = w.w;
  k.points = w.points;
  k.id = c.id;
  k.stream = s;
  k.last = c.ends[0];
}

}  // namespace chemora
