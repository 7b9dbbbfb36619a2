// A CUDA device and the library's kernels played on the host, for tests of the host code that
// chooses, captures and launches them (hosc_api.cu, hosc_pool.cu, which have no device code). Device
// memory is host memory; streams run at once, or append to the graph that is being captured on them; a
// launch writes one line to a log, refuses when told to, and takes a made-up time.

#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

#include <functional>
#include <map>
#include <memory>
#include <set>
#include <string>
#include <vector>

#include "hosc.h"
#include "hosc_internal.h"

using namespace hosc;

namespace {

typedef std::vector<std::function<void()>> Ops;
struct Graph { std::shared_ptr<Ops> ops = std::make_shared<Ops>(); };
struct Stream { std::shared_ptr<Ops> capture; };
struct Event { double at = 0.0; std::shared_ptr<Ops> capture; };

std::set<Stream*> g_streams;
std::string g_log;
cudaError_t g_last = cudaSuccess;
std::map<std::string, int> g_refuse;    // launches of this name left to refuse
std::map<std::string, double> g_cost;   // milliseconds of a launch, 1 where not set
double g_now = 0.0;
Graph g_body_handle;
std::map<void*, size_t> g_sizes;   // of device allocations

void run(cudaStream_t s, std::function<void()> f) {
  Stream* q = (Stream*)s;
  if (q && q->capture) q->capture->push_back(f);
  else f();
}

std::string form(const DevParams& P) {
  if (P.coop) return "one_launch";
  if (!P.krylov_fp32) return "planar";
  if (P.merged) return "merged";
  if (P.tty > 0) return "bulk";
  if (P.sx > 0) return "staged";
  return P.plane ? "plane" : "register";
}

// a launch: its line in the log and its time when it runs, or an error now
void launch(cudaStream_t s, const std::string& name, const std::string& detail,
            std::function<void()> effect = nullptr) {
  auto it = g_refuse.find(name);
  if (it != g_refuse.end() && it->second != 0) {
    if (it->second > 0) it->second -= 1;
    g_last = cudaErrorLaunchOutOfResources;
    return;
  }
  run(s, [=]() {
    g_log += name + (detail.empty() ? "" : " " + detail) + "\n";
    auto c = g_cost.find(name + " " + detail);
    if (c == g_cost.end()) c = g_cost.find(name + " " + detail.substr(0, detail.find(' ')));
    if (c == g_cost.end()) c = g_cost.find(name);
    g_now += c == g_cost.end() ? 1.0 : c->second;
    if (effect) effect();
  });
}
std::string krylov(const DevParams& P) {
  return form(P) + " " + std::to_string(P.kblock) + "x" + std::to_string(P.kz) +
         (P.xr_flat ? " flat" : "");
}

void end_of_solve(const Fields& F) {
  for (int s = 0; s < 4; ++s) {
    F.ks[s].r0norm = 1.0;
    F.ks[s].iters = 1;
    F.ks[s].done = 1;
  }
}
void record(const DevParams& P, const Fields& F) {
  StepRecord r = {};
  r.res = r.div_max = 1.0;
  for (int s = 0; s < 4; ++s) {
    r.iters[s] = F.ks[s].iters;
    const int st = system_status(F.ks[s], P.merged);
    if (st) r.status = st;
  }
  *F.rec = r;
  F.ring[*F.ring_pos % kRing] = r;
  *F.ring_pos += 1;
}

}  // namespace

extern "C" {

const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void fake_refuse(const char* name, int launches) { g_refuse[name] = launches; }   // -1: every one
void fake_cost(const char* name, double ms) { g_cost[name] = ms; }
void fake_reset() {
  g_log.clear();
  g_refuse.clear();
  g_cost.clear();
  g_last = cudaSuccess;
}

// ---------------------------------------------------------------- the runtime

cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {   // zeros that take no memory until they are written
  *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  g_sizes[*p] = n;
  return *p == MAP_FAILED ? cudaErrorMemoryAllocation : cudaSuccess;
}
cudaError_t cudaFree(void* p) { return munmap(p, g_sizes[p]), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = calloc(n, 1), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* a, size_t n, cudaMemcpyKind, cudaStream_t s) {
  run(s, [=]() { memcpy(d, a, n); });
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t s) {
  auto it = g_sizes.find(d);
  if (it != g_sizes.end() && it->second == n) return madvise(d, n, MADV_DONTNEED), cudaSuccess;
  run(s, [=]() { memset(d, v, n); });
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  Stream* q = new Stream();
  g_streams.insert(q);
  *s = (cudaStream_t)q;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  g_streams.erase((Stream*)s);
  delete (Stream*)s;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t) new Event(), cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete (Event*)e, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  ((Event*)e)->at = g_now;
  ((Event*)e)->capture = s ? ((Stream*)s)->capture : nullptr;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  return *ms = (float)(((Event*)b)->at - ((Event*)a)->at), cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (((Event*)e)->capture) ((Stream*)s)->capture = ((Event*)e)->capture;
  return cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return *g = (cudaGraph_t) new Graph(), cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete (Graph*)g, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  return ((Stream*)s)->capture = std::make_shared<Ops>(), cudaSuccess;
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t s, cudaGraph_t g, const cudaGraphNode_t*,
                                          const cudaGraphEdgeData*, size_t, cudaStreamCaptureMode) {
  return ((Stream*)s)->capture = ((Graph*)g)->ops, cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  const std::shared_ptr<Ops> ops = ((Stream*)s)->capture;
  for (Stream* q : g_streams)
    if (q->capture == ops) q->capture = nullptr;
  Graph* out = new Graph();
  out->ops = ops;
  *g = (cudaGraph_t)out;   // where the graph is the caller's this leaks a few bytes
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus* st, unsigned long long*,
                                     cudaGraph_t* g, const cudaGraphNode_t** deps,
                                     const cudaGraphEdgeData**, size_t* n) {
  static std::map<Ops*, Graph> open;
  const std::shared_ptr<Ops> ops = ((Stream*)s)->capture;
  *st = ops ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  open[ops.get()].ops = ops;
  *g = (cudaGraph_t)&open[ops.get()];
  *deps = nullptr;
  *n = 0;
  return cudaSuccess;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned,
                                             unsigned) {
  return *h = 1, cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t g, const cudaGraphNode_t*,
                             const cudaGraphEdgeData*, size_t, cudaGraphNodeParams* p) {
  g_body_handle.ops = std::make_shared<Ops>();
  static cudaGraph_t body = (cudaGraph_t)&g_body_handle;
  p->conditional.phGraph_out = &body;
  const std::shared_ptr<Ops> ops = g_body_handle.ops;
  ((Graph*)g)->ops->push_back([ops]() {   // one pass: the made-up systems are done after it
    for (auto& f : *ops) f();
  });
  return cudaSuccess;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t*, const cudaGraphEdgeData*,
                                                size_t, unsigned) {
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  Graph* x = new Graph();
  x->ops = ((Graph*)g)->ops;
  *e = (cudaGraphExec_t)x;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return delete (Graph*)e, cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  for (auto& f : *((Graph*)e)->ops) f();
  return cudaSuccess;
}

// entry points of other sources that the binding looks up
hosc_status hosc_fp64_peak(int, double*) { return HOSC_ECUDA; }
hosc_status hosc_bicgstab_noalloc(int, const double* const*, const double* const*, double* const*,
                                  double, int, int*, void*) {
  return HOSC_ECUDA;
}

}  // extern "C"

// ---------------------------------------------------------------- the kernels

namespace hosc {

int device_sms() { return 152; }
int red_blocks(long count, int threads) { return (int)((count + threads - 1) / threads); }
long krylov4_blocks(const DevParams& P) {
  const long ni = P.N - 2;
  return ((ni * ni + P.kblock - 1) / P.kblock) * ((ni + P.kz - 1) / P.kz);
}
double krylov4_wave_cost(int N, int kblock, int kz, int, int, int sms) {
  const long ni = N - 2, items = ((ni * ni + kblock - 1) / kblock) * ((ni + kz - 1) / kz);
  return (double)((items + 2 * sms - 1) / (2 * sms)) * (kz + 2);
}
void default_tiles(int N, int* b, int* z) { *b = 384, *z = N - 2 < 8 ? N - 2 : 8; }
bool plane_shape(int N, int* x, int* y, int* z) { return *x = *y = 16, *z = 8, N >= kPlaneMinN; }
void planar_shape(int, int* b, int* z) { *b = 128, *z = 4; }
bool solve_shape_planar(int N, int, int* b, int* z) { return *b = 128, *z = 2, N <= 42; }
bool solve_shape_mixed(int N, int* b, int* z) { return *b = 256, *z = 2, N <= 68; }
size_t staged_smem_bytes(int, int, bool) { return 0; }
double staged_wave_cost(int, int, int, int, int) { return 1.0; }
bool tma_tiles_valid(int, int, int, int) { return false; }
double tma_wave_cost(int, int, int, int, int) { return 1e300; }
bool tma_prepare(const DevParams&, const Fields&, void*) { return false; }
int tma_tile_x(int) { return 0; }

void launch_arm(const Fields& F, int stop, cudaStream_t s) {
  launch(s, "arm", "", [=]() { *F.halt = 0, *F.ring_pos = 0, *F.steady_stop = stop; });
}
void launch_shadow(const DevParams&, const Fields&, int, int, cudaStream_t s) { launch(s, "shadow", ""); }
void launch_viscosity(const DevParams&, const Fields&, int, cudaStream_t s) { launch(s, "viscosity", ""); }
void launch_sources(const DevParams&, const Fields&, int, cudaStream_t s) { launch(s, "sources", ""); }
void launch_rhs(const DevParams&, const Fields& F, int, cudaStream_t s) {
  launch(s, "rhs", "", [=]() { memset((void*)F.ks, 0, 4 * sizeof(KrylovScalars)); });
}
void launch_bicg_init(const DevParams& P, const Fields& F, cudaStream_t s) {
  launch(s, "init", krylov(P), [=]() {
    for (int q = 0; q < 4; ++q) F.ks[q].r0norm = 1.0;
  });
}
void launch_bicg_pv(const DevParams& P, const Fields&, int, bool, cudaStream_t s) { launch(s, "pv", krylov(P)); }
void launch_bicg_st(const DevParams& P, const Fields&, int, bool, cudaStream_t s) { launch(s, "st", krylov(P)); }
void launch_bicg_xr(const DevParams& P, const Fields& F, int, bool, cudaStream_t s) {
  launch(s, P.xr_flat ? "xr_flat" : "xr", krylov(P), [=]() { end_of_solve(F); });
}
void launch_b2(int k, const DevParams& P, const Fields& F, int, bool, cudaStream_t s) {
  launch(s, "b2", krylov(P), [=]() { if (k == 4) end_of_solve(F); });
}
void launch_loop_cond(const Fields&, unsigned long long, cudaStream_t s) { launch(s, "loop", ""); }
void launch_solve(const DevParams& P, const Fields& F, cudaStream_t s) {
  launch(s, "solve", krylov(P), [=]() { end_of_solve(F); });
}
void launch_krylov_activate(const Fields&, cudaStream_t s) {
  run(s, []() {});
}
void launch_update(const DevParams& P, const Fields& F, int, int rec, cudaStream_t s) {
  launch(s, "update", "", [=]() { if (rec) record(P, F); });
}
void launch_finish(const DevParams& P, const Fields& F, cudaStream_t s) {
  launch(s, "finish", "", [=]() { record(P, F); });
}
void launch_diagnostics(const DevParams&, const Fields&, int, int, cudaStream_t s) { launch(s, "diagnostics", ""); }
RoundState* round_state_create() { return nullptr; }
void round_state_destroy(RoundState*) {}
void round_member_shape(RoundMember*) {}
hosc_status launch_flow(RoundState*, const std::vector<RoundMember>&, int, cudaStream_t, char*, size_t) {
  return HOSC_ECUDA;
}

}  // namespace hosc
