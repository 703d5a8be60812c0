// Stand-in for the CUDA runtime, for tests of the host side (api.cu, batch.cu,
// lanes.h) without a GPU (the kernel launchers: fake_launchers.cu). Device memory is host
// memory; a step adds 1 to the first element of every instance it takes, when
// it is issued (or when the graph that captured it is launched), so an
// instance counts its steps; every step launch is logged with its stream; each
// stream has a clock, which a step advances by a settable cost.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Graph {
  std::vector<std::function<void(cudaStream_t)>> ops;
};
struct Stream {
  int id, device, priority;
  Graph* capture = nullptr;
  double clock = 0.0;
};
struct Event {
  Graph* capture = nullptr;
  double clock = 0.0;
};

std::string g_log;
int g_device = 0, g_ids = 0;
double g_launch_cost = 2.0, g_node_cost[2] = {1e-4, 1e-4}, g_tma_cost = 1e-4;
size_t g_fit = size_t(-1);  // instances x bytes above which a node costs g_node_cost[1]
bool g_replaying = false;

Stream* st(cudaStream_t s) { return reinterpret_cast<Stream*>(s); }
Event* ev(cudaEvent_t e) { return reinterpret_cast<Event*>(e); }

void log(const std::string& s) { g_log += s + "\n"; }

void issue(cudaStream_t s, std::function<void(cudaStream_t)> op) {
  if (st(s)->capture) st(s)->capture->ops.push_back(op);
  else op(s);
}

}  // namespace

// One step launch: input and output of each instance, elements of `elem` bytes.
void fake_step(const char* kind, const std::vector<std::pair<const void*, void*>>& inst, int elem, double nodes,
               bool chained, int threads, cudaStream_t s, int tile) {
  const std::string k = kind;
  const size_t bytes = size_t(nodes * 2 * 41 * elem);
  issue(s, [=](cudaStream_t on) {
    for (auto& io : inst) {
      uint64_t v = 0;
      std::memcpy(&v, io.first, size_t(elem));
      ++v;
      std::memcpy(io.second, &v, size_t(elem));
    }
    const double rate = k == "tma" ? g_tma_cost : g_node_cost[bytes > g_fit ? 1 : 0];
    st(on)->clock += g_launch_cost + rate * nodes;
    char line[160];
    std::snprintf(line, sizeof line, "%s stream=%d first=%llx count=%zu chained=%d threads=%d replay=%d tile=%d", k.c_str(),
                  st(on)->id, (unsigned long long)(uintptr_t)inst[0].first, inst.size(), chained ? 1 : 0, threads,
                  g_replaying ? 1 : 0, tile);
    log(line);
  });
}

extern "C" {

const char* fake_take_log() {
  static std::string out;
  out.swap(g_log);
  g_log.clear();
  return out.c_str();
}
void fake_set_device(int d) { g_device = d; }
int fake_device() { return g_device; }
// a step of `bytes` costs launch + nodes * (fits or not) microseconds
void fake_set_costs(double launch, double fits, double not_fits, double fit_bytes, double tma) {
  g_launch_cost = launch;
  g_node_cost[0] = fits;
  g_node_cost[1] = not_fits;
  g_fit = size_t(fit_bytes);
  g_tma_cost = tma;
}
void fake_capture(void* s, int on) { static_cast<Stream*>(s)->capture = on ? new Graph : nullptr; }
void* fake_stream(int priority) { return new Stream{g_ids++, g_device, priority}; }

// ---- runtime ----
cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(1, n); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }

cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int priority) {
  Stream* n = new Stream{g_ids++, g_device, priority};
  *s = reinterpret_cast<cudaStream_t>(n);
  log("create stream=" + std::to_string(n->id) + " device=" + std::to_string(g_device) +
      " priority=" + std::to_string(priority));
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { return cudaStreamCreateWithPriority(s, f, 0); }
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) { *p = st(s)->priority; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete st(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (ev(e)->capture) st(s)->capture = ev(e)->capture;
  else if (ev(e)->clock > st(s)->clock) st(s)->clock = ev(e)->clock;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = st(s)->capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  if (st(s)->capture) return cudaErrorIllegalState;
  st(s)->capture = new Graph;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  *g = reinterpret_cast<cudaGraph_t>(st(s)->capture);
  st(s)->capture = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long) {
  *x = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph*>(g)));
  log("instantiate");
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete reinterpret_cast<Graph*>(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete reinterpret_cast<Graph*>(x); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
  g_replaying = true;
  for (auto& op : reinterpret_cast<Graph*>(x)->ops) op(s);
  g_replaying = false;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(new Event); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete ev(e); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  ev(e)->capture = st(s)->capture;
  ev(e)->clock = st(s)->clock;
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = float((ev(b)->clock - ev(a)->clock) * 1e-3);
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}

}  // extern "C"

