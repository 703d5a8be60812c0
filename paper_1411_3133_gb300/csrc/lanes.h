// Order in which the instances of a batch take the time steps of one call.
//
// The instances do not exchange anything, so a call of n steps may take them
// in groups: a group whose two buffers fit L2 several times over takes all its
// steps before the next one starts, and reads back from L2 what it wrote the
// step before. A group alone would leave SMs idle in its last wave of blocks
// and between its launches, so several groups run side by side on LANES
// streams. Measured on one GB300, GLUPS of 64 x 4 x 256 channels, all 24
// instances a step on one stream against 4 streams of one or two instances:
// cylinder FP32 19.5 / 22.7, FP16 23.0 / 29.0; four-wall ellipsoid FP32 18.1 /
// 22.7, FP16 20.3 / 25.3. The lines: instances are joined up to a quarter of
// 90 MiB, so that four streams hold what L2 keeps, and further up to half of it
// where the launch would be too short to be issued while the others run (about
// 2 us, 60 000 nodes). An instance of its own may be as large as half of it:
// four streams then hold up to 180 MiB and much of the state comes from HBM --
// 12 of 96 x 4 x 340 in FP32 (43 MB each) 78.2 us a step, 79.8 in one launch over
// all, 69.0 on two streams; 4 of 64 x 4 x 256 in FP64 235, 249, 235. A bound of
// 90 MiB on what all streams hold together, with two streams for chunks above a
// quarter of it, costs more than it gives: 24 mixed channels in FP32 3.90 ->
// 3.72 ms for 40 steps, but 20 of 64 x 4 x 300 (25 MB each) 69.9 -> 80.0 us a
// step and batches of 4 to 10 unlike channels up to 1.5 times as long. With an
// instance above half of it the plan is empty. The 2-byte storage's stream table
// counts as held: with the state alone the ellipsoid ran in groups of two whose
// tables (3.4 MB an instance) went to HBM, 68.7 us a step of the 24 in FP16
// against 63.8.
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace lbgm {

constexpr int LANES = 4;
constexpr int LANE_MIN_STEPS = 4;  // fewer steps than this reuse too little

struct LaneChunk {
  int group, first, count, lane;
};

// One instance: its group (only instances of one group share a launch), nodes
// and the bytes its steps use.
struct LaneInst {
  int group;
  size_t nodes, bytes;
};

// The chunks of consecutive instances of one group (at most max_count of them)
// and the stream each runs on, in the order the streams take them; empty where
// one launch a step over everything is the better plan.
inline std::vector<LaneChunk> plan_lanes(const std::vector<LaneInst>& inst, int max_count) {
  constexpr size_t kHold = size_t(90) << 20, kNodes = 60000;
  size_t total = 0;
  for (const LaneInst& i : inst) total += i.bytes;
  const size_t target = std::min(kHold / LANES, total / LANES);
  std::vector<LaneChunk> chunks;
  std::vector<size_t> bytes;
  for (size_t i = 0; i < inst.size();) {
    LaneChunk c{inst[i].group, int(i), 1, 0};
    size_t b = inst[i].bytes, n = inst[i].nodes;
    for (++i; i < inst.size() && inst[i].group == c.group && c.count < max_count; ++i) {
      const size_t more = b + inst[i].bytes;
      if (more > target && (n >= kNodes || more > kHold / 2)) break;
      b = more;
      n += inst[i].nodes;
      ++c.count;
    }
    if (b > kHold / 2) return {};
    chunks.push_back(c);
    bytes.push_back(b);
  }
  if (chunks.size() < 2) return {};
  // the largest chunks first, each to the stream with the least to do
  std::vector<size_t> order(chunks.size()), load(LANES, 0);
  for (size_t i = 0; i < order.size(); ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](size_t a, size_t b) { return bytes[a] > bytes[b]; });
  std::vector<LaneChunk> out;
  for (size_t i : order) {
    const size_t l = std::min_element(load.begin(), load.end()) - load.begin();
    load[l] += bytes[i];
    chunks[i].lane = int(l);
    out.push_back(chunks[i]);
  }
  return out;
}

// Streams and events of the lanes; lane 0 is the owner's stream.
struct LaneStreams {
  cudaStream_t aux[LANES - 1] = {};
  cudaEvent_t fork = nullptr, join[LANES - 1] = {};

  // On `device` and with the priority of the owner's stream, whatever device is
  // current when the first call needs them.
  cudaError_t create(cudaStream_t own, int device) {
    if (fork) return cudaSuccess;
    int current = device, priority = 0;
    cudaError_t e = cudaGetDevice(&current);
    if (e == cudaSuccess && current != device) e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaStreamGetPriority(own, &priority);
    for (int i = 0; i < LANES - 1 && e == cudaSuccess; ++i) {
      if (!aux[i]) e = cudaStreamCreateWithPriority(&aux[i], cudaStreamNonBlocking, priority);
      if (e == cudaSuccess && !join[i]) e = cudaEventCreateWithFlags(&join[i], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
    if (current != device) cudaSetDevice(current);
    return e;
  }
  void destroy() {
    for (int i = 0; i < LANES - 1; ++i) {
      if (aux[i]) cudaStreamDestroy(aux[i]);
      if (join[i]) cudaEventDestroy(join[i]);
    }
    if (fork) cudaEventDestroy(fork);
    *this = LaneStreams{};
  }
  cudaStream_t lane(int i, cudaStream_t own) const { return i == 0 ? own : aux[i - 1]; }
};

// Captured steps of the chunks (LB_OPT_USE_GRAPH): a long call is issued
// REPLAY_STEPS steps of a chunk at a time, so that its caller is free again
// while the GPU works. Launched one by one, a step of 24 groups takes the caller
// 40 us of its 66, and once a stream's queue of about 1000 launches is full the
// call waits for the GPU. Caller's time of 2000 steps, launched / replayed, us a
// step: 24 cylinders of 64 x 4 x 256 in FP32 60 / 1.1 of 65 / 62, one in FP64
// 35 / 0.05 of 72. The steps themselves take 0.96 to 1.06 of their time (four-wall
// ellipsoids FP32 67.7 / 68.9, FP16 62.7 / 60.7; 43 MB instances 77.6 / 82.3), the
// same with 16 to 128 steps in a graph. A graph is made at a chunk's first long
// call, under the steps launched before it; shorter calls would not earn it back.
constexpr int REPLAY_STEPS = 32;
constexpr long long REPLAY_MIN = 8 * REPLAY_STEPS;
constexpr size_t REPLAY_CHUNKS = 256;  // more are launched one by one: graphs hold memory

struct Replays {
  std::vector<cudaGraphExec_t> exec;  // [2 chunk + buffer that the first step reads]
  long long key = -1;                 // of the captured launches

  void clear() {
    for (cudaGraphExec_t x : exec)
      if (x) cudaGraphExecDestroy(x);
    exec.clear();
  }
  // Whether n steps of `chunks` chunks on `own` are replayed; graphs of another
  // key (or another plan) are dropped. Not while the caller captures `own`.
  bool ready(long long n, size_t chunks, long long key_, cudaStream_t own) {
    if (n < REPLAY_MIN || chunks > REPLAY_CHUNKS) return false;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(own, &st) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (st != cudaStreamCaptureStatusNone) return false;
    if (key_ != key || exec.size() != 2 * chunks) {
      clear();
      exec.assign(2 * chunks, nullptr);
      key = key_;
    }
    return true;
  }
  // REPLAY_STEPS steps of a chunk on `on`; step(i, stream) enqueues the i-th one
  // (for the capture, on `work`).
  template <class F>
  cudaError_t launch(size_t at, cudaStream_t work, cudaStream_t on, F&& step) {
    cudaGraphExec_t& x = exec[at];
    if (!x) {
      cudaError_t e = cudaStreamBeginCapture(work, cudaStreamCaptureModeThreadLocal);
      if (e != cudaSuccess) return e;
      for (int i = 0; i < REPLAY_STEPS && e == cudaSuccess; ++i) e = step(i, work);
      cudaGraph_t g = nullptr;
      const cudaError_t e2 = cudaStreamEndCapture(work, &g);
      if (e == cudaSuccess) e = e2;
      if (e == cudaSuccess) e = cudaGraphInstantiate(&x, g, 0);
      if (g) cudaGraphDestroy(g);
      if (e != cudaSuccess) return e;
    }
    return cudaGraphLaunch(x, on);
  }
};

// n steps of every chunk on created streams: launch(chunk, step, stream)
// enqueues one step of one chunk. The streams' launches are issued in turn, and
// every stream is joined back to `own` even after a failed launch. With
// `replays` (ready) all but the first n % REPLAY_STEPS steps are replayed;
// `buffer` is the buffer that step 0 reads.
template <class F>
cudaError_t run_lanes(LaneStreams& ls, const std::vector<LaneChunk>& plan, long long n, cudaStream_t own,
                      Replays* replays, int buffer, F&& launch) {
  std::vector<const LaneChunk*> todo[LANES];
  for (const LaneChunk& c : plan) todo[c.lane].push_back(&c);
  // (one chunk: no event between its chained launches and those before)
  cudaError_t e = plan.size() > 1 ? cudaEventRecord(ls.fork, own) : cudaSuccess;
  if (e != cudaSuccess) return e;
  for (int l = 1; l < LANES && e == cudaSuccess; ++l)
    if (!todo[l].empty()) e = cudaStreamWaitEvent(ls.aux[l - 1], ls.fork, 0);
  size_t longest = 0;
  for (auto& t : todo) longest = std::max(longest, t.size());
  const long long single = replays ? n % REPLAY_STEPS : n;
  for (size_t k = 0; k < longest; ++k)
    for (long long i = 0; i < n; i += i < single ? 1 : REPLAY_STEPS)
      for (int l = 0; l < LANES && e == cudaSuccess; ++l) {
        if (k >= todo[l].size()) continue;
        const LaneChunk& c = *todo[l][k];
        if (i < single)
          e = launch(c, i, ls.lane(l, own));
        else
          e = replays->launch(2 * size_t(&c - plan.data()) + size_t((buffer ^ i) & 1), ls.aux[0], ls.lane(l, own),
                              [&](int j, cudaStream_t s) { return launch(c, i + j, s); });
      }
  for (int l = 1; l < LANES; ++l) {
    if (todo[l].empty()) continue;
    cudaError_t e2 = cudaEventRecord(ls.join[l - 1], ls.aux[l - 1]);
    if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(own, ls.join[l - 1], 0);
    if (e == cudaSuccess) e = e2;
  }
  return e;
}

}  // namespace lbgm
