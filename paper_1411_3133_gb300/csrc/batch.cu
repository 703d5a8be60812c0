// Batches of contexts of different geometry (lb_batch_* of include/lbgm.h).
//
// Every instance of every member becomes one ListInst record; instances are
// grouped by kernel variant (metric kind; in 2-byte storage also the parity of
// n3 and the row kind). One batch step is one work-list launch over the tiles
// of a group's nodes per LIST_MAX of its instances, the launches after the
// first on forked streams.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/lbgm.h"
#include "ctx.h"
#include "launch.h"

using namespace lbgm;

namespace {


struct Group {
  int key = 0;  // variant()
  int K = 0;
  int ninst = 0;
  std::vector<unsigned char> recs;  // ListInst records
  std::vector<int> work;            // nodes (FP32, FP64) or warps (2-byte storage) of each instance
  int blocks_per_sm = 0;            // occupancy of the kernel at the built block size
  Dims d{};                         // 2-byte storage: an instance of the group
  size_t smem = 0;                  // 2-byte storage: staged rows of a block, bytes
};

}  // namespace

struct lb_batch {
  std::vector<lb_ctx*> m;
  lb_precision prec = LB_FP32;
  cudaStream_t stream = nullptr;
  int device = 0;
  int nsm = 0;
  long long nodes = 0;

  // work list, valid while built
  bool built = false;
  int built_threads = 0;
  int built_tile_blocks = 0;
  std::vector<int> base_cur;  // member buffer parity when the records were written
  int parity = 0;             // batch steps since then, mod 2
  std::vector<Group> g;
  int block_work = 0;         // nodes (FP32, FP64) or warps (2-byte storage) of a block

  LaneStreams lanes;
  Replays replays;              // of plan's chunks, or of flat's where there is no plan
  std::vector<LaneChunk> plan;  // a call of several steps: chunks of the groups' instances
  std::vector<LaneChunk> flat;  // one step: every instance, LIST_MAX to a launch

  int threads = 128;
  int tile_blocks = 1;  // LB_OPT_TILE_BLOCKS: nodes per tile = tile_blocks x threads
  int schedule = 0;
  int use_graph = 0;
  long long check_every = 0;
  cudaGraphExec_t graph = nullptr;  // two batch steps, parity 0 then 1
  int graph_threads = 0;
  int graph_tile_blocks = 0;
  int graph_schedule = -1;

  long long step = 0;
  bool poisoned = false;
  std::string err;
};

namespace {

lb_status bfail(lb_batch* b, lb_status s, const std::string& msg) {
  if (!b) return ctx_fail(nullptr, s, msg);
  b->err = msg;
  if (s == LB_ERR_CUDA) b->poisoned = true;
  return s;
}

lb_status bcuda(lb_batch* b, cudaError_t e, const char* what) {
  return bfail(b, LB_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define LB_BCUDA(b, call)                                \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return bcuda(b, e_, #call);   \
  } while (0)

void drop_graph(lb_batch* b) {
  if (b->graph) cudaGraphExecDestroy(b->graph);
  b->graph = nullptr;
  b->replays.clear();
}

template <class S, class R>
ListInst<S, R> record(const lb_ctx* c, int bi, int cur, const GeoDev<R>& geo) {
  ListInst<S, R> r{};
  r.d = c->dims;
  r.d.batch = 1;
  if (c->dims.ref) r.d.ref = c->dims.ref + size_t(bi) * Q * size_t(c->dims.nr) * size_t(c->dims.geo_rows3);
  if (c->dims.st) r.d.st = c->dims.st + size_t(bi) * 2 * ST_K * size_t(c->dims.nr) * size_t(c->dims.st_rows3);
  r.geo = geo;
  r.ip = static_cast<const InstParams<R>*>(c->inst) + bi;
  const size_t off = size_t(bi) * Q * c->ncell;
  r.f0 = static_cast<const S*>(c->f[cur]) + off;
  r.f1 = static_cast<S*>(c->f[1 - cur]) + off;
  r.flag = c->flag;
  return r;
}

// Kernel variant of a member: its group key.
int variant(const lb_ctx* c) {
  return c->K * 4 + (c->elem_bytes == 2 ? (c->dims.n3 % 2) * 2 + (c->dims.st_row_r ? 1 : 0) : 0);
}

template <class S, class R>
void append_records(const lb_batch* b, int key, std::vector<unsigned char>& bytes, int* ninst,
                    const GeoDev<R> lb_ctx::*geo_member) {
  for (const lb_ctx* c : b->m) {
    if (variant(c) != key) continue;
    for (int bi = 0; bi < c->batch; ++bi) {
      const ListInst<S, R> r = record<S, R>(c, bi, c->cur, c->*geo_member);
      const unsigned char* p = reinterpret_cast<const unsigned char*>(&r);
      bytes.insert(bytes.end(), p, p + sizeof(r));
      ++*ninst;
    }
  }
}

int max_threads(lb_precision p) { return p == LB_FP64 ? 256 : 128; }  // the kernels' launch bounds

cudaError_t occupancy(lb_precision p, const Group& g, int threads, int* out) {
  switch (p) {
    case LB_FP64: return step_list_occupancy_f64(g.K, threads, out);
    case LB_FP32: return step_list_occupancy_f32(g.K, threads, out);
    case LB_FP16_SHIFTED: return step_list_occupancy_h16(g.K, g.d, g.smem, threads, out);
    default: return step_list_occupancy_b16(g.K, g.d, g.smem, threads, out);
  }
}

// Write the instance records (with the members' current buffer parity) and plan
// their launches for block size b->threads. Host only: the launches carry the
// records.
lb_status build(lb_batch* b) {
  drop_graph(b);
  b->built = false;
  b->g.clear();
  const bool pairs = b->prec == LB_FP16_SHIFTED || b->prec == LB_BF16_SHIFTED;
  b->block_work = pairs ? b->threads / 32 : b->threads;
  std::vector<int> keys;
  for (int K : {int(KCYL), int(KELL), int(KFLAT)})
    for (int v = 0; v < 4; ++v) keys.push_back(K * 4 + v);
  for (int key : keys) {
    Group gr;
    gr.key = key;
    gr.K = key / 4;
    switch (b->prec) {
      case LB_FP64: append_records<double, double>(b, key, gr.recs, &gr.ninst, &lb_ctx::geo_d); break;
      case LB_FP32: append_records<float, float>(b, key, gr.recs, &gr.ninst, &lb_ctx::geo_f); break;
      case LB_FP16_SHIFTED: append_records<__half, float>(b, key, gr.recs, &gr.ninst, &lb_ctx::geo_f); break;
      default: append_records<__nv_bfloat16, float>(b, key, gr.recs, &gr.ninst, &lb_ctx::geo_f); break;
    }
    if (gr.ninst == 0) continue;
    for (const lb_ctx* c : b->m) {
      if (variant(c) != key) continue;
      gr.work.insert(gr.work.end(), size_t(c->batch), pairs ? int(pair_warps(c->dims)) : c->dims.ncell);
      if (pairs) {
        gr.d = c->dims;
        gr.smem = std::max(gr.smem, pair_smem_bytes(c->dims, b->threads / 32));
      }
    }
    cudaError_t e = occupancy(b->prec, gr, b->threads, &gr.blocks_per_sm);
    if (e != cudaSuccess) return bcuda(b, e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    b->g.push_back(std::move(gr));
  }
  // chunk indices count within their group
  b->flat.clear();
  std::vector<LaneInst> inst;
  std::vector<int> first;
  for (size_t gi = 0; gi < b->g.size(); ++gi) {
    first.push_back(int(inst.size()));
    for (const lb_ctx* c : b->m)
      if (variant(c) == b->g[gi].key)
        inst.insert(inst.end(), size_t(c->batch), {int(gi), c->ncell, c->step_bytes});
    for (int i = 0; i < b->g[gi].ninst; i += LIST_MAX)
      b->flat.push_back({int(gi), i, std::min(LIST_MAX, b->g[gi].ninst - i), int(b->flat.size()) % LANES});
  }
  b->plan = plan_lanes(inst, LIST_MAX);
  for (LaneChunk& c : b->plan) c.first -= first[size_t(c.group)];
  b->base_cur.resize(b->m.size());
  for (size_t i = 0; i < b->m.size(); ++i) b->base_cur[i] = b->m[i]->cur;
  b->parity = 0;
  b->built_threads = b->threads;
  b->built_tile_blocks = b->tile_blocks;
  b->built = true;
  return LB_OK;
}

// The records hold f0 = the buffer each member read when they were written;
// they stay valid while every member has taken exactly the batch's steps.
bool records_current(const lb_batch* b) {
  if (!b->built || b->built_threads != b->threads || b->built_tile_blocks != b->tile_blocks) return false;
  for (size_t i = 0; i < b->m.size(); ++i)
    if (b->m[i]->cur != (b->base_cur[i] ^ b->parity)) return false;
  return true;
}

// One step of a chunk of one group's instances on stream s, at parity `par`;
// chained: see launch_chained. A work item is a tile of tile_blocks blocks'
// worth of nodes, halved while the launch has fewer than two items per SM: the
// groups of lanes.h are short launches, and with tiles of 4 blocks' worth 18 unlike
// channels (300 000 nodes) took 68 us a step in BF16, 35 now (49 before there were
// groups; 35 with tiles of one block's worth).
cudaError_t launch_chunk(const lb_batch* b, const LaneChunk& c, int par, bool chained, cudaStream_t s) {
  const Group& gr = b->g[size_t(c.group)];
  const int grid = b->schedule == 1 ? std::max(1, gr.blocks_per_sm) * b->nsm : 0;
  const void* recs = gr.recs.data() + gr.recs.size() / size_t(gr.ninst) * size_t(c.first);
  int items[LIST_MAX], tile = 0;
  long long n = 0;
  for (int blocks = b->tile_blocks; n == 0 || (n < 2 * b->nsm && blocks > 0); blocks /= 2) {
    tile = b->block_work * blocks;
    n = 0;
    for (int i = 0; i < c.count; ++i) n += items[i] = (gr.work[size_t(c.first + i)] + tile - 1) / tile;
  }
  if (b->prec == LB_FP64) chained = chained && fp64_chains(grid > 0 ? std::min<long long>(grid, n) : n);
  switch (b->prec) {
    case LB_FP64: return launch_step_list_f64(gr.K, recs, c.count, items, tile, b->threads, grid, par, chained, s);
    case LB_FP32: return launch_step_list_f32(gr.K, recs, c.count, items, tile, b->threads, grid, par, chained, s);
    case LB_FP16_SHIFTED:
      return launch_step_list_h16(gr.K, gr.d, gr.smem, recs, c.count, items, tile, b->threads, grid, par, chained, s);
    default:
      return launch_step_list_b16(gr.K, gr.d, gr.smem, recs, c.count, items, tile, b->threads, grid, par, chained, s);
  }
}

// n batch steps: the chunks read the same buffers and write disjoint nodes, so
// they run side by side on the lanes; several steps in the order of lanes.h.
lb_status steps(lb_batch* b, long long n, Replays* replays) {
  const std::vector<LaneChunk>& plan = n >= LANE_MIN_STEPS && !b->plan.empty() ? b->plan : b->flat;
  const int par = b->parity;
  // one chunk: chained launches; several without a plan meet after every step
  const bool chained = plan.size() == 1;
  const long long each = !chained && &plan == &b->flat ? 1 : n;
  cudaError_t e = cudaSuccess;
  for (long long i0 = 0; i0 < n && e == cudaSuccess; i0 += each)
    e = run_lanes(b->lanes, plan, each, b->stream, replays, par, [&](const LaneChunk& c, long long i, cudaStream_t s) {
      return launch_chunk(b, c, int(par ^ ((i0 + i) & 1)), chained, s);
    });
  if (e != cudaSuccess) return bcuda(b, e, "step kernel launch");
  b->parity = int(par ^ (n & 1));
  return LB_OK;
}

lb_status step_once(lb_batch* b) { return steps(b, 1, nullptr); }

void advance_members(lb_batch* b, long long n) {
  for (lb_ctx* c : b->m) {
    c->step += n;
    if (n & 1) c->cur ^= 1;
  }
  b->step += n;
}

lb_status check_members(lb_batch* b) {
  for (size_t i = 0; i < b->m.size(); ++i) {
    lb_ctx* c = b->m[i];
    int h = 0;
    LB_BCUDA(b, cudaMemcpyAsync(&h, c->flag, sizeof(int), cudaMemcpyDeviceToHost, b->stream));
    LB_BCUDA(b, cudaStreamSynchronize(b->stream));
    if (h) {
      const std::string m = "non-finite density in batch member " + std::to_string(i) + " after step " +
                            std::to_string(c->step);
      ctx_fail(c, LB_ERR_NONFINITE, m);
      return bfail(b, LB_ERR_NONFINITE, m);
    }
  }
  return LB_OK;
}

lb_status ready(lb_batch* b) {
  if (!b) return bfail(nullptr, LB_ERR_ARG, "null batch");
  if (b->poisoned) return bfail(b, LB_ERR_STATE, "batch poisoned by an earlier failure: " + b->err);
  for (size_t i = 0; i < b->m.size(); ++i) {
    lb_status s;
    if (!ctx_usable(b->m[i], &s))
      return bfail(b, LB_ERR_STATE, "member " + std::to_string(i) + ": " + b->m[i]->err);
    if (b->m[i]->K == KELT)
      return bfail(b, LB_ERR_ARG, "member " + std::to_string(i) +
                                      " is a theta-resolved ellipsoid, which only the plain step kernel carries");
    if (b->m[i]->any_shift)
      return bfail(b, LB_ERR_ARG, "member " + std::to_string(i) +
                                      " uses the half-force velocity (old_forcing 2), which only the plain "
                                      "step kernel carries");
  }
  return LB_OK;
}

// n > 0 steps without a check: in groups where that pays (lanes.h), else a step at a time.
lb_status advance(lb_batch* b, long long n, bool graph) {
  const bool grouped = n >= LANE_MIN_STEPS && !b->plan.empty();
  const bool replay = graph && b->use_graph && (grouped || b->flat.size() == 1) &&
                      b->replays.ready(n, grouped ? b->plan.size() : 1, b->schedule, b->stream);
  if (grouped || replay) {
    lb_status s = steps(b, n, replay ? &b->replays : nullptr);
    if (s == LB_OK) advance_members(b, n);
    return s;
  }
  if (graph && b->use_graph && b->check_every == 0 && n >= 3 && b->flat.size() > 1) {
    if (b->parity != 0) {  // the captured pair starts at parity 0
      lb_status s = step_once(b);
      if (s != LB_OK) return s;
      advance_members(b, 1);
      --n;
    }
    if (!b->graph || b->graph_threads != b->threads || b->graph_schedule != b->schedule ||
        b->graph_tile_blocks != b->tile_blocks) {
      drop_graph(b);
      cudaGraph_t g = nullptr;
      LB_BCUDA(b, cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
      lb_status s1 = step_once(b);
      lb_status s2 = s1 == LB_OK ? step_once(b) : s1;
      cudaError_t e = cudaStreamEndCapture(b->stream, &g);
      if (s2 != LB_OK) return s2;
      if (e != cudaSuccess) return bcuda(b, e, "cudaStreamEndCapture");
      e = cudaGraphInstantiate(&b->graph, g, 0);
      cudaGraphDestroy(g);
      if (e != cudaSuccess) return bcuda(b, e, "cudaGraphInstantiate");
      b->graph_threads = b->threads;
      b->graph_tile_blocks = b->tile_blocks;
      b->graph_schedule = b->schedule;
    }
    const long long pairs = n / 2;
    for (long long i = 0; i < pairs; ++i) LB_BCUDA(b, cudaGraphLaunch(b->graph, b->stream));
    advance_members(b, 2 * pairs);
    n &= 1;
  }
  for (long long i = 0; i < n; ++i) {
    lb_status s = step_once(b);
    if (s != LB_OK) return s;
    advance_members(b, 1);
  }
  return LB_OK;
}

// n steps; trials of the autotuner pass graph = false.
lb_status run(lb_batch* b, long long n, bool graph) {
  lb_status s;
  if (!records_current(b) && (s = build(b)) != LB_OK) return s;
  while (n > 0) {  // from check to check
    const long long k = b->check_every > 0 ? std::min(n, b->check_every - b->step % b->check_every) : n;
    if ((s = advance(b, k, graph)) != LB_OK) return s;
    n -= k;
    if (b->check_every > 0 && b->step % b->check_every == 0 && (s = check_members(b)) != LB_OK) return s;
  }
  return LB_OK;
}

}  // namespace

extern "C" {

lb_status lb_batch_create(lb_ctx* const* members, int count, lb_batch** out) {
  if (!members || !out) return bfail(nullptr, LB_ERR_ARG, "null argument");
  *out = nullptr;
  if (count < 1) return bfail(nullptr, LB_ERR_ARG, "need count >= 1");
  lb_batch* b = new lb_batch();
  auto bail = [&](lb_status s, const std::string& m) {
    lb_batch_destroy(b);
    return bfail(nullptr, s, m);
  };
  long long nodes = 0;
  for (int i = 0; i < count; ++i) {
    lb_ctx* c = members[i];
    if (!c) return bail(LB_ERR_ARG, "member " + std::to_string(i) + " is NULL");
    for (int j = 0; j < i; ++j)
      if (members[j] == c) return bail(LB_ERR_ARG, "member " + std::to_string(i) + " appears twice");
    if (i > 0 && (c->prec != b->prec || c->device != b->device || c->stream != b->stream))
      return bail(LB_ERR_ARG, "member " + std::to_string(i) + " differs in precision, device or stream");
    if (i == 0) {
      b->prec = c->prec;
      b->device = c->device;
      b->stream = c->stream;
    }
    b->m.push_back(c);
    nodes += (long long)c->batch * (long long)c->ncell;
  }
  b->nodes = nodes;
  int cur_dev = 0;
  cudaError_t e = cudaGetDevice(&cur_dev);
  if (e == cudaSuccess && cur_dev != b->device) e = cudaErrorInvalidDevice;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->nsm, cudaDevAttrMultiProcessorCount, b->device);
  if (e == cudaSuccess) e = b->lanes.create(b->stream, b->device);
  if (e != cudaSuccess) return bail(LB_ERR_CUDA, std::string("batch setup: ") + cudaGetErrorString(e));
  *out = b;
  return LB_OK;
}

lb_status lb_batch_step(lb_batch* b, long long n) {
  lb_status s = ready(b);
  if (s != LB_OK) return s;
  if (n < 0) return bfail(b, LB_ERR_ARG, "need n >= 0");
  return run(b, n, true);
}

lb_status lb_batch_set_option(lb_batch* b, int option, long long value) {
  if (!b) return bfail(nullptr, LB_ERR_ARG, "null batch");
  switch (option) {
    case LB_OPT_CHECK_EVERY:
      if (value < 0) return bfail(b, LB_ERR_ARG, "need k >= 0");
      b->check_every = value;
      return LB_OK;
    case LB_OPT_BLOCK_THREADS:
      if (value < 64 || value > 256 || value % 32) return bfail(b, LB_ERR_ARG, "need 64..256, multiple of 32");
      // tiles are block-sized: the work-list kernel's bound (128 with FP32
      // arithmetic) caps the block
      b->threads = std::min(int(value), max_threads(b->prec));
      return LB_OK;
    case LB_OPT_USE_GRAPH:
      b->use_graph = value ? 1 : 0;
      return LB_OK;
    case LB_OPT_SCHEDULE:
      if (value < 0 || value > 1) return bfail(b, LB_ERR_ARG, "need 0 (tile per block) or 1 (persistent)");
      b->schedule = int(value);
      return LB_OK;
    case LB_OPT_TILE_BLOCKS:
      if (value != 1 && value != 2 && value != 4) return bfail(b, LB_ERR_ARG, "need 1, 2 or 4 blocks per tile");
      b->tile_blocks = int(value);
      return LB_OK;
    default:
      return bfail(b, LB_ERR_ARG, "option not available for batches");
  }
}

lb_status lb_batch_autotune(lb_batch* b, int steps_per_trial, lb_tune* best, lb_tune* trials, int max_trials,
                            int* n_trials) {
  lb_status s = ready(b);
  if (s != LB_OK) return s;
  if (steps_per_trial < 1) return bfail(b, LB_ERR_ARG, "need steps_per_trial >= 1");
  if (max_trials < 0 || (max_trials > 0 && !trials)) return bfail(b, LB_ERR_ARG, "bad trials buffer");
  std::vector<lb_tune> cand;
  for (int t : {64, 96, 128, 192, 256})
    if (t <= max_threads(b->prec))
      for (int sc : {0, 1})
        for (int tb : {1, 2, 4}) cand.push_back({t, sc, t * tb, 0.0});
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  LB_BCUDA(b, cudaEventCreate(&e0));
  cudaError_t e = cudaEventCreate(&e1);
  if (e != cudaSuccess) {
    cudaEventDestroy(e0);
    return bcuda(b, e, "cudaEventCreate");
  }
  const long long keep_check = b->check_every;
  b->check_every = 0;
  for (lb_tune& k : cand) {
    b->threads = k.block_threads;
    b->schedule = k.schedule;
    b->tile_blocks = k.tile_nodes / k.block_threads;
    s = run(b, 1, false);  // rebuilds the tiles for this block size; untimed
    if (s != LB_OK) break;
    if ((e = cudaEventRecord(e0, b->stream)) != cudaSuccess) {
      s = bcuda(b, e, "cudaEventRecord");
      break;
    }
    s = run(b, steps_per_trial, false);
    if (s != LB_OK) break;
    float ms = 0.f;
    e = cudaEventRecord(e1, b->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e != cudaSuccess) {
      s = bcuda(b, e, "timing a trial");
      break;
    }
    k.ms_per_step = double(ms) / steps_per_trial;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  b->check_every = keep_check;
  if (s != LB_OK) return s;
  size_t ib = 0;
  for (size_t i = 1; i < cand.size(); ++i)
    if (cand[i].ms_per_step < cand[ib].ms_per_step) ib = i;
  b->threads = cand[ib].block_threads;
  b->schedule = cand[ib].schedule;
  b->tile_blocks = cand[ib].tile_nodes / cand[ib].block_threads;
  if (best) *best = cand[ib];
  const int n = int(cand.size());
  for (int i = 0; i < n && i < max_trials; ++i) trials[i] = cand[i];
  if (n_trials) *n_trials = n;
  if (keep_check > 0) return check_members(b);
  return LB_OK;
}

long long lb_batch_nodes(const lb_batch* b) { return b ? b->nodes : -1; }

long long lb_batch_step_count(const lb_batch* b) { return b ? b->step : -1; }

void lb_batch_destroy(lb_batch* b) {
  if (!b) return;
  if (b->stream) cudaStreamSynchronize(b->stream);
  drop_graph(b);
  b->lanes.destroy();
  delete b;
}

const char* lb_batch_last_error(const lb_batch* b) { return b ? b->err.c_str() : lb_last_error(nullptr); }

}  // extern "C"
