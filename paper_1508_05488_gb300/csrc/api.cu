// api.cu -- the C ABI (include/cch.h): argument checks, per-stream
// workspaces, launch planning and the kernel sequence of one call.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <vector>

#include "cch.h"
#include "cch_internal.cuh"

namespace cch {
namespace {

constexpr size_t kAlign = 256;
size_t up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

struct Dims {
  int64_t N;
  int32_t nsets;
  int32_t nchunk1;
  int32_t ntile2;
  int64_t max_sort_tiles, max_spa_tiles, max_chain_blks, max_out_tiles, Nc;
};

Dims make_dims(int64_t N, int32_t nsets, int32_t nchunk1, int32_t ntile2) {
  Dims d;
  d.N = N;
  d.nsets = nsets;
  d.nchunk1 = nchunk1;
  d.ntile2 = ntile2;
  d.Nc = N + 8 * (int64_t)nsets;
  d.max_sort_tiles = N / kSortTile + nsets + 1;
  d.max_spa_tiles = N / kSpaTile + 4 * (int64_t)nsets + 1;
  d.max_chain_blks = d.Nc / kChainBlk + 4 * (int64_t)nsets + 1;
  d.max_out_tiles = d.Nc / kOutTile + 4 * (int64_t)nsets + 1;
  return d;
}

// Byte layout of a workspace; `base` null -> sizes only.
struct Layout {
  size_t total = 0;
  size_t ctl_bytes = 0;                  // ctl + ctr (cleared each call)
  size_t status_off = 0, status_bytes = 0;   // look-back words (cleared on epoch wrap)
  Ws w{};
};

Layout layout(const Dims& d, char* base) {
  Layout L;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t r = o; o = up(o + bytes); return base ? base + r : nullptr; };
  L.w.ctl = (SetCtl*)take(sizeof(SetCtl) * d.nsets);
  L.w.ctr = (uint32_t*)take(sizeof(uint32_t) * CT_COUNT);
  L.w.ptot = (uint4*)take(16 * ((size_t)d.ntile2 / kPlanTiles + d.nsets + 1));
  L.ctl_bytes = o;
  L.status_off = o;
  L.w.st_sort = (uint64_t*)take(8 * 256 * (size_t)d.max_sort_tiles);
  L.w.st_spa = (SpaStat*)take(sizeof(SpaStat) * (size_t)d.max_spa_tiles);
  L.w.st_spa_cnt = (uint64_t*)take(8 * (size_t)d.max_spa_tiles);
  L.w.st_out = (uint64_t*)take(8 * (size_t)d.max_out_tiles);
  L.status_bytes = o - L.status_off;
  L.w.part = (Part*)take(sizeof(Part) * (size_t)std::max(d.nchunk1, 1));
  L.w.tcnt = (uint64_t*)take(8 * 8 * (size_t)std::max(d.ntile2, 1));
  L.w.small_seg = (uint32_t*)take(4 * 4 * (size_t)d.nsets);
  L.w.keyA = (uint64_t*)take(8 * (size_t)d.N);
  L.w.keyB = (uint64_t*)take(8 * (size_t)d.N);
  L.w.valA = (uint32_t*)take(4 * (size_t)d.N);
  L.w.valB = (uint32_t*)take(4 * (size_t)d.N);
  L.w.spvA = (uint64_t*)take(8 * (size_t)d.N);
  L.w.spvB = (uint64_t*)take(8 * (size_t)d.N);
  L.w.hist = (uint32_t*)take(4 * (size_t)kSortPasses * 256 * d.nsets);
  L.w.sort_start = (uint32_t*)take(4 * ((size_t)d.nsets + 1));
  L.w.spa_start = (uint32_t*)take(4 * (4 * (size_t)d.nsets + 1));
  L.w.cpts = take(16 * (size_t)d.Nc);
  L.w.cidx = (uint32_t*)take(4 * (size_t)d.Nc);
  L.w.cprev = (uint32_t*)take(4 * (size_t)d.Nc);
  L.w.cnext = (uint32_t*)take(4 * (size_t)d.Nc);
  L.w.calive = (uint8_t*)take((size_t)d.Nc);
  L.w.chain_start = (uint32_t*)take(4 * (4 * (size_t)d.nsets + 1));
  L.w.blk_head = (int32_t*)take(4 * (size_t)d.max_chain_blks);
  L.w.blk_tail = (int32_t*)take(4 * (size_t)d.max_chain_blks);
  L.w.out_start = (uint32_t*)take(4 * (4 * (size_t)d.nsets + 1));
  L.w.stairs = (uint32_t*)take(4 * 4 * (size_t)kStairB * d.nsets);
  L.w.sv_hdr = (SieveHdr*)take(sizeof(SieveHdr) * d.nsets);
  L.w.sv_tab = (float4*)take(2 * sizeof(float4) * std::max<size_t>(kSvRefineRows + 2, (size_t)(kSvBatchRows + 2) * d.nsets));
  L.w.sv_cnt = (uint32_t*)take(4 * std::max<size_t>(kSvMaxUnits, kSvWarps * ((size_t)d.N / (kSvWarps * kSvBatchLen) + d.nsets + 1)));
  L.total = o;
  return L;
}

struct Workspace {
  std::mutex mu;                     // held while a call of the stream is enqueued
  bool released = false;             // by cch_release_workspace: the stream's next call takes a new one
  char* dev = nullptr;
  size_t bytes = 0;
  Dims cap{};
  uint32_t epoch = 0;                // of the last plain call
  bool uncleared = false;            // allocated while a graph was captured: cleared by its runs only
  bool captured = false;             // a graph holds `dev`
  std::vector<char*> retired;        // earlier buffers and tables that a graph holds
  std::vector<char*> retired_host;   // its tables' staging
  char* host_tab = nullptr;          // pinned staging of a batch's tables
  char* dev_tab = nullptr;           // their device copy
  size_t tab_bytes = 0;              // size of both
  cudaEvent_t tab_done = nullptr;    // staging buffer free again
  cudaStream_t side = nullptr;       // the pipeline beside k_set (run)
  cudaEvent_t fork = nullptr, join = nullptr;
  void* h2d = nullptr;               // device copy of host points (cch_hull_host)
  size_t h2d_bytes = 0;
  int32_t* dcount = nullptr;         // device counts (cch_hull_host)
  int32_t* didx = nullptr;
  size_t didx_bytes = 0;
};

// g_mu guards the table of workspaces and the stage events; each workspace has a
// lock of its own, so that calls on different streams are enqueued side by side
// (8 threads on as many streams, 60,001 points: 43 us a call behind one lock,
// 30 so).
std::mutex g_mu;
std::map<cudaStream_t, std::shared_ptr<Workspace>> g_ws;
std::atomic<uint64_t> g_launches{0};

// Optional stage timing: CUDA events around the stages of every call, read
// back (and summed) by cch_profile_read.
constexpr int kStages = 8;   // a1, stairs, a2, gather, small path, multi-block path, chain, blocked SPA
// The sieve's kernels, timed with the stages they stand for: k_table (sample),
// k_sieve (a2), k_refine (gather) and k_set on the lists (chain hull, output).
constexpr int kSieveStages = 4, kSieveStage[kSieveStages] = {1, 2, 3, 6};
struct ProfRec { cudaEvent_t ev[kStages + 1], sv[kSieveStages + 1]; uint32_t mask; bool sieve; };
std::atomic<uint32_t> g_prof{0};   // stages whose boundaries get events (bit k: stage k)
std::vector<ProfRec> g_prof_pending, g_prof_free;

cudaEvent_t* prof_begin(ProfRec& rec) {
  const uint32_t mask = g_prof;
  if (!mask) return nullptr;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_prof_free.empty()) { rec = g_prof_free.back(); g_prof_free.pop_back(); }
  else {
    for (auto& e : rec.ev) cudaEventCreate(&e);
    for (auto& e : rec.sv) cudaEventCreate(&e);
  }
  rec.mask = mask;
  rec.sieve = false;
  return rec.ev;
}
int g_sms = 0;
int g_occ[4] = {0, 0, 0, 0};   // a1 CTAs per SM, by input format

int sm_count() {
  if (g_sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_sms <= 0) g_sms = 1;
  }
  return g_sms;
}

bool fits(const Dims& c, const Dims& d) {
  return d.N <= c.N && d.nsets <= c.nsets && d.nchunk1 <= c.nchunk1 && d.ntile2 <= c.ntile2;
}

// The workspace of `stream`, locked.
std::shared_ptr<Workspace> lock_workspace(cudaStream_t stream, std::unique_lock<std::mutex>& lk) {
  for (;;) {
    std::shared_ptr<Workspace> ws;
    {
      std::lock_guard<std::mutex> g(g_mu);
      auto& slot = g_ws[stream];
      if (!slot) slot = std::make_shared<Workspace>();
      ws = slot;
    }
    lk = std::unique_lock<std::mutex>(ws->mu);
    if (!ws->released) return ws;
    lk.unlock();
  }
}

// Grow the workspace `ws` of `stream` to dims `d`; `graph`: the stream is being
// captured.  A buffer that a graph holds stays allocated until the workspace is
// released: the graph may be launched again.  Called with its lock held.
int acquire(cudaStream_t stream, const Dims& d, Workspace* ws, bool graph) {
  if (!ws->dev || !fits(ws->cap, d)) {
    Dims c = d;
    if (ws->dev) {   // grow by at least 1.5x to amortise
      c.N = std::max(d.N, ws->cap.N + ws->cap.N / 2);
      c.nsets = std::max(d.nsets, ws->cap.nsets);
      c.nchunk1 = std::max(d.nchunk1, ws->cap.nchunk1);
      c.ntile2 = std::max(d.ntile2, ws->cap.ntile2);
      c = make_dims(c.N, c.nsets, c.nchunk1, (int32_t)std::max<int64_t>(c.ntile2, c.N / kClsMinTile + c.nsets + 1));
      if (cudaStreamSynchronize(stream) != cudaSuccess) return CCH_ERR_CUDA;
      if (ws->captured) ws->retired.push_back(ws->dev);
      else cudaFree(ws->dev);
      ws->dev = nullptr;
      ws->captured = false;
    }
    Layout L = layout(c, nullptr);
    if (cudaMalloc(&ws->dev, L.total) != cudaSuccess) {
      cudaGetLastError();
      ws->dev = nullptr;
      return CCH_ERR_NOMEM;
    }
    if (cudaMemsetAsync(ws->dev, 0, L.total, stream) != cudaSuccess) return CCH_ERR_CUDA;
    if (!ws->side) {                 // optional: without it everything stays on the caller's stream
      if (cudaStreamCreateWithFlags(&ws->side, cudaStreamNonBlocking) != cudaSuccess ||
          cudaEventCreateWithFlags(&ws->fork, cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&ws->join, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        ws->join = nullptr;
      }
    }
    ws->bytes = L.total;
    ws->cap = c;
    ws->epoch = 0;
    ws->uncleared = graph;
  } else if (ws->uncleared && !graph) {
    if (cudaMemsetAsync(ws->dev, 0, ws->bytes, stream) != cudaSuccess) return CCH_ERR_CUDA;
    ws->uncleared = false;
  }
  ws->captured |= graph;
  return CCH_OK;
}

int a1_target(int dtype) {
  if (!g_occ[dtype]) g_occ[dtype] = extremes_blocks_per_sm(dtype);
  return sm_count() * g_occ[dtype];
}

int grid_cap() { return sm_count() * 4; }

struct StageOut {
  int32_t* r1_idx;
  int32_t* r1_region;
  int32_t* spa_idx;
};

// The sets of a batch: the pipeline's, and the small ones of k_set by class.
struct Batch {
  std::vector<SetDesc> sets;
  std::vector<SieveSet> sieve;           // of the pipeline's sets
  std::vector<int32_t> cta;              // set of every k_sieve CTA
  std::vector<SetItem> items[kSetClasses];
};

// Staging for a batch's tables: the workspace's, free of the last call's copy.
// A graph copies from the staging on every run, so a captured call has its own,
// kept until the workspace is released (an event recorded under a capture could
// not be waited for, and a later call would change the graph's tables).
int stage_tables(Workspace* ws, size_t bytes, cudaStream_t stream, bool graph, char*& host, char*& dev) {
  if (graph) {
    host = dev = nullptr;
    if (cudaMallocHost(&host, bytes) != cudaSuccess || cudaMalloc(&dev, bytes) != cudaSuccess) {
      cudaGetLastError();
      if (host) cudaFreeHost(host);
      return CCH_ERR_NOMEM;
    }
    ws->retired_host.push_back(host);
    ws->retired.push_back(dev);
    return CCH_OK;
  }
  if (!ws->tab_done && cudaEventCreateWithFlags(&ws->tab_done, cudaEventDisableTiming) != cudaSuccess) return CCH_ERR_CUDA;
  if (cudaEventSynchronize(ws->tab_done) != cudaSuccess) return CCH_ERR_CUDA;
  if (ws->tab_bytes < bytes) {
    if (cudaStreamSynchronize(stream) != cudaSuccess) return CCH_ERR_CUDA;   // earlier calls read the old copy
    if (ws->host_tab) cudaFreeHost(ws->host_tab);
    if (ws->dev_tab) cudaFree(ws->dev_tab);
    ws->host_tab = ws->dev_tab = nullptr;
    ws->tab_bytes = 0;
    const size_t cap = bytes + bytes / 2;
    if (cudaMallocHost(&ws->host_tab, cap) != cudaSuccess || cudaMalloc(&ws->dev_tab, cap) != cudaSuccess) {
      cudaGetLastError();
      if (ws->host_tab) cudaFreeHost(ws->host_tab);
      ws->host_tab = ws->dev_tab = nullptr;
      return CCH_ERR_NOMEM;
    }
    ws->tab_bytes = cap;
  }
  host = ws->host_tab;
  dev = ws->dev_tab;
  return CCH_OK;
}

// Copy a batch's tables (small sets by class, then the larger sets) to the
// device; *items: the small sets'.  `graph`: the stream is being captured.
// Called with its lock held.
int copy_tables(Job& j, const Batch& b, Workspace* ws, cudaStream_t stream, bool graph, const SetItem** items) {
  size_t ibytes = 0;
  for (const auto& v : b.items) ibytes += sizeof(SetItem) * v.size();
  const size_t sets_off = (ibytes + 63) / 64 * 64;
  const size_t sv_off = sets_off + (sizeof(SetDesc) * b.sets.size() + 63) / 64 * 64;
  const size_t cta_off = sv_off + sizeof(SieveSet) * b.sieve.size();
  const size_t bytes = cta_off + sizeof(int32_t) * b.cta.size();
  char *host, *dev;
  const int st = stage_tables(ws, bytes, stream, graph, host, dev);
  if (st != CCH_OK) return st;
  size_t o = 0;
  for (const auto& v : b.items) {
    if (!v.empty()) memcpy(host + o, v.data(), sizeof(SetItem) * v.size());
    o += sizeof(SetItem) * v.size();
  }
  if (!b.sets.empty()) {
    memcpy(host + sets_off, b.sets.data(), sizeof(SetDesc) * b.sets.size());
    memcpy(host + sv_off, b.sieve.data(), sizeof(SieveSet) * b.sieve.size());
    if (!b.cta.empty()) memcpy(host + cta_off, b.cta.data(), sizeof(int32_t) * b.cta.size());
  }
  if (cudaMemcpyAsync(dev, host, bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess) return CCH_ERR_CUDA;
  if (!graph && cudaEventRecord(ws->tab_done, stream) != cudaSuccess) return CCH_ERR_CUDA;
  *items = reinterpret_cast<const SetItem*>(dev);
  if (!b.cta.empty()) {
    j.sv_sets = reinterpret_cast<const SieveSet*>(dev + sv_off);
    j.sv_cta = reinterpret_cast<const int32_t*>(dev + cta_off);
    j.sv_nctas = (int32_t)b.cta.size();
    j.sv_all = b.sets.size() <= (size_t)sm_count();
  }
  j.sets = reinterpret_cast<const SetDesc*>(dev + sets_off);
  return CCH_OK;
}

// k_set on a batch's small sets; the number of kernels launched.  Beside larger
// sets they run on the workspace's stream, launched last: they take the SMs that
// the others' latency-bound kernels leave (64 float64 sets of up to 2^18 points,
// most of them small: 163 us one after the other, 127 so; launched first: 129, and
// 203 against 199 on 64 int32 sets of up to 2^20).
int launch_small_sets(const Job& j, const Batch& b, const SetItem* items, cudaStream_t stream) {
  int nk = 0;
  size_t o = 0;
  for (int c = 0; c < kSetClasses; c++) o += b.items[c].size();
  // the largest sets first; a class starts beside the one before it where that
  // leaves SMs free (1024 int32 sets, 213, 103, 94 and 205 of them small: 285 us
  // a call, 343 one class after the other); where it does not, sharing an SM
  // costs both their L1 (4096 float64 sets of 256 to 4096 points: 259 us
  // beside, 224 one after the other)
  const size_t sms = (size_t)sm_count(), above = b.items[1].size() + b.items[2].size() + b.items[3].size();
  size_t prev = 0;
  for (int c = kSetClasses - 1; c >= 0; c--) {
    o -= b.items[c].size();
    const size_t count = b.items[c].size();
    const bool beside = prev != 0 && prev <= 2 * sms, split = set_splits(j, c) && 4 * above <= sms;
    if (count) prev = split ? 4 * count : count;
    nk += launch_set(j, c, items + o, (int)count, split, beside, stream);
  }
  return nk;
}

// Launch the whole call: k_set on a batch's small sets, the pipeline on the
// others (`batch` nullptr: the single set of j.one).  `stages` hooks the
// stage extraction.
int run(Job& j, const Batch* batch, cudaStream_t stream, StageOut* stages, std::shared_ptr<Workspace>* ws_out) {
  Dims d = make_dims(j.N, j.nsets, j.nchunk1, j.ntile2);
  std::unique_lock<std::mutex> lk;
  const std::shared_ptr<Workspace> held = lock_workspace(stream, lk);
  Workspace* ws = held.get();
  int nk = 0;
  const bool graph = capturing(stream);
  // every allocation first: a call that fails for want of memory launches nothing
  if (!batch || !batch->sets.empty()) {
    const int st = acquire(stream, d, ws, graph);
    if (st != CCH_OK) return st;
  }
  const SetItem* items = nullptr;
  bool small = false;                  // small sets beside larger ones, launched after them
  if (batch) {
    const int st = copy_tables(j, *batch, ws, stream, graph, &items);
    if (st != CCH_OK) return st;
    size_t nsmall = 0;
    for (const auto& v : batch->items) nsmall += v.size();
    small = nsmall != 0 && !batch->sets.empty() && ws->join && !g_prof;
    if (!small) nk += launch_small_sets(j, *batch, items, stream);
    else if (cudaEventRecord(ws->fork, stream) != cudaSuccess) return CCH_ERR_CUDA;
    if (batch->sets.empty()) {
      g_launches += (uint64_t)nk;
      return cudaGetLastError() == cudaSuccess ? CCH_OK : CCH_ERR_CUDA;
    }
  }
  Layout L = layout(ws->cap, ws->dev);
  if (graph) {
    j.epoch = kEpochGraph;
  } else {
    if (++ws->epoch > kEpochLast) {
      if (cudaMemsetAsync(ws->dev + L.status_off, 0, L.status_bytes, stream) != cudaSuccess) return CCH_ERR_CUDA;
      ws->epoch = 1;
    }
    j.epoch = ws->epoch;
  }
  // (a sieved single set's: by k_table)
  if (!j.sieve.nunit && cudaMemsetAsync(ws->dev, 0, L.ctl_bytes, stream) != cudaSuccess) return CCH_ERR_CUDA;
  if (stages) { j.r1_idx = stages->r1_idx; j.r1_region = stages->r1_region; }
  ProfRec rec{};
  cudaEvent_t* ev = prof_begin(rec);
  // The sieve's lists, then k_set on them and the pipeline, which has nothing
  // to do for a sieved call: each of its nine launches still waits for the one
  // before it, 10 us in all after k_set, so it runs on a stream of the
  // workspace beside k_set and joins the caller's (not when stages are timed).
  bool side = false;
  if (j.sieve.nunit || j.sv_sets) {
    rec.sieve = true;
    // sieve event k marks the start of its stage k (and the end of k - 1)
    auto mark_sv = [&](int k) {
      if (ev && ((k < kSieveStages && (rec.mask >> kSieveStage[k]) & 1u) || (k > 0 && (rec.mask >> kSieveStage[k - 1]) & 1u)))
        cudaEventRecord(rec.sv[k], stream);
    };
    mark_sv(0);
    nk += launch_table(j, L.w, sm_count(), stream);
    mark_sv(1);
    nk += launch_sieve(j, L.w, stream);
    mark_sv(2);
    nk += launch_refine(j, L.w, stream);
    side = !ev && !j.sv_sets && ws->join;
    if (side && (cudaEventRecord(ws->fork, stream) != cudaSuccess ||
                 cudaStreamWaitEvent(ws->side, ws->fork, 0) != cudaSuccess)) return CCH_ERR_CUDA;
    mark_sv(3);
    nk += launch_set_list(j, L.w, sm_count(), stream);
    mark_sv(4);
  }
  // (on the pipeline's stream: a sieved run's lists do not wait for it)
  if (graph && cudaMemsetAsync(ws->dev + L.status_off, 0, L.status_bytes, side ? ws->side : stream) != cudaSuccess)
    return CCH_ERR_CUDA;
  Launch La{side ? ws->side : stream, grid_cap(), j.tune.cls_per_sm * sm_count()};
  // event k marks the start of stage k (and the end of stage k - 1)
  auto mark = [&](int k) {
    if (ev && ((rec.mask >> k) & 1u || (k > 0 && (rec.mask >> (k - 1)) & 1u))) cudaEventRecord(ev[k], stream);
  };
  mark(0);
  nk += launch_extremes(j, L.w, La);
  mark(1);
  nk += launch_stairs(j, L.w, La);
  mark(2);
  nk += launch_classify(j, L.w, La);
  mark(3);
  nk += launch_gather(j, L.w, La);
  mark(4);
  nk += launch_small(j, L.w, La);
  mark(5);
  nk += launch_big(j, L.w, La);
  mark(6);
  nk += launch_chain(j, L.w, La);
  mark(7);
  if (small) {
    if (cudaStreamWaitEvent(ws->side, ws->fork, 0) != cudaSuccess) return CCH_ERR_CUDA;
    nk += launch_small_sets(j, *batch, items, ws->side);
  }
  if ((side || small) && (cudaEventRecord(ws->join, ws->side) != cudaSuccess ||
                          cudaStreamWaitEvent(stream, ws->join, 0) != cudaSuccess)) return CCH_ERR_CUDA;
  if (stages) {
    if (j.opts & OPT_BLOCKED_SPA) nk += launch_spa_blocked(j, L.w, stages->spa_idx, stream);
    else { launch_extract_spa(j, L.w, stages->spa_idx, stream); nk++; }
  }
  mark(8);
  if (ev) {
    std::lock_guard<std::mutex> g(g_mu);
    g_prof_pending.push_back(rec);
  }
  g_launches += (uint64_t)nk;
  if (cudaGetLastError() != cudaSuccess) return CCH_ERR_CUDA;
  if (ws_out) *ws_out = held;
  return CCH_OK;
}

int check_common(const void* points, int64_t n, int dtype, const void* out_idx, const void* out_count) {
  if (dtype != CCH_I32 && dtype != CCH_F64) return CCH_ERR_DTYPE;
  if (n < 0 || !out_idx || !out_count) return CCH_ERR_INVALID;
  if (n > 0 && !points) return CCH_ERR_INVALID;
  if (n > kMaxSetPoints) return CCH_ERR_RANGE;
  uintptr_t a = (uintptr_t)points;
  if (a % (dtype == CCH_F64 ? 16 : 8)) return CCH_ERR_INVALID;
  return CCH_OK;
}

// Single-set job.
Job single_job(const void* points, int64_t n, int dtype, int32_t* out_idx, int32_t* out_count,
               uint32_t opts) {
  Job j{};
  j.pts = points;
  j.N = n;
  j.nsets = 1;
  j.dtype = dtype;
  j.opts = opts;
  j.tune = tune_for(dtype, n, 1);
  j.fast_max = j.tune.small_max == kTuneDefault.small_max ? kFastSmallMax : (uint32_t)j.tune.small_max;
  int target = a1_target(dtype);
  int64_t len = (n + target - 1) / std::max(target, 1);
  len = std::max<int64_t>(j.tune.a1_len_min, (len + 1023) / 1024 * 1024);
  j.chunk1_len = len;
  int32_t nch = (int32_t)((n + len - 1) / len);
  j.nchunk1 = nch;
  const int ct = cls_tile(dtype);
  j.ntile2 = (int32_t)((n + ct - 1) / ct);
  j.nchunk3 = n > 0 ? (int32_t)((stairs_sample(n, j.tune) + kStairChunk - 1) / kStairChunk) : 0;
  j.nchunkP = (j.ntile2 + kPlanTiles - 1) / kPlanTiles;
  j.sets = nullptr;
  j.one = SetDesc{0, n, 0, nch, 0, j.ntile2, 0, j.nchunk3, 0, j.nchunkP, 0};
  j.out_idx = out_idx;
  j.out_counts = out_count;
  return j;
}

// A single set small enough for k_set: one launch, no workspace.
Job set_job(const void* points, const float* ys, int64_t n, int dtype, int32_t* out_idx, int32_t* out_count) {
  Job j{};
  j.pts = points;
  j.ys = ys;
  j.N = n;
  j.nsets = 1;
  j.dtype = dtype;
  j.out_idx = out_idx;
  j.out_counts = out_count;
  return j;
}

int run_set(const Job& j, cudaStream_t stream) {
  const int cls = set_class(j.N);
  g_launches += (uint64_t)launch_set(j, cls, nullptr, 1, set_splits(j, cls), false, stream);
  return cudaGetLastError() == cudaSuccess ? CCH_OK : CCH_ERR_CUDA;
}

}  // namespace

void count_launches(uint64_t n) { g_launches += n; }

}  // namespace cch

using namespace cch;

extern "C" {

const char* cch_status_string(int status) {
  switch (status) {
    case CCH_OK: return "ok";
    case CCH_ERR_INVALID: return "invalid argument";
    case CCH_ERR_DTYPE: return "unsupported dtype (use CCH_I32 or CCH_F64)";
    case CCH_ERR_NONFINITE: return "non-finite float64 coordinate";
    case CCH_ERR_RANGE: return "size or coordinate magnitude outside the supported range";
    case CCH_ERR_NOMEM: return "out of memory";
    case CCH_ERR_CUDA: return "CUDA runtime error";
    case CCH_ERR_TIMEOUT: return "bounded device wait expired";
    case CCH_ERR_BUSY: return "server queue full";
    case CCH_ERR_NOTFOUND: return "unknown ticket";
    default: return "unknown status";
  }
}

int cch_hull(const void* points, int64_t n, int dtype, int32_t* out_idx, int32_t* out_count,
             void* stream) {
  int st = check_common(points, n, dtype, out_idx, out_count);
  if (st != CCH_OK) return st;
  if (n <= kSetOne) return run_set(set_job(points, nullptr, n, dtype, out_idx, out_count), (cudaStream_t)stream);
  Job j = single_job(points, n, dtype, out_idx, out_count, 0);
  j.sieve = sieve_set(0, n, dtype, sm_count());
  j.fast_sort = dtype != CCH_I32;
  return run(j, nullptr, (cudaStream_t)stream, nullptr, nullptr);
}

int cch_hull_batched(const void* points, const int64_t* offsets, int32_t nsets, int dtype,
                     int32_t* out_idx, int32_t* out_counts, void* stream) {
  if (dtype != CCH_I32 && dtype != CCH_F64) return CCH_ERR_DTYPE;
  if (nsets < 0 || !offsets || !out_idx || !out_counts) return CCH_ERR_INVALID;
  if (nsets == 0) return CCH_OK;
  if (offsets[0] != 0) return CCH_ERR_INVALID;
  const int64_t N = offsets[nsets];
  if (N > 0x7FFFFFFFll) return CCH_ERR_RANGE;
  if (N > 0 && !points) return CCH_ERR_INVALID;
  if ((uintptr_t)points % (dtype == CCH_F64 ? 16 : 8)) return CCH_ERR_INVALID;
  if (nsets == 1) return cch_hull(points, N, dtype, out_idx, out_counts, stream);   // one set's kernels, not a batch's
  Batch batch;
  const Tune tune = tune_for(dtype, N, nsets);
  int target = a1_target(dtype);
  int64_t len = std::max<int64_t>(tune.a1_len_min, ((N + target - 1) / std::max(target, 1) + 1023) / 1024 * 1024);
  int64_t nch = 0, nt = 0, n3 = 0, np_ = 0;
  const int ct = cls_tile(dtype);
  int32_t small[kSetClasses] = {}, larger = 0, large = 0;   // k_set's by class, others, those above the sieve of few
  for (int32_t s = 0; s < nsets; s++) {
    const int64_t n = offsets[s + 1] - offsets[s];
    if (n < 0) return CCH_ERR_INVALID;
    if (n > kMaxSetPoints) return CCH_ERR_RANGE;
    const int cls = set_class(n);
    if (cls >= 0) small[cls]++;
    else larger++;
    large += n > (int64_t)kSvBatchFew * kSvBatchLen;
  }
  for (int c = 0; c < kSetClasses; c++) batch.items[c].reserve(small[c]);
  batch.sets.reserve(larger);
  batch.sieve.reserve(larger);
  const int32_t units =
      large >= sm_count() ? kSvBatchUnits : large == 0 || larger - large >= kSvBatchSets ? kSvBatchFew : 0;
  for (int32_t s = 0; s < nsets; s++) {
    const int64_t n = offsets[s + 1] - offsets[s];
    const int cls = set_class(n);
    if (cls >= 0) {
      batch.items[cls].push_back(SetItem{offsets[s], (int32_t)n, s});
      continue;
    }
    int32_t c = (int32_t)((n + len - 1) / len);
    int32_t t = (int32_t)((n + ct - 1) / ct);
    int32_t c3 = (int32_t)((stairs_sample(n, tune) + kStairChunk - 1) / kStairChunk);
    int32_t cp = (t + kPlanTiles - 1) / kPlanTiles;
    batch.sets.push_back(
        SetDesc{offsets[s], n, (int32_t)nch, c, (int32_t)nt, t, (int32_t)n3, c3, (int32_t)np_, cp, s});
    const SieveSet sv = sieve_batch_set(offsets[s], n, (int32_t)batch.cta.size(), units);
    batch.cta.insert(batch.cta.end(), (size_t)(sv.nunit + kSvWarps - 1) / kSvWarps, (int32_t)batch.sieve.size());
    batch.sieve.push_back(sv);
    nch += c;
    nt += t;
    n3 += c3;
    np_ += cp;
  }
  Job j{};
  j.pts = points;
  j.N = N;
  j.nsets = (int32_t)batch.sets.size();
  j.dtype = dtype;
  j.tune = tune;
  j.nchunk1 = (int32_t)nch;
  j.ntile2 = (int32_t)nt;
  j.nchunk3 = (int32_t)n3;
  j.nchunkP = (int32_t)np_;
  j.chunk1_len = len;
  j.out_idx = out_idx;
  j.out_counts = out_counts;
  return run(j, &batch, (cudaStream_t)stream, nullptr, nullptr);
}

int cch_hull_host(const void* points_host, int64_t n, int dtype, int32_t* out_idx_host,
                  int32_t* out_count, void* stream) {
  if (dtype != CCH_I32 && dtype != CCH_F64) return CCH_ERR_DTYPE;
  if (n < 0 || !out_idx_host || !out_count || (n > 0 && !points_host)) return CCH_ERR_INVALID;
  if (n > kMaxSetPoints) return CCH_ERR_RANGE;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t pbytes = (size_t)n * (dtype == CCH_F64 ? 16 : 8);
  void* dpts = nullptr;
  int32_t* dcount = nullptr;
  int32_t* didx = nullptr;
  {
    std::unique_lock<std::mutex> lk;
    const std::shared_ptr<Workspace> ws = lock_workspace(s, lk);
    if (ws->h2d_bytes < pbytes) {
      if (ws->h2d) { cudaStreamSynchronize(s); cudaFree(ws->h2d); }
      ws->h2d = nullptr;
      ws->h2d_bytes = 0;
      if (cudaMalloc(&ws->h2d, pbytes) != cudaSuccess) { cudaGetLastError(); return CCH_ERR_NOMEM; }
      ws->h2d_bytes = pbytes;
    }
    size_t ib = 4 * (size_t)std::max<int64_t>(n, 1);
    if (ws->didx_bytes < ib) {
      if (ws->didx) { cudaStreamSynchronize(s); cudaFree(ws->didx); }
      ws->didx = nullptr;
      ws->didx_bytes = 0;
      if (cudaMalloc(&ws->didx, ib) != cudaSuccess) { cudaGetLastError(); return CCH_ERR_NOMEM; }
      ws->didx_bytes = ib;
    }
    if (!ws->dcount && cudaMalloc(&ws->dcount, 16) != cudaSuccess) { cudaGetLastError(); return CCH_ERR_NOMEM; }
    dpts = ws->h2d;
    dcount = ws->dcount;
    didx = ws->didx;
  }
  if (pbytes && cudaMemcpyAsync(dpts, points_host, pbytes, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return CCH_ERR_CUDA;
  int st = cch_hull(dpts, n, dtype, didx, dcount, stream);
  if (st != CCH_OK) return st;
  if (cudaMemcpyAsync(out_count, dcount, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess) return CCH_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return CCH_ERR_CUDA;
  if (*out_count < 0) return *out_count;
  if (*out_count > 0 &&
      cudaMemcpyAsync(out_idx_host, didx, 4 * (size_t)*out_count, cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return CCH_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return CCH_ERR_CUDA;
  return CCH_OK;
}

int cch_hull_f32soa(const float* x, const float* y, int64_t n, int32_t* out_idx, int32_t* out_count,
                    void* stream) {
  if (n < 0 || !out_idx || !out_count || (n > 0 && (!x || !y))) return CCH_ERR_INVALID;
  if ((((uintptr_t)x | (uintptr_t)y) & 3u) != 0) return CCH_ERR_INVALID;
  if (n > kMaxSetPoints) return CCH_ERR_RANGE;
  if (n <= kSetOne) return run_set(set_job(x, y, n, DT_F32, out_idx, out_count), (cudaStream_t)stream);
  Job j = single_job(x, n, DT_F32, out_idx, out_count, 0);
  j.ys = y;
  j.sieve = sieve_set(0, n, DT_F32, sm_count());
  j.fast_sort = 1;
  return run(j, nullptr, (cudaStream_t)stream, nullptr, nullptr);
}

int cch_hull_stages(const void* points, int64_t n, int dtype, uint32_t opts, int32_t* r1_idx,
                    int32_t* r1_region, int32_t* spa_idx, int64_t* counts_host, int32_t* out_idx,
                    int32_t* out_count, void* stream) {
  int st = check_common(points, n, dtype, out_idx, out_count);
  if (st != CCH_OK) return st;
  if (!r1_idx || !r1_region || !spa_idx || !counts_host) return CCH_ERR_INVALID;
  if (opts & ~(uint32_t)(OPT_NO_FILTER | OPT_NO_PREFILTER | OPT_BLOCKED_SPA | OPT_OCTAGON)) return CCH_ERR_INVALID;
  if (opts & (OPT_BLOCKED_SPA | OPT_OCTAGON)) opts |= OPT_NO_PREFILTER;   // the paper's round 1 (or its octagon form)
  Job j = single_job(points, n, dtype, out_idx, out_count, opts);
  StageOut so{r1_idx, r1_region, spa_idx};
  std::shared_ptr<Workspace> ws;
  cudaStream_t s = (cudaStream_t)stream;
  st = run(j, nullptr, s, &so, &ws);
  if (st != CCH_OK) return st;
  SetCtl c;
  uint32_t ctr[CT_COUNT];
  Layout L = layout(ws->cap, ws->dev);
  if (cudaMemcpyAsync(&c, L.w.ctl, sizeof(SetCtl), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CCH_ERR_CUDA;
  if (cudaMemcpyAsync(ctr, L.w.ctr, sizeof(ctr), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CCH_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return CCH_ERR_CUDA;
  counts_host[0] = c.s1;
  for (int r = 0; r < 4; r++) counts_host[1 + r] = c.cnt[r];
  for (int r = 0; r < 4; r++) counts_host[5 + r] = (opts & OPT_BLOCKED_SPA) ? c.sb[r] : c.s2[r];
  counts_host[9] = c.status != 0 ? c.status : (int32_t)ctr[CT_ERR];
  counts_host[10] = c.passes;
  for (int r = 0; r < 4; r++) counts_host[11 + r] = (opts & OPT_OCTAGON) ? c.didx[r] : -1;
  counts_host[15] = 0;
  return CCH_OK;
}

int cch_profile(int enable) {
  std::lock_guard<std::mutex> lk(g_mu);
  g_prof = enable != 0 ? (1u << kStages) - 1u : 0u;
  return CCH_OK;
}

int cch_profile_stages(uint32_t mask) {
  std::lock_guard<std::mutex> lk(g_mu);
  g_prof = mask & ((1u << kStages) - 1u);
  return CCH_OK;
}

int cch_profile_read(double* stage_ms, int max_stages, int64_t* calls) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (!stage_ms || max_stages < 0) return CCH_ERR_INVALID;
  for (int k = 0; k < max_stages; k++) stage_ms[k] = 0.0;
  int64_t n = 0;
  for (auto& rec : g_prof_pending) {
    int last = 0;
    for (int k = 0; k < kStages; k++)
      if ((rec.mask >> k) & 1u) last = k + 1;
    if (cudaEventSynchronize(rec.ev[last]) != cudaSuccess) return CCH_ERR_CUDA;
    for (int k = 0; k < kStages && k < max_stages; k++) {
      if (!((rec.mask >> k) & 1u)) continue;
      float ms = 0.f;
      cudaEventElapsedTime(&ms, rec.ev[k], rec.ev[k + 1]);
      stage_ms[k] += ms;
    }
    for (int q = 0; rec.sieve && q < kSieveStages; q++) {
      const int k = kSieveStage[q];
      if (!((rec.mask >> k) & 1u) || k >= max_stages) continue;
      float ms = 0.f;
      cudaEventElapsedTime(&ms, rec.sv[q], rec.sv[q + 1]);
      stage_ms[k] += ms;
    }
    g_prof_free.push_back(rec);
    n++;
  }
  g_prof_pending.clear();
  if (calls) *calls = n;
  return kStages;
}

uint64_t cch_launch_count(void) { return g_launches.load(); }

int cch_route(void* stream, int32_t* route) {
  if (!route) return CCH_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  std::unique_lock<std::mutex> lk;
  const std::shared_ptr<Workspace> ws = lock_workspace(s, lk);
  if (!ws->dev) return CCH_ERR_NOTFOUND;
  const uint32_t* src = layout(ws->cap, ws->dev).w.ctr;
  uint32_t c[CT_COUNT];
  if (cudaMemcpyAsync(c, src, sizeof c, cudaMemcpyDeviceToHost, s) != cudaSuccess) return CCH_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return CCH_ERR_CUDA;
  route[0] = (int32_t)c[CT_SIEVED];
  route[1] = (int32_t)c[CT_SIEVE_SETS];
  route[2] = (int32_t)c[CT_SMALL_TOTAL];
  route[3] = (int32_t)c[CT_SORT_TOTAL];
  route[4] = (int32_t)c[CT_FAST_RUNS];
  route[5] = (c[CT_FAST_FAIL] | c[CT_FAST_FAIL2]) != 0;
  return CCH_OK;
}

namespace cch {
namespace {
// One thread waits on a flag that nothing sets, with the library's bounded
// wait; the error word it records is the result.
__global__ void k_selftest_wait(uint32_t* words, int32_t* status) {
  uint32_t* flag = words + CT_COUNT;
  uint32_t spins = 0;
  while (ld_acq_u32(flag) == 0)
    if (!spin_step(spins, words)) break;
  *status = (int32_t)ld_acq_u32(words + CT_ERR);
}
}  // namespace
}  // namespace cch

int cch_selftest_wait(int32_t* status_dev, void* stream) {
  if (!status_dev) return CCH_ERR_INVALID;
  static uint32_t* words = nullptr;           // CT_COUNT error words + the flag
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!words && cudaMalloc(&words, sizeof(uint32_t) * (CT_COUNT + 1)) != cudaSuccess) {
      cudaGetLastError();
      words = nullptr;
      return CCH_ERR_NOMEM;
    }
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemsetAsync(words, 0, sizeof(uint32_t) * (CT_COUNT + 1), st) != cudaSuccess) return CCH_ERR_CUDA;
  k_selftest_wait<<<1, 1, 0, st>>>(words, status_dev);
  g_launches += 1;
  return cudaGetLastError() == cudaSuccess ? CCH_OK : CCH_ERR_CUDA;
}

size_t cch_workspace_bytes(int64_t n, int dtype) {
  if (n < 0 || (dtype != CCH_I32 && dtype != CCH_F64)) return 0;
  int target = 1216;
  int64_t len = std::max<int64_t>(4096, ((n + target - 1) / target + 1023) / 1024 * 1024);
  Dims d = make_dims(n, 1, (int32_t)((n + len - 1) / len), (int32_t)((n + cls_tile(dtype) - 1) / cls_tile(dtype)));
  return layout(d, nullptr).total;
}

void cch_release_workspace(void) {
  std::map<cudaStream_t, std::shared_ptr<Workspace>> all;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    all.swap(g_ws);
  }
  for (auto& kv : all) {
    std::lock_guard<std::mutex> lk(kv.second->mu);   // a call that is being enqueued comes first
    kv.second->released = true;
  }
  cudaDeviceSynchronize();
  serve_release_pinned();
  for (auto& kv : all) {
    Workspace* ws = kv.second.get();
    if (ws->dev) cudaFree(ws->dev);
    for (char* p : ws->retired) cudaFree(p);
    for (char* p : ws->retired_host) cudaFreeHost(p);
    if (ws->host_tab) cudaFreeHost(ws->host_tab);
    if (ws->dev_tab) cudaFree(ws->dev_tab);
    if (ws->tab_done) cudaEventDestroy(ws->tab_done);
    if (ws->side) cudaStreamDestroy(ws->side);
    if (ws->fork) cudaEventDestroy(ws->fork);
    if (ws->join) cudaEventDestroy(ws->join);
    if (ws->h2d) cudaFree(ws->h2d);
    if (ws->dcount) cudaFree(ws->dcount);
    if (ws->didx) cudaFree(ws->didx);
  }
}

}  // extern "C"
