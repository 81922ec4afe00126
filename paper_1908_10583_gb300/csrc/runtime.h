// Host-side state of the query engine, shared by capi.cu and server.cu.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <condition_variable>
#include <functional>
#include <mutex>

#include "fora.h"
#include "fora_engine.cuh"

namespace fora {

// The residual list's unit counts of small batches have a buffer of this many pairs; larger
// batches keep theirs in the top-k scratch, which is free then.
constexpr int kUnitPairs = 4096;

// Device bytes of every buffer of a query workspace for nsrc sources of a graph with n
// nodes and hub_chunks hub items (workspace_sizes).  The workspace allocates exactly
// these; the server's admission and fora_workspace_bytes count them.
struct WorkspaceSizes {
  size_t N = 0;  // nsrc * n
  size_t r = 0, res = 0, tally = 0, q = 0, fa = 0, hub = 0, small = 0, work = 0, alist = 0,
         slot_cnt = 0, pre = 0, ps = 0, err = 0, sources = 0, rmax = 0, stats = 0, stopped = 0,
         light = 0, tile_dirty = 0, last_edges = 0, blk = 0,
         topk = 0, feat = 0, pred = 0, rmax_learned = 0, out_ids = 0, out_vals = 0;
  size_t total() const;  // q and hub count twice (Workspace::q, Workspace::hub)
};
WorkspaceSizes workspace_sizes(int64_t n, uint64_t hub_chunks, int nsrc);

template <typename T>
void dfree(T*& p) {
  if (p) cudaFree((void*)p);
  p = nullptr;
}

// Device and pinned host buffers of one in-flight batched query (up to `cap` sources).
// A graph owns one for its own entry points; the server owns one per lane.  A
// workspace serves one call at a time (its mutex).
struct Workspace {
  // workspace for up to `cap` sources
  int cap = 0;
  double* r = nullptr;
  double* res = nullptr;
  // walk ends of every source (BatchDev::acc), then the walk counts of a debug call
  unsigned long long* tally = nullptr;
  // q[0]: the frontier, then the residual entries; q[1]: the take's list of units and the copies
  // of the hot nodes' residues, then the walk offsets.  hub[0]: hub items, hub[1]: their lengths.
  unsigned long long* q[2] = {nullptr, nullptr};
  unsigned long long* hub[2] = {nullptr, nullptr};
  double* fa = nullptr;  // increments, then walk weights, then estimates
  unsigned long long* small = nullptr;  // PushCtl, totals[2] (from 4 on), walk_next (6)
  unsigned long long* work = nullptr;   // work counters of the spread, meeting points of the push
  uint32_t* alist = nullptr;      // groups of sources that the next take scans whole
  uint32_t* slot_cnt = nullptr;   // [4][nsrc] frontier entries and hub items of each group
  unsigned long long* pre = nullptr;  // [2][nsrc + 1] prefixes of the groups' items and hub items
  uint32_t* err = nullptr;
  int32_t* sources = nullptr;
  double* rmax = nullptr;
  SlotStats* stats = nullptr;
  uint32_t* stopped = nullptr;        // [nsrc] balanced push: the cost rule stopped the source
  uint8_t* light = nullptr;           // state of each group in the push (BatchDev::light)
  uint8_t* tile_dirty = nullptr;      // bits of the units a light round's spread touched
  unsigned long long* last_edges = nullptr;  // [nsrc]
  unsigned long long* blk = nullptr;  // [2][kUnitPairs]
  void* topk_scratch = nullptr;
  float* feat = nullptr;        // learned r_max: features [cap][16], predictions, r_max
  float* pred = nullptr;
  double* rmax_learned = nullptr;
  int32_t* out_ids = nullptr;  // device staging of host-bound results [cap][FORA_MAX_K]
  double* out_vals = nullptr;
  // pinned host mirrors
  unsigned long long* h_counters = nullptr;
  SlotStats* h_stats = nullptr;
  uint32_t* h_err = nullptr;
  int32_t* h_sources = nullptr;
  double* h_rmax = nullptr;
  uint32_t* go_host = nullptr;      // pinned: PushState::go of the host-driven push loop
  uint32_t* push_err = nullptr;     // pinned: err after a launch of a push that sources can join
  PushHost* push_host = nullptr;    // pinned
  cudaEvent_t part_ev[2] = {};      // ends of a long push's launches, by turn
  cudaEvent_t ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};

  PushState* ps = nullptr;
  std::mutex mu;

  void release() {
    dfree(ps);
    dfree(r); dfree(res); dfree(tally);
    dfree(q[0]); dfree(q[1]); dfree(hub[0]); dfree(hub[1]); dfree(fa);
    dfree(small); work = nullptr; dfree(alist); dfree(slot_cnt); dfree(pre); dfree(err); dfree(sources); dfree(rmax); dfree(stats); dfree(stopped); dfree(light); dfree(tile_dirty); dfree(last_edges); dfree(blk);
    if (topk_scratch) cudaFree(topk_scratch);
    topk_scratch = nullptr;
    dfree(out_ids); dfree(out_vals); dfree(feat); dfree(pred); dfree(rmax_learned);
    if (h_counters) cudaFreeHost(h_counters);
    if (h_stats) cudaFreeHost(h_stats);
    if (h_err) cudaFreeHost(h_err);
    if (h_sources) cudaFreeHost(h_sources);
    if (h_rmax) cudaFreeHost(h_rmax);
    if (go_host) cudaFreeHost(go_host);
    if (push_err) cudaFreeHost(push_err);
    if (push_host) cudaFreeHost(push_host);
    h_counters = nullptr; h_stats = nullptr; h_err = nullptr; h_sources = nullptr; h_rmax = nullptr;
    go_host = nullptr; push_err = nullptr; push_host = nullptr;
    cap = 0;
  }
  ~Workspace() {
    release();
    for (int i = 0; i < 5; ++i)
      if (ev[i]) cudaEventDestroy(ev[i]);
    for (int i = 0; i < 2; ++i)
      if (part_ev[i]) cudaEventDestroy(part_ev[i]);
  }
};

}  // namespace fora

namespace fora {

// Ordering between consecutive parts of a pipelined batch: the later part's push waits
// on the device until the earlier part's push is done.  The earlier part's host thread records `ev` after
// enqueueing its push and signals; it signals without recording if it stops early.
struct PipeLink {
  std::mutex m;
  std::condition_variable cv;
  bool signalled = false;
  bool recorded = false;
  cudaEvent_t ev = nullptr;
  void signal(bool rec) {
    {
      std::lock_guard<std::mutex> lk(m);
      if (signalled) return;
      signalled = true;
      recorded = rec;
    }
    cv.notify_all();
  }
  bool wait() {  // true if ev was recorded
    std::unique_lock<std::mutex> lk(m);
    cv.wait(lk, [&] { return signalled; });
    return recorded;
  }
};
struct PipeHook {
  PipeLink* before = nullptr;  // wait for this one before the push
  PipeLink* after = nullptr;   // signal this one after enqueueing the push
};
constexpr int kMaxPipeline = 4;

// Device memory of short calls (the select alone, the network's), in the order of a stream.  It
// comes from a pool of the library's, one per device, that keeps up to kScratchKept bytes between
// calls, for any thread and stream, and gives them back when a graph is destroyed.  (Out of the
// device's default pool, which keeps nothing over a synchronise, the scratch of 24 rows took 145
// of the 328 us of fora_topk.)
constexpr uint64_t kScratchKept = 64ull << 20;
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st);
void scratch_free(void* p, cudaStream_t st);
void scratch_trim(int device);

// Admission of further sources while a batch is in its push rounds (the serving lanes):
// `poll`, called again and again meanwhile (so it is cheap while nothing is new), may write up to `room` sources to `dst` (HOST) and
// returns how many; after the running round they join the batch as its next slots and
// their queries run exactly as they would alone.  The batch then has *nsrc_final sources
// (outputs and stats are sized for `cap`).
struct JoinHook {
  int cap = 0;
  std::function<int(int32_t* dst, int room)> poll;
  int* nsrc_final = nullptr;
};

}  // namespace fora

struct fora_graph {
  int64_t n = 0, m = 0, max_deg = 0;
  uint64_t hub_chunks = 0;  // sum over nodes with d > kHubChunk of ceil(d / kHubChunk)
  uint32_t* row = nullptr;
  int32_t* col = nullptr;
  uint32_t* indeg = nullptr;  // in-degrees (features of the learned r_max)
  double* invd = nullptr;     // RN(1 / d(v)) per node
  float* fdeg = nullptr;      // RN32(d(v)) per node
  // the walks' numbering and adjacency (GraphDev::wcol and the following)
  uint32_t* wcol = nullptr;
  uint32_t* wid = nullptr;
  uint2* wcls = nullptr;
  uint2* wesc = nullptr;
  int ncls = 0, wbits = 1;
  uint32_t* scol = nullptr;   // the spread's target codes (GraphDev::scol), or null
  uint32_t* hot_node = nullptr;
  uint8_t* hot_first = nullptr;  // GraphDev::hot_first
  int nhot = 0;
  // FORA+ walk index (Section 3.3): ends of omega_max(v) walks from every v
  unsigned long long* idx_off = nullptr;  // [n + 1] exclusive prefix of omega_max
  uint32_t* idx_dest = nullptr;           // [idx_entries] walk ends (walk ids)
  int64_t idx_entries = 0;
  double idx_rmax = 0.0, idx_scale = 0.0, idx_alpha = 0.0;
  uint64_t idx_seed = 0;
  bool idx_zero_hop = false;  // the stored walks are zero-hop walks (Section 4.1)
  int device = 0;
  int num_sms = 0;
  fora::Tuning tune;
  std::mutex mu;              // guards `tune`
  std::atomic<long long> push_launches{0};  // of k_push, of all calls so far
  fora::Workspace ws;         // the graph's own entry points
  // parts of a pipelined batch: a workspace and a stream each
  fora::Workspace pipe_ws[fora::kMaxPipeline];
  cudaStream_t pipe_stream[fora::kMaxPipeline] = {};
  fora::GraphDev dev() const {
    return fora::GraphDev{n,    m,    row,  col,   invd, fdeg, wcol,     wid,
                          wcls, wesc, ncls, wbits, fora::end_cols(n, wbits), scol, hot_node, hot_first, nhot};
  }
};

namespace fora {

// Engine entry points (capi.cu).
int report_error(int code, const char* fmt, ...);
struct RmaxSource {
  const double* host = nullptr;
  const double* device = nullptr;
};
// Allocate w for nsrc queries of g now (under w's lock).
int reserve_workspace(fora_graph* g, Workspace* w, int nsrc);
int run_batch_ws(fora_graph* g, Workspace* w, const fora_params* p, const int32_t* sources,
                 int nsrc, int32_t* out_ids, double* out_vals, fora_stats* st,
                 const fora_debug_io* dbg, uint32_t dbg_flags, cudaStream_t stream,
                 RmaxSource rsrc, const PipeHook* hook = nullptr,
                 const fora_balance* bal = nullptr, const JoinHook* join = nullptr);

}  // namespace fora
