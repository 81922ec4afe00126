// Internal declarations of the FORA query engine (device state and kernel
// launchers).  Not part of the C ABI (include/fora.h is).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fora {

// Nodes with more out-edges than this are pushed in chunks of this many edges,
// one warp per chunk, so that a hub never serialises a round on one warp.
constexpr uint32_t kHubChunk = 256;

// Residues of one group of sources that a warp of the push's take reads at a time: 256 / gw
// nodes, whose changes in a light push round share one mark.
constexpr int kTakeUnit = 256;
// Nodes per entry of GraphDev::hot_first.
constexpr uint32_t kHotSpan = 64;
// Copies of the hot nodes' residues that a push spreads its pushes to them over.
constexpr int kHotCopies = 8;
// State of a group of sources in the push (BatchDev::light).
constexpr uint32_t kGroupLight = 1u;   // its next take scans the listed tiles only
constexpr uint32_t kGroupActive = 2u;  // it takes part in the next take
constexpr uint32_t kMaxPolls = 1u << 25;  // polls of a block at the push's barrier (about 30 s)
// Words (of 4 bytes) of a launch's part of BatchDev::meet.
constexpr int kMeetArrived = 0;  // arrivals of its blocks
constexpr int kMeetEntered = 1;  // blocks that have entered
constexpr int kMeetReady = 2;    // blocks that have cleared their part of the state
constexpr int kMeetWord = 8;     // 8 bytes, in another sector: the last meeting (k_push)
constexpr int kMeetWords = 32;   // from one launch's part to the other's

// Units of the residual list: all of a call (scanned by one block), and of one slot.
constexpr int kMaxUnits = 32768;
constexpr int kMaxSlotUnits = 4096;

// Top-k radix select: 96-bit keys (estimate bits : ~id), 12-bit digits.
constexpr int kDigitBits = 12;
constexpr int kBins = 1 << kDigitBits;
constexpr uint32_t kSortCap = 8192;  // candidates sorted in shared memory at the end

// Indexed walks: residues of more than kIndexedMost walks are listed, in a list whose length is
// counted in one word: the listed nodes from bit kListBits on, their chunks of kIndexedMost walks
// below.  A list serves at most index_list_groups groups of sources, so that neither count can
// leave its bits: a source has fewer than 2^32 walks (kErrWalkOverflow), so a group of gw sources
// lists at most gw * 2^32 / kIndexedMost nodes, and their chunks are at most as many again.
constexpr uint32_t kIndexedMost = 1024;
constexpr int kListBits = 36;
inline int64_t index_list_groups(int64_t n, int gw) {
  const int64_t most = (int64_t)gw * ((1ll << 32) / kIndexedMost);
  const int64_t nodes = n < most ? n : most, chunks = nodes + most;
  const int64_t a = ((1ll << (64 - kListBits)) - 1) / nodes, b = ((1ll << kListBits) - 1) / chunks;
  return a < b ? a : b;
}

// Device error bits (ORed into BatchDev::err).
constexpr uint32_t kErrWalkCap = 1u;
constexpr uint32_t kErrWalkOverflow = 2u;
constexpr uint32_t kErrPushNotConverged = 4u;
constexpr uint32_t kErrIndexRange = 8u;  // a residue needs more walks than the index holds
constexpr uint32_t kErrBounds = 16u;     // a device index check failed (FORA_DEBUG builds)
constexpr uint32_t kErrBarrier = 32u;    // a wait of the push's blocks for each other ran out
constexpr uint32_t kErrMissing = 64u;    // no push: the device had no room for all its blocks

// Device index checks of the FORA_DEBUG build: FORA_IN_RANGE(err, i, n) is true when
// i < n; otherwise it records kErrBounds in *err and is false, and the caller skips the
// access (the query then fails with FORA_ERR_BOUNDS).  In other builds it is `true` and
// costs nothing.
#ifdef FORA_DEBUG
__device__ __forceinline__ bool in_range_checked(uint32_t* err, unsigned long long i,
                                                 unsigned long long n) {
  if (i < n) return true;
  atomicOr(err, kErrBounds);
  return false;
}
#define FORA_IN_RANGE(err, i, n) \
  ::fora::in_range_checked((err), (unsigned long long)(i), (unsigned long long)(n))
#else
#define FORA_IN_RANGE(err, i, n) true
#endif
constexpr uint32_t kMaxPushRounds = 100000u;  // default cap of the push rounds

// Where the push loop stands: the parity of the current frontier queue, the number of
// rounds done, and the shape of the current frontier.  Kept on the device so the loop
// runs without the host.
struct PushState {
  int cur;
  uint32_t round;
  uint32_t go;      // the loop condition of the last round
  uint32_t pad;
  unsigned long long ngroups;  // items of `span` entries of the current frontier, over all groups
  unsigned long long nhub;     // hub items of the current frontier, over all groups
};
// A launch that runs part of a push: it ends after the round in which `slice` microseconds have
// passed or, when it may be stopped, a non-zero `stop` was seen, and after the spread of a round
// that takes longer.
struct PushHost {  // pinned host memory
  uint32_t stop;   // written by the host
  uint32_t go[2];  // what the launch with this turn left: kPushDone, kPushLeft, kPushMissing
};
constexpr uint32_t kPushDone = 0u;     // the push is through
constexpr uint32_t kPushLeft = 1u;     // rounds are left
constexpr uint32_t kPushMissing = 2u;  // nothing done: the device had no room for all blocks
struct PushPart {
  int resume;      // 0: from the start of the push, 1: where the launch before it ended
  int turn;        // alternates between 0 and 1, from 0
  uint32_t slice;  // kNoSlice: no limit
  int stops;       // read host->stop every round
  int sure;        // a cooperative launch: all blocks run together, whenever they can
  PushHost* host;  // may be null
};
constexpr uint32_t kNoSlice = 0xFFFFFFFFu;
struct PushCtl {
  uint32_t nheavy;  // groups that the next take scans whole (listed in BatchDev::alist)
  uint32_t nlist;   // units listed of the others (BatchDev::tlist)
  uint32_t span;    // entries of an item of the spread
  uint32_t cut;     // the launch ends after the spread, and the next begins with the take
};

struct GraphDev {
  int64_t n;
  int64_t m;
  const uint32_t* row;  // [n+1] edge offsets (m < 2^32)
  const int32_t* col;   // [m]
  const double* invd;   // [n] RN(1 / d(v)): the push increment is a product, not a quotient
  const float* fdeg;    // [n] RN32(d(v)), of the frontier test
  // The walks' own numbering and adjacency.  Nodes of equal out-degree have consecutive walk
  // ids and consecutive rows of wcol, so a node's first edge is wcls[c].x + id * d with its
  // degree class c (d = wcls[c].y), and an edge record {class : 32 - wbits bits, walk id :
  // wbits bits} holds all that the next move needs: one 4-byte gather per move.  (A gather
  // of a node record and one of a packed target, 2.8 sectors per move, kept the walks at the
  // SMs' limit of one gathered sector per clock.)  The lowest ncls degrees have classes; the
  // other nodes have the class ncls and the lowest walk ids, their {first edge, degree} in
  // wesc[id].
  const uint32_t* wcol;  // [m] edge records
  const uint32_t* wid;   // [n] record of node v
  const uint2* wcls;     // [ncls]
  const uint2* wesc;     // [nodes of class ncls]
  int ncls;
  int wbits;
  uint32_t ecols;        // end_cols(n, wbits)
  // The spread's copy of the targets (null when the graph has no hot nodes): the target
  // id, or kHotBit | h for the h-th hot node (a node of high in-degree, hot_node[h]), whose
  // increments go to one of several copies of its residue.
  const uint32_t* scol;
  const uint32_t* hot_node;  // [nhot] ascending ids
  const uint8_t* hot_first;  // [ceil(n / kHotSpan) + 1]: hot nodes below node t * kHotSpan
  int nhot;
};

// Hot targets of the spread: at most kHotSlots nodes, each of in-degree >= kHotMinIndeg.
// Their residues are added up in kHotCopies copies (256 sources of a 2^20-node R-MAT graph, r_max
// of the network: 121.5 ms of push, 187.2 without the copies, as the reductions that meet in one
// sector take turns there).
constexpr int kHotSlots = 128;
constexpr uint32_t kHotMinIndeg = 64;
constexpr uint32_t kHotBit = 0x80000000u;

// Degree classes of the walk records: their table (8 bytes each) sits in shared memory of
// the walk kernel.  The 2^20-node R-MAT graph has 743 distinct degrees.
constexpr uint32_t kMaxWalkClasses = 1023;

// Walk id of a record.
__device__ __forceinline__ uint32_t walk_id(const GraphDev& g, uint32_t rec) {
  return rec & ((1u << g.wbits) - 1u);
}

// Where a node's walk ends are summed, by walk id: neighbouring ids lie 32 sums (256 bytes)
// apart.  Walk ids follow the out-degree, so the nodes where most walks end have neighbouring
// ids, and sums of theirs in one sector would queue at one L2 slice.
// end_rows = 2^(wbits - 5), end_cols = ceil(n / end_rows); a source has end_rows * end_cols
// places, fewer than n + end_rows.
__host__ __device__ __forceinline__ uint32_t end_shift(int wbits) {
  return wbits > 5 ? (uint32_t)(wbits - 5) : 0u;
}
__host__ __device__ __forceinline__ uint32_t end_cols(int64_t n, int wbits) {
  const uint32_t k = end_shift(wbits);
  return (uint32_t)(((uint64_t)n + (1ull << k) - 1) >> k);
}
__host__ __device__ __forceinline__ unsigned long long end_places(int64_t n, int wbits) {
  return (unsigned long long)end_cols(n, wbits) << end_shift(wbits);
}
__device__ __forceinline__ uint32_t end_place(const GraphDev& g, uint32_t id) {
  const uint32_t k = end_shift(g.wbits);
  return (id & ((1u << k) - 1u)) * g.ecols + (id >> k);
}

// Per-source counters kept on the device during a call.
struct SlotStats {
  unsigned long long pushes;
  unsigned long long edge_pushes;
  unsigned long long residual_nodes;
  unsigned long long walks;
  unsigned long long walk_steps;
  double rsum;
  double moved;    // sum of alpha r(v) over the pushes (balanced push: r_sum = 1 - moved)
  uint32_t rounds;
  uint32_t pad;
};

// Top-k select state of one row.
struct TopkSlot {
  unsigned long long pa;  // known bits of the key's upper 64 bits (estimate bits)
  uint32_t pb;            // known bits of the key's lower 32 bits (~id)
  uint32_t plen;          // number of leading key bits fixed so far
  uint32_t kk;            // how many keys still to take from the current bucket
  uint32_t done;
  uint32_t ncand;
  uint32_t arrived;       // blocks of the row that are through with a kernel
};

// Pointers into a call's workspace.  The push keeps its sources in groups of gw (1 or 4): value
// (slot, v) of r, res and fa is at g n gw + v w + slot % gw, with g = slot / gw and w the slots
// of the group (gw, fewer in the last group of a layout of `lay` slots).
struct BatchDev {
  int32_t nsrc;
  int lay, gw;
  int ngrp, lgrp;            // groups of nsrc and of lay slots
  double alpha;
  double walk_scale;         // C = omega / r_sum
  uint32_t alpha_threshold;  // floor(alpha * 2^32)
  uint64_t seed;
  uint2 round_key[10];       // Philox round keys of `seed` (key + i * (0x9E3779B9, 0xBB67AE85))
  int zero_hop;              // walk phase with zero-hop pruning (Section 4.1)
  int want_count;            // tally walk counts too (only a debug output reads them)
  uint32_t* walk_dest;       // non-null: k_walks stores walk g's end (a walk id) in
                             // walk_dest[g] (building a walk index) instead of tallying it
  double* r;                 // residue
  double* res;               // reserve
  // Walk ends: the sum of walk weights (2^-63 units) at [slot * ends + end_place(walk id)],
  // and, when want_count, the number of walks.
  unsigned long long* acc;
  uint32_t* wcount;
  unsigned long long ends;  // end_places of the graph
  int side_by_side;         // the sums of a group's sources lie side by side (indexed walks)
  int first_grp, end_grp;   // groups of this launch of the indexed walks
  // Frontier of group g: entry e < slot_cnt[par][g] (par: the round's parity) is a node with
  // {first edge, degree} q[g * gw * n + e] and increments fa[g * gw * n + e * w + slot % gw]; its
  // hub items, i < slot_cnt[2 + par][g], are {entry, first edge} hub[g * gw * hub_stride + i]
  // with hub_len edges each.
  uint2* q;
  double* fa;                // per frontier entry and source: (1 - alpha) r(v) / d(v)
  uint2* hub;
  uint32_t* hub_len;
  unsigned long long hub_stride;
  uint32_t* slot_cnt;        // [4][cnt_stride]: entries of parity 0, 1; hub items of parity 0, 1
  int cnt_stride;            // slots per row of slot_cnt (the workspace's capacity)
  unsigned long long* gpre;  // [ngrp + 1]: exclusive prefix of ceil(entries / 32), current
  unsigned long long* hpre;  // [ngrp + 1]: exclusive prefix of hub items, current
  uint32_t* alist;           // the groups that the next take scans whole
  uint32_t* tlist;           // units (g * tiles + t) that the next take scans of the others
  double* hotr;              // [hot_copies][lgrp][nhot][gw] copies of the hot nodes' residues
  int hot_copies;            // 0: every push goes to r
  unsigned long long* work;  // dynamic work counters of the spread ([0] and [16])
  PushState* ps;
  PushCtl* ctl;
  uint32_t* meet;            // [2][kMeetWords] meeting points of the push, by turn; zero before it
  const int32_t* sources;    // [nsrc]
  const double* rmax;        // [nsrc]
  SlotStats* stats;          // [nsrc]
  uint32_t* err;
  // walk phase
  unsigned long long* wr_entry;   // residual list: (slot << 32) | v
  unsigned long long* wr_offset;  // exclusive walk offsets, [|R| + 1]
  unsigned long long* wr_weight;  // fixed-point weight per walk        (aliases fa)
  // entries and walks of each slot's share of the nodes: counts, then offsets
  unsigned long long* unit_cnt;    // [nsrc][units]
  unsigned long long* unit_walks;  // [nsrc][units]
  int units;                       // shares of the nodes, a warp's work each
  unsigned long long* totals;     // [2]: |R|, W
  unsigned long long* walk_next;  // shares of the walk range taken beyond the first (zeroed)
  int spread_width;  // interleaved segments of the frontier the spread visits at once
  int walk_blocks;   // resident walk blocks per SM (3, 4 or 5)
  uint32_t max_rounds;  // push rounds allowed before kErrPushNotConverged
  // Balanced push (Section 4.2, Alg. 3): balance != 0 makes rmax the per-source threshold
  // theta (halved on the device when no node is above it) and stops a source's push before
  // a round once cost_edge * edge pushes + cost_push * pushes >= ((1 - moved) * bal_scale)
  // * cost_walk, with bal_scale = C' (C, or (1 - alpha) C with zero-hop pruning).
  int balance;
  double bal_scale, cost_edge, cost_push, cost_walk;
  double* theta;       // [nsrc] the thresholds (the same array as rmax)
  uint32_t* stopped;   // [nsrc] 1 once the cost rule stopped the source's push
  // Light rounds: after every take each node of an active source is at or below its
  // threshold, so only nodes the next spread adds to can cross.  When a group's new frontier
  // spreads fewer than light_edges edges, its spread marks the units of kTakeUnit residues that
  // it touches (one bit each) and lists them in tlist, and its take scans only those (clearing
  // the marks); otherwise the take scans every unit.
  uint8_t* light;                  // [ngrp] kGroupLight | kGroupActive
  uint32_t* dirty;                 // [lgrp][tiles] bits
  unsigned long long* last_edges;  // [nsrc] the source's edge pushes at the last advance
  uint32_t tiles;                  // units per group, ceil(n / (kTakeUnit / gw))
  unsigned long long light_edges;
};

// The sums of a slot's walk ends: that of place p at first + p * step.
struct EndSums {
  unsigned long long first, step;
  __device__ __forceinline__ unsigned long long at(uint32_t place) const {
    return first + (unsigned long long)place * step;
  }
};
__device__ __forceinline__ EndSums end_sums(const BatchDev& b, int slot) {
  if (!b.side_by_side) return EndSums{(unsigned long long)slot * b.ends, 1ull};
  const int gr = slot / b.gw;
  return EndSums{(unsigned long long)gr * b.gw * b.ends + (unsigned long long)(slot % b.gw),
                 (unsigned long long)min(b.gw, b.lay - gr * b.gw)};
}

// Launch-shape parameters of a graph (set through fora_graph_tune or the autotuner).
struct Tuning {
  int spread_width = 1;
  int spread_hot = 1;      // 1: pushes to hot nodes go to copies of their residues
  int walk_blocks = 4;
  int index_groups = 0;    // groups per list of the indexed walks, 0: index_list_groups
  int push_host_loop = 0;  // 1: rounds launched from a host loop instead of one launch
  int push_slice = 1000;   // microseconds after which a long push starts another launch
  int pipeline = 1;        // parts of a batch run on their own streams, pushes staggered
  uint32_t max_push_rounds = kMaxPushRounds;
};

// capi.cu: record a failure for fora_last_error() and return `code`.
int report_error(int code, const char* fmt, ...);
// capi.cu: resident blocks per SM of `kernel` launched with `threads` threads and no
// dynamic shared memory on the current device (at least 1; 0 if the query fails).
// Cached per (device, kernel) under a lock, so concurrent host threads may call it.
int resident_blocks(const void* kernel, int threads);
// capi.cu: cudaMalloc through the library's allocation hook (fora_debug_fail_alloc):
// returns cudaErrorMemoryAllocation without allocating when the hook says so.
cudaError_t device_alloc(void** p, size_t bytes);

// push.cu: the whole push in one launch (from zeroing r and res on), or a part of it.  Where the
// device has no room for all its blocks at once nothing is done, and host->go or (without host)
// kErrMissing tells.
cudaError_t launch_push(const GraphDev& g, const BatchDev& b, int num_sms, const PushPart* part,
                        cudaStream_t st);
// The same in steps for a host loop that reads PushState::go after each round: start, rounds,
// finish.  They are loaded with the first graph: loaded when first launched they would wait for
// whatever kernel is running, and it is beside such a kernel that they are needed.
cudaError_t load_push_phases();
cudaError_t launch_push_start(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st);
cudaError_t launch_push_round(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st);
cudaError_t launch_push_finish(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st);
// push.cu: a [slot][n] array from (to_rows) or into the batch's grouped layout.
cudaError_t launch_regroup(double* grouped, double* rows, const BatchDev& b, int64_t n,
                           bool to_rows, int num_sms, cudaStream_t st);
// push.cu: slots [first, first + k) join a batch between two push rounds (host loop only).
cudaError_t launch_push_join(const GraphDev& g, const BatchDev& b, int first, int k,
                             cudaStream_t st);
// push.cu: the frontier test r > RN(r_max * d) of the take, on given triples.
cudaError_t launch_threshold_table(const double* r, const double* rm, const uint32_t* d,
                                   uint8_t* out, int count, cudaStream_t st);

// walk.cu
// Residual units per slot: a multiple of a warp's nodes, at most kMaxUnits in all so that one
// block scans them, and at most what the top-k scratch of a slot holds.
int residual_units(int64_t n, int nsrc);
cudaError_t launch_residuals(const GraphDev& g, const BatchDev& b, cudaStream_t st);
cudaError_t launch_walks(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st);
// walk.cu, FORA+ (Section 3.3): r[v] = RN(rmax * d(v)) for one slot (the residues whose
// omega_v are the index's omega_max(v)), and the walk phase served from an index.
cudaError_t launch_index_residue(const GraphDev& g, double* r, double rmax, cudaStream_t st);
// Several lists of at most `groups` groups of sources each where one cannot hold them all.
cudaError_t launch_walks_indexed(const GraphDev& g, const BatchDev& b, int num_sms, int groups,
                                 const unsigned long long* idx_off, const uint32_t* idx_dest,
                                 cudaStream_t st);
// The walk ends of a batch as [nsrc][n] arrays over node ids (either output may be null).
cudaError_t launch_unpack_ends(const GraphDev& g, const BatchDev& b, uint32_t* cnt,
                               unsigned long long* acc, int num_sms, cudaStream_t st);
// wcol of a graph whose other walk arrays are in place.
cudaError_t launch_walk_records(const GraphDev& g, uint32_t* wcol, int num_sms, cudaStream_t st);
cudaError_t launch_philox_table(const uint32_t* ctr_key, uint32_t* out, int count,
                                cudaStream_t st);

// learn.cu
cudaError_t launch_indegree(const GraphDev& g, uint32_t* indeg, int num_sms, cudaStream_t st);
cudaError_t launch_features(const GraphDev& g, const uint32_t* indeg, const int32_t* sources,
                            int nsrc, double alpha, double rmax_rule, float* out, cudaStream_t st);
cudaError_t launch_mlp_forward(const float* master, const float* norm, const float* X, int n,
                               float* Y, cudaStream_t st);
cudaError_t launch_mlp_grad(const float* master, const float* norm, const float* X,
                            const float* T, const int32_t* idx, int n, float* partial,
                            float* loss_partial, float* grad, cudaStream_t st);
float2 adam_correction(int step);
bool mlp_train_fits(int batch);
cudaError_t launch_mlp_epoch(float* master, float* m, float* v, const float* norm, const float* X,
                             const float* T, const int32_t* idx, const float2* corrections, int n,
                             int batch, float lr, float* loss, cudaStream_t st);
size_t mlp_partial_floats(int n);
cudaError_t launch_adam(float* master, float* m, float* v, const float* grad, int step, float lr,
                        cudaStream_t st);
cudaError_t launch_pred_to_rmax(const float* pred, int n, double rmax_rule, float lo, float hi,
                                double* rmax, cudaStream_t st);


// topk.cu
// est [nsrc][n]; with zero-hop pruning the estimate also takes alpha * r.
cudaError_t launch_estimate(const GraphDev& g, const BatchDev& b, double* est, cudaStream_t st);
// Scratch of the top-k select: hist [nrows][kBins], slots [nrows], cand [nrows][kSortCap].
struct TopkScratch {
  uint32_t* hist;
  TopkSlot* slots;
  unsigned long long* cand_key;  // estimate bits
  uint32_t* cand_id;
};
size_t topk_scratch_bytes(int nrows);
TopkScratch topk_scratch_carve(void* base, int nrows);
cudaError_t launch_topk(const double* est, int64_t n, int nrows, uint32_t k, int32_t* out_ids,
                        double* out_vals, const TopkScratch& s, int num_sms, cudaStream_t st);

}  // namespace fora
