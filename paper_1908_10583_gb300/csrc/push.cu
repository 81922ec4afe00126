// Forward Push (Alg. 1) as synchronous frontier rounds over a batch of sources.
//
// Sources are kept in groups of G (1 or 4): the residues, reserves and increments of a group's
// sources at one node lie side by side (r[group][node][source]), so the take reads a node's
// degree once per group and the spread adds to the G sources of a target in one 32-byte
// sector.  (The L2 takes 2.0e11 scattered FP64 reductions a second, and 5.1e11 where four fill
// a sector; after the first rounds the sources of a batch push from much the same nodes: four
// sources of the 2^20-node R-MAT graph share 74% of their frontier edges at 0.35 of the rule's
// r_max, 38% at the rule's.)
//
// F_t holds, per group, the nodes v that some source of the group takes in round t, i.e. with
// r(v) > r_max * d(v) at its start, and per source the increment inc_v = (1 - alpha) a_v / d(v)
// of its taken residue a_v (0: the source does not take v).  Round t:
//   spread   r(u) += inc_v for every out-edge (v, u) of F_t: FP64 reductions that return
//            nothing, so a warp never waits on an atomic.
//   take     F_{t+1} = {u : r(u) > r_max * d(u)} over the groups that pushed in round t (every
//            other r is unchanged and below its threshold), in one pass over their residues;
//            each crossing node is appended to its group's queue and taken at once:
//            a_u = r(u); reserve(u) += alpha a_u; r(u) = 0;
//            inc_u = (1 - alpha) a_u / d(u)   (the first half of round t+1), computed as
//            RN(RN((1 - alpha) a_u) * RN(1 / d(u))) with the graph's reciprocal degrees (within
//            an ulp or so of the quotient; this GPU's FP64 division costs about ten FP64
//            instructions).
//   advance  one block: per-group prefix of the new frontier's items, the groups still
//            pushing, the loop condition.
// The take of round t+1 happens after every add of round t, so residue arriving at a frontier
// node during a round waits for the next round.
//
// k_push runs the rounds in one launch: its blocks meet after each phase, and the first of them
// runs the advance while the others wait at the take's.  (As three launches in a conditional graph
// node a round cost 39 us however small; 22 rounds of a 2^14-node graph took 0.89 ms, now 0.39.)
// A launch does its work only if all its blocks run at once: each enters as it starts, and when
// some have not come after a tenth of a millisecond (other kernels hold their places) those that
// have leave, and the host runs a round as kernels of its own, the phases one by one, which need no
// places held, before it tries again.  So no block waits for one that has not started, and nothing
// else on the device can hold a push back.  (Working on with the blocks that were there, and
// admitting the others round by round, let lanes of a server block each other: a round begun by a
// few blocks took 600 times as long, its late blocks holding the SMs meanwhile.)  So that a push
// does not hold back others either, a long one is a sequence of launches of about a millisecond,
// between which kernels of other streams start (a single query beside batches of 256 sources of
// 2^20 nodes waited for the whole push of one).  A serving batch that requests join ends its launch
// after a round and resumes.  The phases are launched one by one by push_host_loop too.
//
// Pushes to the graph's hot nodes (the up to 128 nodes of highest in-degree) would queue at the
// L2 slices that hold their residues: each block adds them to one of kHotCopies copies, and the
// take adds the copies to the residue before it reads it.
//
// Bounds: the spread by the reductions' rate at L2 (heavy rounds run at 2.4e11 to 2.7e11 pushes
// a second, 1.2e11 sectors, of the 1.27e11 sectors that four neighbouring FP64 reductions each
// reached in isolation), the take by the pass over the residues, light rounds by the latency of
// a few dependent L2 accesses and two barriers (about 17 us).  Measured against one reduction per
// push and source (with hot pushes summed in shared memory, and the rounds in a graph): 256
// sources of a 2^20-node R-MAT graph, r_max of the network, 185 -> 121.5 ms of push; 64 of 2^18
// 7.5 -> 6.9; 100 of a 200003-node graph without hubs 8.9 -> 6.3; one of 2^20 1.86 -> 1.45.
#include "fora_engine.cuh"

namespace fora {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kPushThreads = 256;
constexpr int kPushWarps = kPushThreads / 32;
constexpr uint32_t kSpan = 32;  // most entries of an item of the spread
constexpr int kUnit = kTakeUnit;  // residues a warp of the take reads at a time

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const T t = __shfl_up_sync(kFull, x, off);
    if ((int)lane_id() >= off) x += t;
  }
  return x;
}

// Block-wide exclusive scan of two counters; returns the block totals too.
__device__ __forceinline__ void block_scan2(unsigned long long a, unsigned long long b,
                                            unsigned long long* ae, unsigned long long* be,
                                            unsigned long long* at, unsigned long long* bt) {
  __shared__ unsigned long long sa[32], sb[32];
  __shared__ unsigned long long ta, tb;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned long long ai = warp_incl_scan(a), bi = warp_incl_scan(b);
  if (lane == 31) { sa[wid] = ai; sb[wid] = bi; }
  __syncthreads();
  if (wid == 0) {
    const unsigned long long x = lane < nw ? sa[lane] : 0, y = lane < nw ? sb[lane] : 0;
    const unsigned long long xi = warp_incl_scan(x), yi = warp_incl_scan(y);
    if (lane < nw) { sa[lane] = xi - x; sb[lane] = yi - y; }
    if (lane == 31) { ta = xi; tb = yi; }
  }
  __syncthreads();
  *ae = sa[wid] + ai - a;
  *be = sb[wid] + bi - b;
  *at = ta;
  *bt = tb;
  __syncthreads();
}

__device__ __forceinline__ uint32_t hub_chunks_of(uint32_t d) {
  return d > kHubChunk ? (d + kHubChunk - 1) / kHubChunk : 0u;
}

// r > RN(rm * d), the frontier test, without FP64 arithmetic but near the threshold (this GPU
// issues about two FP64 operations per clock per SM, so the test itself would bound the scan).
// tf = RN32(rmf * RN32(d)) with rmf = RN32(rm) is within 2^-22 of V = rm * d, and T = RN64(V) is
// within 2^-53 of V.  The upper word of an FP64 value (exponent and 20 mantissa bits) is
// floor(bits / 2^32), that of tf is (bits of tf >> 3) + 0x38000000, and a relative change of
// 2^-21 moves it by at most 1; so r's word below tf's word - 1 implies r < T, and above tf's
// word + 1 implies r > T.  Valid for rmf in [2^-100, 2^60] (`fast`), where tf is a normal
// number; r may be anything (r >= 0: its words order as its values).  Returns 0 (below), 1
// (above) or 2 (undecided); the FP64 test decides the undecided ones.
__device__ __forceinline__ uint32_t threshold_word(float rmf, float d) {
  return (__float_as_uint(rmf * d) >> 3) + 0x38000000u;
}
__device__ __forceinline__ uint32_t threshold_fast(double r, float rmf, bool fast, float d) {
  const uint32_t hi = (uint32_t)((unsigned long long)__double_as_longlong(r) >> 32);
  const uint32_t t = threshold_word(rmf, d);
  return !fast ? 2u : hi < t - 1u ? 0u : hi > t + 1u ? 1u : 2u;
}

// The FP64 test, kept out of line so that it is not evaluated for every node.
__device__ __noinline__ bool threshold_exact(double r, double rm, uint32_t d) {
  return r > __dmul_rn(rm, (double)d);
}

__device__ __forceinline__ bool above_threshold(double r, double rm, float rmf, bool fast,
                                                uint32_t d) {
  const uint32_t f = threshold_fast(r, rmf, fast, __uint2float_rn(d));
  return f == 2u ? threshold_exact(r, rm, d) : f == 1u;
}

// The group whose range [pre[s], pre[s + 1]) holds x, for a non-decreasing prefix with
// x < pre[count]: the largest s with pre[s] <= x (empty ones have pre[s] = pre[s + 1]).
__device__ __forceinline__ int group_of(const unsigned long long* pre, int count,
                                        unsigned long long x) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Sources of group gr side by side in the layout: G, fewer in the last group.
template <int G>
__device__ __forceinline__ uint32_t width_of(const BatchDev& b, uint32_t gr) {
  return min((uint32_t)G, (uint32_t)b.lay - gr * G);
}

// Marks the unit of node u of a group for its next take, listing it once.
template <int G>
__device__ __forceinline__ void mark_unit(const BatchDev& b, uint32_t gr, uint32_t u) {
  const unsigned long long t = (unsigned long long)gr * b.tiles + u / (kUnit / G);
  uint32_t* word = b.dirty + (t >> 5);
  const uint32_t bit = 1u << (t & 31);
  if (*(volatile uint32_t*)word & bit) return;
  if (!(atomicOr(word, bit) & bit)) b.tlist[atomicAdd(&b.ctl->nlist, 1u)] = (uint32_t)t;
}

// Before the first round: r(s) = 1 for every source (Alg. 1), every group in the first take,
// which scans the sources' units alone.  Called by the threads of one block.
template <int G>
__device__ void seed_phase(const GraphDev& g, const BatchDev& b) {
  for (int slot = threadIdx.x; slot < b.nsrc; slot += blockDim.x) {
    const uint32_t src = (uint32_t)b.sources[slot], gr = (uint32_t)slot / G;
    b.r[(unsigned long long)gr * G * (unsigned long long)g.n +
        (unsigned long long)src * width_of<G>(b, gr) + slot % G] = 1.0;
    mark_unit<G>(b, gr, src);
    if (slot % G == 0) {
      b.alist[gr] = gr;
      b.light[gr] = kGroupLight | kGroupActive;
    }
    if (b.balance) {
      // the cost rule before any push: FC = 0 against the walk cost of r_sum = 1
      const bool stop = 0.0 >= __dmul_rn(__dmul_rn(1.0, b.bal_scale), b.cost_walk);
      b.stopped[slot] = stop ? 1u : 0u;
      // Alg. 3 starts from threshold 1 and halves it while no node is above it: before the
      // first push only r(s) = 1 is non-zero, so theta halves until 1 > theta d(s)
      double theta = 1.0;
      const double ds = (double)(g.row[src + 1] - g.row[src]);
      if (!stop)
        while (!(1.0 > __dmul_rn(theta, ds))) theta = __dmul_rn(0.5, theta);
      b.theta[slot] = theta;
    }
  }
  if (threadIdx.x == 0) {
    PushState* ps = b.ps;
    ps->cur = 1;
    ps->round = 0;
    ps->go = 1;
    ps->ngroups = 0;
    ps->nhub = 0;
    b.ctl->span = kSpan;
  }
}

// ---------------------------------------------------------------- spread

// Where the pushes of one group go: its residues, and this block's copies of its hot nodes'.
template <int G>
struct SpreadTarget {
  double* r;
  double* hot;  // null: no copies (then no code has kHotBit)
  uint32_t w;
};

template <int G>
__device__ __forceinline__ SpreadTarget<G> spread_target(const GraphDev& g, const BatchDev& b,
                                                         uint32_t gr) {
  SpreadTarget<G> t;
  t.w = width_of<G>(b, gr);
  t.r = b.r + (unsigned long long)gr * G * (unsigned long long)g.n;
  t.hot = b.hot_copies ? b.hotr + ((unsigned long long)(blockIdx.x % b.hot_copies) * b.lgrp + gr) *
                                      (unsigned long long)(g.nhot * G)
                       : nullptr;
  return t;
}

// *p += x with nothing returned, in global memory for certain (where the compiler cannot tell the
// address space of p, an FP64 atomicAdd becomes a loop).
__device__ __forceinline__ void red_add(double* p, double x) {
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "d"(x)
               : "memory");
}

constexpr uint32_t kNoEdge = 0xFFFFFFFFu;

// r(u) += inc for source j of the group and the target of a code.
template <int G>
__device__ __forceinline__ void add_to(const GraphDev& g, const BatchDev& b,
                                       const SpreadTarget<G>& t, uint32_t code, uint32_t j,
                                       double inc) {
  if (code & kHotBit) {
    const uint32_t h = code & ~kHotBit;
    if (FORA_IN_RANGE(b.err, h, (uint32_t)g.nhot)) red_add(t.hot + (h * G + j), inc);
  } else if (FORA_IN_RANGE(b.err, code, g.n)) {
    red_add(t.r + ((unsigned long long)code * t.w + j), inc);
  }
}

// x is not zero, for x >= 0 (never -0), without the FP64 pipe: at its rate the comparison alone
// bounds a kernel that makes it for every value.
__device__ __forceinline__ bool nonzero(double x) { return __double_as_longlong(x) != 0; }

// 0, 1, ..., 32 as FP64: lengths of runs.
__constant__ double kRunLength[33] = {0,  1,  2,  3,  4,  5,  6,  7,  8,  9,  10,
                                      11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 21,
                                      22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32};

// 32 consecutive edges of one source: rows are sorted, so the copies of a multi-edge lie in
// neighbouring lanes, and their increments are added at once, k copies as k * inc by the first
// (one rounding instead of k, which reorders the FP64 sum as the reductions do).
// Only for large batches without groups: the balanced push of 256 sources of a 2^20-node R-MAT
// graph, 4% of whose edges are copies (more of what hubs push), 295.6 -> 276.9 ms; a graph whose
// edges all have 16 copies, 32 sources of 2^18 nodes, 14.2 -> 11.7.  In the small launches the
// shuffles cost more than they save (one of 2^14 nodes 0.44 -> 0.46), and groups of four, whose
// lanes of one edge lie side by side, are no slower without (64 sources, 16 copies: 6.1 ms, 6.1
// where each copy of a source was merged).
__device__ __forceinline__ void spread_runs(const GraphDev& g, const BatchDev& b,
                                            const SpreadTarget<1>& t, uint32_t code,
                                            uint32_t place, double inc) {
  const uint32_t lane = lane_id();
  const uint32_t code0 = __shfl_up_sync(kFull, code, 1), place0 = __shfl_up_sync(kFull, place, 1);
  const bool goes_on = lane > 0 && code0 == code && place0 == place;
  const uint32_t starts = __ballot_sync(kFull, !goes_on);
  if (goes_on || code == kNoEdge || !nonzero(inc)) return;
  const uint32_t later = starts & ~((2u << lane) - 1u);
  const uint32_t k = (later ? (uint32_t)__ffs(later) - 1u : 32u) - lane;
  add_to<1>(g, b, t, code, 0u, k > 1u ? __dmul_rn(inc, kRunLength[k]) : inc);
}

// The adds of 32 edges (each lane's target code and the place of its entry's increments in
// inc[place][G]) for the G sources of the group, lanes of one edge side by side.
template <int G, bool kRuns>
__device__ __forceinline__ void spread_slice(const GraphDev& g, const BatchDev& b,
                                             const SpreadTarget<G>& t, uint32_t code,
                                             uint32_t place, const double* inc) {
  const uint32_t lane = lane_id(), j = lane % G;
  if constexpr (kRuns) {
    spread_runs(g, b, t, code, place, inc[place]);
  } else {
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const int from = k * (32 / G) + (int)(lane / G);
      const uint32_t c = G == 1 ? code : __shfl_sync(kFull, code, from);
      const uint32_t p = G == 1 ? place : __shfl_sync(kFull, place, from);
      const double a = inc[p * G + j];
      if (c != kNoEdge && nonzero(a)) add_to<G>(g, b, t, c, j, a);
    }
  }
}

template <int G>
__device__ __forceinline__ void spread_marks(const GraphDev& g, const BatchDev& b, uint32_t gr,
                                             uint32_t code) {
  if (code == kNoEdge) return;
  const uint32_t u = (code & kHotBit) ? g.hot_node[code & ~kHotBit] : code;
  if (u < (uint32_t)g.n) mark_unit<G>(b, gr, u);
}

// A warp's increments of the 32 entries of an item, and of the next item.
template <int G>
struct SpreadStage {
  double inc[2][32 * G];
};

__device__ __forceinline__ void copy_async8(void* to, const void* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(to)),
               "l"(from)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// An item of the spread: the entries from `first` on of group gr.
struct SpreadItem {
  uint32_t gr, first, have;
};

// Starts the loads of an item: its entries' {first edge, degree}, one per lane (returned; of a
// node with more than kHubChunk edges the degree is 0), and their increments into inc.
template <int G>
__device__ __forceinline__ uint2 fetch_item(const GraphDev& g, const BatchDev& b,
                                            const SpreadItem& it, double* inc) {
  const uint32_t lane = lane_id(), w = width_of<G>(b, it.gr);
  const unsigned long long g0 = (unsigned long long)it.gr * G * (unsigned long long)g.n;
  uint2 e = make_uint2(0u, 0u);
  if (lane < it.have) {
    e = __ldcg(&b.q[g0 + it.first + lane]);
    if (e.y > kHubChunk) e.y = 0;
  }
  const double* fa = b.fa + g0 + (unsigned long long)it.first * w;
  if (w == (uint32_t)G) {
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const uint32_t x = k * 32 + lane;
      if (x < it.have * G) copy_async8(inc + x, fa + x);
    }
  } else {
    for (uint32_t x = lane; x < it.have * G; x += 32) {
      if (x % G < w) copy_async8(inc + x, fa + x / G * w + x % G);
      else inc[x] = 0.0;
    }
  }
  return e;
}

// The edge lists of an item's entries, walked one after the other, 128 edges per iteration with
// the next 128 targets on their way.
template <int G, bool kRuns>
__device__ __forceinline__ void spread_item(const GraphDev& g, const BatchDev& b,
                                            const uint32_t* codes, uint32_t gr, bool light,
                                            uint2 entry, const double* inc) {
  const uint32_t lane = lane_id();
  const SpreadTarget<G> t = spread_target<G>(g, b, gr);
  const uint32_t incl = warp_incl_scan(entry.y);
  const uint32_t total = __shfl_sync(kFull, incl, 31);
  const uint32_t off = entry.x - (incl - entry.y);  // first edge minus the item's edges before
  constexpr int kSlices = 4;
  uint32_t code[kSlices], own = 0;  // own: 5 bits per slice
  auto fetch = [&](uint32_t base, uint32_t* c, uint32_t* o) {
    uint32_t packed = 0;
#pragma unroll
    for (int k = 0; k < kSlices; ++k) {
      const uint32_t e = base + 32 * k + lane;
      int lo = 0, hi = 31;  // owner: the first lane whose inclusive prefix exceeds e
#pragma unroll
      for (int s2 = 0; s2 < 5; ++s2) {
        const int mid = (lo + hi) >> 1;
        if (__shfl_sync(kFull, incl, mid) > e) hi = mid; else lo = mid + 1;
      }
      const uint32_t at = __shfl_sync(kFull, off, lo) + e;
      packed |= (uint32_t)(lo & 31) << (5 * k);
      c[k] = e < total ? __ldg(codes + at) : kNoEdge;
    }
    *o = packed;
  };
  if (total) fetch(0, code, &own);
  for (uint32_t base = 0; base < total; base += 32 * kSlices) {
    uint32_t next[kSlices], next_own = 0;
#pragma unroll
    for (int k = 0; k < kSlices; ++k) next[k] = kNoEdge;
    if (base + 32 * kSlices < total) fetch(base + 32 * kSlices, next, &next_own);
#pragma unroll
    for (int k = 0; k < kSlices; ++k)
      if (base + 32 * k < total) spread_slice<G, kRuns>(g, b, t, code[k], (own >> (5 * k)) & 31u, inc);
    if (light) {  // warp-uniform
#pragma unroll
      for (int k = 0; k < kSlices; ++k) spread_marks<G>(g, b, gr, code[k]);
    }
#pragma unroll
    for (int k = 0; k < kSlices; ++k) code[k] = next[k];
    own = next_own;
  }
}

// A hub item: up to kHubChunk consecutive out-edges of one frontier entry.
template <int G, bool kRuns>
__device__ __forceinline__ void spread_hub(const GraphDev& g, const BatchDev& b,
                                           const uint32_t* codes, uint32_t gr, bool light,
                                           uint2 rec, uint32_t len, double* inc) {
  const uint32_t lane = lane_id();
  const SpreadTarget<G> t = spread_target<G>(g, b, gr);
  const unsigned long long g0 = (unsigned long long)gr * G * (unsigned long long)g.n;
  uint32_t code[kHubChunk / 32];
#pragma unroll
  for (int k = 0; k < (int)(kHubChunk / 32); ++k) {
    const uint32_t p = 32 * k + lane;
    code[k] = p < len ? __ldg(codes + rec.y + p) : kNoEdge;
  }
  const uint32_t j = lane % G;
  const double a = j < t.w ? __ldcg(b.fa + g0 + (unsigned long long)rec.x * t.w + j) : 0.0;
  __syncwarp();  // inc free
  if (lane < (uint32_t)G) inc[lane] = a;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < (int)(kHubChunk / 32); ++k)
    if (32u * k < len) spread_slice<G, kRuns>(g, b, t, code[k], 0u, inc);
  if (light) {  // warp-uniform
#pragma unroll
    for (int k = 0; k < (int)(kHubChunk / 32); ++k) spread_marks<G>(g, b, gr, code[k]);
  }
}

// A block's share of a list of items: its warps take them one by one from shared memory, and one
// global atomic brings the next kChunk.  The items in flight are then a narrow window of the
// list, so the residues that they add into stay in L2, at an atomic per kChunk items (a counter
// that every warp used bounded the spread: 256 sources of a 2^20-node R-MAT graph took 224, 166
// and 127 ms of push with 1, 2 and 4 items an atomic, and 151 and 183 with 16 and 32, whose
// window no longer fits; this takes 121.5, and 121.8 and 123.1 with chunks of 16 and 32).
constexpr uint32_t kChunk = 8;
struct ItemShare {
  unsigned long long state;  // first item of the chunk << 8 | items taken of it
  unsigned long long next;   // the next chunk's number + 1, 0: not known yet
};

struct ItemCursor {
  unsigned long long items, total, seg, width;
  const unsigned long long* pre;
  unsigned long long* counter;
  ItemShare* share;
  bool few, done;  // at most one item per warp
  uint32_t gr;
  unsigned long long lo, hi;  // the items of group gr
  bool light;
  uint32_t cnt;

  __device__ __forceinline__ void attach(const BatchDev& b, unsigned long long items_,
                                         const unsigned long long* pre_, unsigned long long* ctr,
                                         ItemShare* share_) {
    items = items_;
    width = (unsigned long long)b.spread_width;
    seg = width == 1 ? items : (items + width - 1) / width;
    total = seg * width;
    pre = pre_;
    counter = ctr;
    share = share_;
    few = total <= (unsigned long long)gridDim.x * kPushWarps;
    done = false;
    gr = 0;
    lo = 1;
    hi = 0;
    light = false;
    cnt = 0;
  }
  // A place in the list, `total` or more when there is none left.  Lane 0.
  __device__ __forceinline__ unsigned long long pop(uint32_t* err) {
    for (uint32_t tries = 0; tries < kMaxPolls; ++tries) {
      const unsigned long long old = atomicAdd(&share->state, 1ull);
      const uint32_t k = (uint32_t)(old & 255u);
      const unsigned long long x = (old >> 8) + k;
      if (x >= total) return x;
      if (k < kChunk) {
        if (k == kChunk / 2)  // ask for the next chunk in good time
          *(volatile unsigned long long*)&share->next = atomicAdd(counter, 1ull) + 1ull;
        return x;
      }
      if (k == kChunk) {  // this warp opens the next chunk
        unsigned long long n = 0;
        for (uint32_t polls = 0; polls < kMaxPolls && n == 0; ++polls)
          n = *(volatile unsigned long long*)&share->next;
        if (n == 0) break;
        *(volatile unsigned long long*)&share->next = 0;
        const unsigned long long first = ((unsigned long long)gridDim.x + n - 1ull) * kChunk;
        atomicExch(&share->state, first << 8 | 1ull);
        return first;
      }
      for (uint32_t polls = 0; polls < kMaxPolls; ++polls)
        if ((*(volatile unsigned long long*)&share->state & 255u) <= kChunk) break;
    }
    atomicOr(err, kErrBarrier);
    return ~0ull;
  }
  // The next item's place in the list, or false.
  __device__ __forceinline__ bool step(uint32_t* err, unsigned long long* it) {
    for (;;) {
      unsigned long long x = 0;
      if (few) {
        if (done) return false;
        x = (unsigned long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
        done = true;
      } else {
        if (lane_id() == 0) x = pop(err);
        x = __shfl_sync(kFull, x, 0);
      }
      if (x >= total) return false;
      *it = width == 1 ? x : (x % width) * seg + x / width;
      if (*it < items) return true;
    }
  }
  // Makes gr the group of item `it`, with its light flag and (for parity cur) entry count.
  __device__ __forceinline__ void locate(const BatchDev& b, unsigned long long it, int cur) {
    if (it >= lo && it < hi) return;  // warp-uniform
    if (b.ngrp == 1) {
      lo = 0;
      hi = items;
    } else {
      gr = (uint32_t)group_of(pre, b.ngrp, it);
      lo = pre[gr];
      hi = pre[gr + 1];
    }
    light = (__ldcg(&b.light[gr]) & kGroupLight) != 0;
    cnt = __ldcg(&b.slot_cnt[(size_t)cur * b.cnt_stride + gr]);
  }
};

template <int G, bool kRuns>
__device__ void spread_phase(const GraphDev& g, const BatchDev& b, int cur,
                             unsigned long long nhub, unsigned long long nitems, uint32_t span,
                             SpreadStage<G>& st) {
  const uint32_t* codes = b.hot_copies ? g.scol : (const uint32_t*)g.col;
  __shared__ ItemShare shares[2];
  ItemCursor c;
  unsigned long long it;
  if (threadIdx.x < 2) {
    shares[threadIdx.x].state = (unsigned long long)blockIdx.x * kChunk << 8;
    shares[threadIdx.x].next = 0;
  }
  __syncthreads();
  if (nhub) {
    c.attach(b, nhub, b.hpre, &b.work[16], &shares[0]);
    auto fetch = [&](uint2* rec, uint32_t* len) {
      c.locate(b, it, cur);
      const unsigned long long at =
          (unsigned long long)c.gr * G * b.hub_stride + (it - c.lo);
      *rec = __ldcg(&b.hub[at]);
      *len = __ldcg(&b.hub_len[at]);
    };
    bool more = c.step(b.err, &it);
    uint2 rec = make_uint2(0u, 0u);
    uint32_t len = 0;
    if (more) fetch(&rec, &len);
    while (more) {
      const uint32_t gr = c.gr;
      const bool light = c.light;
      const uint2 r = rec;
      const uint32_t l = len;
      more = c.step(b.err, &it);
      if (more) fetch(&rec, &len);
      spread_hub<G, kRuns>(g, b, codes, gr, light, r, l, st.inc[0]);
    }
    __syncwarp();
  }
  if (nitems) {
    c.attach(b, nitems, b.gpre, &b.work[0], &shares[1]);
    auto locate = [&](SpreadItem* x) {
      c.locate(b, it, cur);
      x->gr = c.gr;
      x->first = (uint32_t)(it - c.lo) * span;
      x->have = min(span, c.cnt - x->first);
    };
    SpreadItem x;
    uint2 entry = make_uint2(0u, 0u);
    int half = 0;
    bool more = c.step(b.err, &it);
    if (more) {
      locate(&x);
      entry = fetch_item<G>(g, b, x, st.inc[0]);
    }
    while (more) {
      copy_async_wait();
      __syncwarp();  // this item's increments are in place, the other half is free
      const uint32_t gr = x.gr;
      const bool light = c.light;
      const uint2 now = entry;
      more = c.step(b.err, &it);
      if (more) {
        locate(&x);
        entry = fetch_item<G>(g, b, x, st.inc[half ^ 1]);
      }
      spread_item<G, kRuns>(g, b, codes, gr, light, now, st.inc[half]);
      half ^= 1;
    }
  }
}

// ---------------------------------------------------------------- take

// Adds the copies of hot node h's residues in group gr to them and clears the copies.  A warp.
template <int G>
__device__ __noinline__ void fold_hot(const GraphDev& g, const BatchDev& b, uint32_t gr,
                                      uint32_t h) {
  const uint32_t lane = lane_id(), j = lane % G, w = width_of<G>(b, gr);
  double sum = 0.0;
  for (uint32_t c = lane / G; c < (uint32_t)b.hot_copies; c += 32 / G) {
    double* p = b.hotr + ((unsigned long long)c * b.lgrp + gr) * (unsigned long long)(g.nhot * G) +
                (h * G + j);
    const double x = __ldcg(p);
    if (nonzero(x)) {
      sum = __dadd_rn(sum, x);
      *p = 0.0;
    }
  }
  if (!__any_sync(kFull, nonzero(sum))) return;
#pragma unroll
  for (int o = 16; o >= G; o >>= 1) sum = __dadd_rn(sum, __shfl_xor_sync(kFull, sum, o));
  if (lane < w && nonzero(sum)) {
    double* p = b.r + (unsigned long long)gr * G * (unsigned long long)g.n +
                (unsigned long long)g.hot_node[h] * w + lane;
    *p = __dadd_rn(__ldcg(p), sum);
  }
  __syncwarp();
}

// A warp's stage of crossing nodes of one group: those of one unit, and up to kCarry of the
// units before (where few nodes cross, the take of a stage serves many units).
constexpr uint32_t kCarry = 32;
template <int G>
struct TakeStage {
  static constexpr uint32_t kCap = kUnit / G + kCarry;
  double a[kCap * G];      // [entry][G] the taken residues (0: not taken), then the increments
  uint32_t u[kCap];        // [entry] node
  uint32_t d[kCap];        // [entry] out-degree
  uint32_t rb[kCap];       // [entry] first edge
  uint16_t pair[kCap * G];  // the places in `a` of the taken residues
};

// Counters of one group that a warp has not added to the batch's yet: of the source lane % G.
struct TakeCount {
  uint32_t gr = 0xFFFFFFFFu;
  uint32_t cnt = 0;
  unsigned long long deg = 0;
  double moved = 0.0;  // sum of alpha a (balanced push)
};

// Sums a warp's counters over the lanes of each source.
template <int G>
__device__ __forceinline__ void sum_count(const BatchDev& b, TakeCount& t) {
#pragma unroll
  for (int o = 16; o >= G; o >>= 1) {
    t.cnt += __shfl_xor_sync(kFull, t.cnt, o);
    t.deg += __shfl_xor_sync(kFull, t.deg, o);
    if (b.balance) t.moved = __dadd_rn(t.moved, __shfl_xor_sync(kFull, t.moved, o));
  }
}

__device__ __forceinline__ void add_count(const BatchDev& b, uint32_t slot, uint32_t cnt,
                                          unsigned long long deg, double moved) {
  if (cnt == 0) return;
  SlotStats& s = b.stats[slot];
  atomicAdd(&s.pushes, (unsigned long long)cnt);
  atomicAdd(&s.edge_pushes, deg);
  if (b.balance) red_add(&s.moved, moved);
}

// What a warp of the take knows of the group it is at.
struct TakeGroup {
  uint32_t gr = 0xFFFFFFFFu;
  uint32_t w = 0;
  float rmf = 0.0f;             // this lane's source: RN32(r_max)
  uint32_t mask = 0;            // ~0 where the frontier test's fast form holds for it
  bool live = false;
  uint32_t mine = 0, pairs = 0;  // entries and taken residues in the stage
};

// Takes the stage: one atomic per counter reserves the entries' places in the group's queue, and
// the FP64 arithmetic runs on packed lanes.
template <int G>
__device__ __noinline__ void take_stage(const GraphDev& g, const BatchDev& b, int nx,
                                        uint32_t gr, uint32_t w, uint32_t mine, uint32_t pairs,
                                        TakeStage<G>& st, TakeCount& tc) {
  const uint32_t lane = lane_id(), j = lane % G;
  const double alpha = b.alpha, beta = __dadd_rn(1.0, -b.alpha);
  const unsigned long long g0 = (unsigned long long)gr * G * (unsigned long long)g.n;
  __syncwarp();
  // the entries' degrees; their chunks of kHubChunk edges (of distinct nodes of one group: at
  // most the graph's); places in the queue
  uint32_t hubs = 0;
  for (uint32_t e = lane; e < mine; e += 32) {
    const uint32_t u = st.u[e], rb = __ldg(g.row + u), d = __ldg(g.row + u + 1) - rb;
    st.rb[e] = rb;
    st.d[e] = d;
    hubs += hub_chunks_of(d);
  }
  const uint32_t hsum = __reduce_add_sync(kFull, hubs);
  uint32_t qb = 0, hb = 0;
  if (lane == 0) {
    qb = atomicAdd(&b.slot_cnt[(size_t)nx * b.cnt_stride + gr], mine);
    if (hsum) hb = atomicAdd(&b.slot_cnt[(size_t)(2 + nx) * b.cnt_stride + gr], hsum);
  }
  __syncwarp();
  if (b.balance) {
    for (uint32_t x = lane; x < mine * G; x += 32)
      tc.moved = __dadd_rn(tc.moved, __dmul_rn(alpha, st.a[x]));
    __syncwarp();
  }
  // the take of every taken residue: reserve += alpha a, r = 0, spread increment
  for (uint32_t i = lane; i < pairs; i += 32) {
    const uint32_t p = st.pair[i], u = st.u[p / G];
    const unsigned long long at = g0 + (unsigned long long)u * w + p % G;
    const double a = st.a[p];
    const double rs = __ldcg(b.res + at), inv = __ldg(g.invd + u);
    b.r[at] = 0.0;
    b.res[at] = __fma_rn(alpha, a, rs);
    st.a[p] = __dmul_rn(__dmul_rn(beta, a), inv);  // (1 - alpha) a / d
  }
  qb = __shfl_sync(kFull, qb, 0);
  hb = __shfl_sync(kFull, hb, 0);
  __syncwarp();
  for (uint32_t x = lane; x < mine * G; x += 32) {  // increments, and the sources' counters
    const uint32_t e = x / G;
    const double inc = st.a[x];
    if (nonzero(inc)) {
      ++tc.cnt;
      tc.deg += st.d[e];
    }
    if (j < w && FORA_IN_RANGE(b.err, qb + e, g.n))
      b.fa[g0 + (unsigned long long)(qb + e) * w + j] = inc;
  }
  const unsigned long long h0 = (unsigned long long)gr * G * b.hub_stride;
  for (uint32_t e0 = 0; e0 < mine; e0 += 32) {
    const uint32_t e = e0 + lane;
    uint32_t rb = 0, d = 0;
    if (e < mine) {
      rb = st.rb[e];
      d = st.d[e];
      if (FORA_IN_RANGE(b.err, qb + e, g.n)) b.q[g0 + qb + e] = make_uint2(rb, d);
    }
    if (hsum) {  // warp-uniform
      const uint32_t nch = hub_chunks_of(d);
      const uint32_t incl = warp_incl_scan(nch);  // lower entries first
      const uint32_t at = hb + incl - nch;
      if (nch && FORA_IN_RANGE(b.err, hb + incl, (unsigned long long)w * b.hub_stride + 1)) {
        for (uint32_t c = 0; c < nch; ++c) {
          b.hub[h0 + at + c] = make_uint2(qb + e, rb + c * kHubChunk);
          b.hub_len[h0 + at + c] = min(kHubChunk, d - c * kHubChunk);
        }
      }
      hb += __shfl_sync(kFull, incl, 31);
    }
  }
  __syncwarp();
}

// Makes gr the warp's group: takes what is staged of the one before and adds its counters.
template <int G>
__device__ __forceinline__ void take_enter(const GraphDev& g, const BatchDev& b, int nx,
                                           uint32_t gr, TakeStage<G>& st, TakeGroup& tg,
                                           TakeCount& tc) {
  const uint32_t lane = lane_id(), j = lane % G;
  if (tg.mine) take_stage<G>(g, b, nx, tg.gr, tg.w, tg.mine, tg.pairs, st, tc);
  if (__any_sync(kFull, tc.cnt != 0)) {
    sum_count<G>(b, tc);
    if (lane < (uint32_t)G) add_count(b, tc.gr * G + lane, tc.cnt, tc.deg, tc.moved);
  }
  tc = TakeCount();
  tc.gr = gr;
  tg = TakeGroup();
  tg.gr = gr;
  tg.w = width_of<G>(b, gr);
  const uint32_t slot = gr * G + j;
  tg.live = j < tg.w && slot < (uint32_t)b.nsrc && !(b.balance && __ldcg(&b.stopped[slot]));
  tg.rmf = __double2float_rn(tg.live ? __ldcg(&b.rmax[slot]) : 1.0);
  tg.mask = tg.rmf >= 0x1p-100f && tg.rmf <= 0x1p60f ? ~0u : 0u;
}

// Part `unit` of the warp's group (L loads per lane, so 32 L / G consecutive nodes; a unit is
// 8 / L of them): the nodes that cross their source's threshold go to the stage.
template <int G, int L>
__device__ __forceinline__ void take_unit(const GraphDev& g, const BatchDev& b, int nx,
                                          uint32_t unit, TakeStage<G>& st, TakeGroup& tg,
                                          TakeCount& tc) {
  constexpr uint32_t kNodes = 32 * L / G;  // nodes of a part
  constexpr uint32_t kStep = 32 / G;       // nodes per load
  constexpr uint32_t kEach = (uint32_t)(0xFFFFFFFFull / ((1ull << G) - 1));  // every G-th bit
  const uint32_t lane = lane_id(), j = lane % G, w = tg.w;
  const uint32_t n = (uint32_t)g.n;
  const uint32_t ub = unit * kNodes;
  if (ub >= n) return;
  if (b.hot_copies) {
    const uint32_t h1 = g.hot_first[(min(ub + kNodes, n) - 1) / kHotSpan + 1];
    for (uint32_t h = g.hot_first[ub / kHotSpan]; h < h1; ++h) {
      const uint32_t v = __ldg(g.hot_node + h);
      if (v >= ub && v < ub + kNodes) fold_hot<G>(g, b, tg.gr, h);
    }
  }
  const unsigned long long g0 = (unsigned long long)tg.gr * G * (unsigned long long)n;
  const uint32_t first = ub + lane / G;  // this lane's nodes: first, first + kStep, ...
  const uint32_t mine = tg.live && first < n ? (n - first + kStep - 1) / kStep : 0u;
  const double* r = b.r + g0 + (unsigned long long)first * w + j;
  const float* deg = g.fdeg + first;
  double rv[L];
  uint32_t cand = 0, above = 0;  // bit k: the node of load k may be, is above its threshold
  {
    float d[L];
#pragma unroll
    for (int k = 0; k < L; ++k) {
      rv[k] = k < mine ? __ldcg(r + (unsigned long long)(k * kStep) * w) : 0.0;
      d[k] = k < mine ? __ldg(deg + k * kStep) : 1.0f;
    }
    // threshold_fast(...): the upper word of r against the threshold's -1 and +1
#pragma unroll
    for (int k = 0; k < L; ++k) {
      const uint32_t hi = (uint32_t)((unsigned long long)__double_as_longlong(rv[k]) >> 32);
      const uint32_t t = threshold_word(tg.rmf, d[k]);
      if (k < mine && hi >= ((t - 1u) & tg.mask)) cand |= 1u << k;
      if (hi > (t + 1u | ~tg.mask)) above |= 1u << k;
    }
    above &= cand;
  }
  if (!__any_sync(kFull, cand != 0)) return;
  uint32_t open = cand & ~above;
  while (__any_sync(kFull, open != 0)) {  // a residue within 2^-19 of its threshold: rare
    if (open) {
      const uint32_t k = __ffs(open) - 1;
      open &= open - 1;
      double x = rv[0];
#pragma unroll
      for (uint32_t k2 = 1; k2 < L; ++k2) x = k2 == k ? rv[k2] : x;
      const uint32_t u = first + k * kStep;
      if (threshold_exact(x, __ldcg(&b.rmax[tg.gr * G + j]),
                          __ldg(g.row + u + 1) - __ldg(g.row + u)))
        above |= 1u << k;
    }
  }
#pragma unroll
  for (int k = 0; k < L; ++k) {
    const bool cross = (above >> k) & 1u;
    const uint32_t bal = __ballot_sync(kFull, cross);
    if (bal == 0) continue;  // warp-uniform
    uint32_t m = bal;  // one bit per node that some source takes
    if (G > 1) {
#pragma unroll
      for (int s = 1; s < G; s <<= 1) m |= m >> s;
      m &= kEach;
    }
    const uint32_t e = tg.mine + __popc(m & ((1u << (lane / G * G)) - 1u));
    if ((m >> (lane / G * G)) & 1u) {
      if (j == 0) st.u[e] = ub + k * kStep + lane / G;
      st.a[e * G + j] = cross ? rv[k] : 0.0;
    }
    if (cross) st.pair[tg.pairs + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(e * G + j);
    tg.mine += __popc(m);
    tg.pairs += __popc(bal);
  }
  if (tg.mine > kCarry) {
    take_stage<G>(g, b, nx, tg.gr, w, tg.mine, tg.pairs, st, tc);
    tg.mine = tg.pairs = 0;
  }
}

// The take: every unit of a group with a heavy round (listed in b.alist), and the listed units
// of the groups with light ones.  A warp reads consecutive units, so its counters belong to one
// or two groups; what is left of them at the end a block adds together.
// Without groups (the balanced push) sources may differ much in what they take, and in large
// scans a warp's units come from places far apart, kStretch at a time: the balanced push of 256
// sources of a 2^20-node graph 317 ms with one stretch and 299 with four, 277 and 271 with four and
// with stretches of kStretch since runs are added at once (64 sources 78.4 and 76.2).  100 of 2^18,
// whose warps scan 21 units a round, 33.3 -> 33.9 with four: so from 48 units a warp on, and a
// kernel of its own, as the loop costs the others 3%.
constexpr unsigned kStretch = 13;
constexpr unsigned long long kFarUnits = 48;
template <int G, int L, bool kFar>
__device__ void take_phase(const GraphDev& g, const BatchDev& b, int nx, uint32_t nheavy,
                           uint32_t nlist, TakeStage<G>& st) {
  const unsigned long long nwarps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
  const unsigned long long warp =
      (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  TakeCount tc;
  TakeGroup tg;
  constexpr uint32_t kParts = 8 / L;  // of a unit
  const uint32_t per = b.tiles * kParts;
  const unsigned long long units = (unsigned long long)nheavy * per;
  // A warp scans a stretch of consecutive units, with kFar several stretches far apart.
  unsigned long long x = units * warp / nwarps;
  unsigned long long end = units * (warp + 1) / nwarps;
  const unsigned pieces =
      kFar ? (unsigned)min(max(units / (nwarps * kStretch), 1ull), 64ull) : 1u;
  for (unsigned k = 0;;) {
    if (kFar && pieces > 1) {
      x = units * (k * nwarps + warp) / (pieces * nwarps);
      end = units * (k * nwarps + warp + 1) / (pieces * nwarps);
    }
    if (x < end) {
      unsigned long long ga = x / per;
      uint32_t unit = (uint32_t)(x - ga * per);
      uint32_t gr = b.ngrp == 1 ? 0u : __ldcg(&b.alist[ga]);
      for (;;) {
        if (gr != tg.gr) take_enter<G>(g, b, nx, gr, st, tg, tc);
        take_unit<G, L>(g, b, nx, unit, st, tg, tc);
        if (++x >= end) break;
        if (++unit == per) {
          unit = 0;
          gr = __ldcg(&b.alist[++ga]);
        }
      }
    }
    if (!kFar || ++k >= pieces) break;
  }
  const unsigned long long listed = (unsigned long long)nlist * kParts;
  x = listed * warp / nwarps;
  const unsigned long long lend = listed * (warp + 1) / nwarps;
  for (; x < lend; ++x) {
    const uint32_t t = __ldcg(&b.tlist[x / kParts]);
    const uint32_t gr = t / b.tiles;
    if (lane_id() == 0) b.dirty[t >> 5] = 0;  // every unit marked in the word is listed
    // a group that a joining source made heavy is scanned above
    if (!(__ldcg(&b.light[gr]) & kGroupLight)) continue;
    if (gr != tg.gr) take_enter<G>(g, b, nx, gr, st, tg, tc);
    take_unit<G, L>(g, b, nx, (t - gr * b.tiles) * kParts + (uint32_t)(x % kParts), st, tg, tc);
  }
  if (tg.mine) take_stage<G>(g, b, nx, tg.gr, tg.w, tg.mine, tg.pairs, st, tc);
  __shared__ uint32_t s_gr[kPushWarps], s_cnt[kPushWarps][G];
  __shared__ unsigned long long s_deg[kPushWarps][G];
  __shared__ double s_moved[kPushWarps][G];
  const uint32_t wid = threadIdx.x >> 5;
  sum_count<G>(b, tc);
  if (lane_id() < (uint32_t)G) {
    s_cnt[wid][lane_id()] = tc.cnt;
    s_deg[wid][lane_id()] = tc.deg;
    s_moved[wid][lane_id()] = tc.moved;
    s_gr[wid] = tc.gr;
  }
  __syncthreads();
  if (threadIdx.x < G) {
    uint32_t cnt = 0;
    unsigned long long deg = 0;
    double moved = 0.0;
    for (int k = 0; k < kPushWarps; ++k) {
      cnt += s_cnt[k][threadIdx.x];
      deg += s_deg[k][threadIdx.x];
      if (b.balance) moved = __dadd_rn(moved, s_moved[k][threadIdx.x]);
      if (k + 1 == kPushWarps || s_gr[k + 1] != s_gr[k]) {
        add_count(b, s_gr[k] * G + threadIdx.x, cnt, deg, moved);
        cnt = 0;
        deg = 0;
        moved = 0.0;
      }
    }
  }
}

// ---------------------------------------------------------------- advance

// What the advance decides for group gr from its sources' counters: its next take, and whether
// that scans every node.
template <int G>
__device__ __forceinline__ void advance_group(const BatchDev& b, int gr, bool* light,
                                              bool* heavy) {
  bool take = false, halved = false;
  unsigned long long round_edges = 0;
  unsigned long long ep[G], last[G];
#pragma unroll
  for (int j = 0; j < G; ++j) {
    const int s = min(gr * G + j, b.nsrc - 1);
    ep[j] = __ldcg(&b.stats[s].edge_pushes);
    last[j] = __ldcg(&b.last_edges[s]);
  }
#pragma unroll
  for (int j = 0; j < G; ++j) {
    const int s = gr * G + j;
    if (s >= b.nsrc) break;
    const unsigned long long pushed = ep[j] - last[j];  // this round's
    if (pushed) {
      b.last_edges[s] = ep[j];
      atomicAdd(&b.stats[s].rounds, 1u);  // a push round of this source
      round_edges += pushed;
    }
    // does the source's next take run: it found a frontier, or (balanced push) the cost
    // rule lets it go on, with the threshold halved when no node was above it
    bool on = pushed > 0;
    if (b.balance) {
      on = false;
      if (!__ldcg(&b.stopped[s])) {
        const SlotStats& st = b.stats[s];
        const double fc = __dadd_rn(__dmul_rn(b.cost_edge, (double)ep[j]),
                                    __dmul_rn(b.cost_push, (double)__ldcg(&st.pushes)));
        const double wc = __dmul_rn(__dmul_rn(__dadd_rn(1.0, -__ldcg(&st.moved)), b.bal_scale),
                                    b.cost_walk);
        if (fc >= wc) {
          b.stopped[s] = 1u;  // the frontier just taken is still spread
        } else {
          if (!pushed) {
            b.theta[s] = __dmul_rn(0.5, __ldcg(&b.theta[s]));
            halved = true;
          }
          on = true;
        }
      }
    }
    take |= on;
  }
  // the frontier just taken is spread next; a light one lets the next take scan only the
  // tiles it touches (a halved threshold needs a full scan)
  *light = take && !halved && round_edges < b.light_edges;
  *heavy = take && !*light;
}

// End of a round (one block; up to 32 groups: its first warp): the new frontier's per-group item
// prefixes, the list of groups that still push, zeroed counters for the round after, and the
// loop condition (at most b.max_rounds push rounds), which thread 0 returns, with about how long the
// round takes (its spread and its full scans) in *us.  Items of the spread
// are 32 entries, fewer where 32 would leave some of nwarps warps without one.
template <int G>
__device__ bool advance_phase(const GraphDev& g, const BatchDev& b, int nx, uint32_t nwarps,
                              float* us) {
  PushState* ps = b.ps;
  const size_t cs = (size_t)b.cnt_stride;
  const uint32_t* cnt_nx = b.slot_cnt + (size_t)nx * cs;
  const uint32_t* hcnt_nx = b.slot_cnt + (size_t)(2 + nx) * cs;
  uint32_t* cnt_cur = b.slot_cnt + (size_t)(nx ^ 1) * cs;
  uint32_t* hcnt_cur = b.slot_cnt + (size_t)(2 + (nx ^ 1)) * cs;
  const bool small = b.ngrp <= 32;
  if (small && threadIdx.x >= 32) return false;
  unsigned long long carry_g = 0, carry_h = 0, carry_heavy = 0, carry_light = 0;
  const uint32_t round = __ldcg(&ps->round) + 1;
  uint32_t span = kSpan;
  for (int base = 0; base < b.ngrp; base += blockDim.x) {
    const int gr = base + (int)threadIdx.x;
    const uint32_t c = gr < b.ngrp ? __ldcg(&cnt_nx[gr]) : 0u;
    const uint32_t h = gr < b.ngrp ? __ldcg(&hcnt_nx[gr]) : 0u;
    bool light = false, heavy = false;
    if (gr < b.ngrp) advance_group<G>(b, gr, &light, &heavy);
    if (small) {
      const uint32_t all = __reduce_add_sync(kFull, min(c, 1u << 26));
      while (span > 4 && all < span / 2 * nwarps) span /= 2;
    }
    const unsigned long long items = (c + span - 1u) / span;
    unsigned long long ge, he, gt, ht, ae, le, at, lt;
    if (small) {
      const uint32_t mh = __ballot_sync(kFull, heavy), ml = __ballot_sync(kFull, light);
      ge = warp_incl_scan(items);
      he = warp_incl_scan((unsigned long long)h);
      gt = __shfl_sync(kFull, ge, 31);
      ht = __shfl_sync(kFull, he, 31);
      ge -= items;
      he -= h;
      ae = __popc(mh & ((1u << lane_id()) - 1u));
      at = __popc(mh);
      lt = __popc(ml);
    } else {
      block_scan2(items, h, &ge, &he, &gt, &ht);
      block_scan2(heavy ? 1u : 0u, light ? 1u : 0u, &ae, &le, &at, &lt);
    }
    if (gr < b.ngrp) {
      b.gpre[gr] = carry_g + ge;
      b.hpre[gr] = carry_h + he;
      b.light[gr] =
          (uint8_t)((light ? kGroupLight : 0u) | (light || heavy ? kGroupActive : 0u));
      if (heavy) b.alist[carry_heavy + ae] = (uint32_t)gr;
      cnt_cur[gr] = 0;  // counters of the frontier just spread: they serve the round after
      hcnt_cur[gr] = 0;
    }
    carry_g += gt;
    carry_h += ht;
    carry_heavy += at;
    carry_light += lt;
  }
  // ps->round passes have run; the last one took the frontier of push round ps->round (the
  // first pass only finds F_0), so going on is allowed while that is <= the cap.  Another pass
  // is needed while a group takes again or a taken frontier waits for its spread (of a source
  // the cost rule just stopped).
  const bool more = carry_heavy + carry_light > 0 || carry_g > 0 || carry_h > 0;
  const bool go = more && round <= b.max_rounds;
  if (threadIdx.x == 0) {
    b.gpre[b.ngrp] = carry_g;
    b.hpre[b.ngrp] = carry_h;
    ps->ngroups = carry_g;
    ps->nhub = carry_h;
    // edge pushes at 2.5e11 a second, scanned residues at 6 TB/s
    *us = G * (float)(carry_g * span * ((float)g.m / (float)g.n) + carry_h * kHubChunk) * 4e-6f +
          (float)carry_heavy * (float)b.tiles * (kUnit * 8 / 6e6f);
    b.ctl->nheavy = (uint32_t)carry_heavy;
    b.ctl->nlist = 0;
    b.ctl->span = span;
    ps->cur = nx;
    ps->round = round;
    b.work[0] = 0;  // dynamic work counters of the next spread
    b.work[16] = 0;
    if (more && !go) atomicOr(b.err, kErrPushNotConverged);
    ps->go = go ? 1u : 0u;
  }
  return go;
}

// After the last round: copies of hot nodes that no take has added (sources that the cost rule
// stopped).
template <int G>
__device__ void finish_phase(const GraphDev& g, const BatchDev& b) {
  if (!b.hot_copies) return;
  const unsigned long long nwarps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
  const unsigned long long warp =
      (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const unsigned long long total = (unsigned long long)b.ngrp * g.nhot;
  for (unsigned long long x = warp; x < total; x += nwarps)
    fold_hot<G>(g, b, (uint32_t)(x / g.nhot), (uint32_t)(x % g.nhot));
}

// ---------------------------------------------------------------- kernels

// Zeroes `bytes` bytes at a 16-byte aligned address with all threads of the grid.
__device__ __forceinline__ void grid_zero(void* p, unsigned long long bytes) {
  const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned long long nt = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long quads = bytes / 16;
  for (unsigned long long i = t; i < quads; i += nt) ((uint4*)p)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (unsigned long long i = quads * 16 + t; i < bytes; i += nt) ((uint8_t*)p)[i] = 0;
}

// The state a push starts from, but for what seed_phase sets.
__device__ __forceinline__ void zero_phase(const GraphDev& g, const BatchDev& b) {
  const unsigned long long cells =
      (unsigned long long)min(b.ngrp * b.gw, b.lay) * (unsigned long long)g.n;
  grid_zero(b.r, cells * sizeof(double));
  grid_zero(b.res, cells * sizeof(double));
  grid_zero(b.hotr, (unsigned long long)b.hot_copies * b.lgrp * g.nhot * b.gw * sizeof(double));
  grid_zero(b.dirty, ((unsigned long long)b.lgrp * b.tiles + 31) / 32 * 4);
  grid_zero(b.slot_cnt, 4ull * b.cnt_stride * sizeof(uint32_t));
  grid_zero(b.last_edges, (unsigned long long)b.lay * sizeof(unsigned long long));
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    b.work[0] = b.work[16] = 0;
    b.ctl->nheavy = b.ctl->nlist = 0;
  }
}

// What a block keeps in shared memory of the launch's meetings (thread 0 writes it).
struct MeetState {
  uint32_t arrivals;  // up to the last meeting
  uint32_t value;
  uint32_t begin;     // kBeginTake or kBeginSpread, with the round's parity
};
constexpr uint32_t kBeginTake = 0u, kBeginSpread = 2u;

// The word of the last meeting with work: the arrivals up to it + 1 (0: none yet), and what follows.
constexpr uint32_t kStop = 0u, kGo = 1u, kGoCut = 3u;  // kGoCut: as far as the end of the spread
__device__ __forceinline__ unsigned long long meet_word(const BatchDev& b) {
  return *(volatile unsigned long long*)(b.meet + kMeetWord);
}
__device__ __forceinline__ void write_meet_word(const BatchDev& b, uint32_t arrivals,
                                                uint32_t next) {
  *(volatile unsigned long long*)(b.meet + kMeetWord) =
      ((unsigned long long)arrivals + 1ull) << 2 | next;
}
constexpr unsigned long long kClocksPerUs = 2000;  // about (2070 MHz at most)
constexpr uint32_t kClosed = 0x80000000u;  // in kMeetEntered: the launch leaves, blocks are missing
constexpr uint32_t kNotBegun = 2u;  // PushState::go where not even the start was done
constexpr long long kPatience = 100 * (long long)kClocksPerUs;

// Enters the launch; true if all its blocks have, within kPatience of the first (they do within a
// microsecond on an idle device), or however long it takes where the launch guarantees it
// (`sure`).  At the start of a push (`fresh`) a block clears its share of the state as it enters,
// and when all have the first block sets the sources' residues.  A block that comes after the first
// has given up leaves at once and clears nothing.
template <int G>
__device__ bool all_enter(const GraphDev& g, const BatchDev& b, bool fresh, bool sure,
                          MeetState& ms) {
  if (threadIdx.x == 0) {
    const uint32_t old = atomicAdd(b.meet + kMeetEntered, 1u);
    ms.value = old & kClosed ? 0u : 1u;
    ms.arrivals = old;
  }
  __syncthreads();
  const bool in = ms.value != 0, first = ms.arrivals == 0;
  __syncthreads();  // ms free
  if (!in) return false;
  if (fresh) {
    zero_phase(g, b);
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(b.meet + kMeetReady, 1u);
    }
  }
  if (first) {  // block-uniform
    if (threadIdx.x == 0) {
      volatile uint32_t* entered = b.meet + kMeetEntered;
      volatile uint32_t* ready = b.meet + kMeetReady;
      const long long t0 = clock64();
      uint32_t n = *entered, polls = 0;
      bool all;
      for (;;) {
        all = n == gridDim.x && (!fresh || *ready == n);
        if (all || ++polls > kMaxPolls) break;
        // blocks that have entered a fresh push finish clearing before the launch gives up
        if (!sure && n < gridDim.x && clock64() - t0 > kPatience && (!fresh || *ready == n) &&
            atomicCAS(b.meet + kMeetEntered, n, n | kClosed) == n)
          break;
        n = *entered;
      }
      if (polls > kMaxPolls) atomicOr(b.err, kErrBarrier);
      __threadfence();
      ms.value = all ? 1u : 0u;
    }
    __syncthreads();
    const bool all = ms.value != 0;
    if (all && fresh) seed_phase<G>(g, b);
    if (!all && fresh && threadIdx.x == 0) b.ps->go = kNotBegun;
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      write_meet_word(b, 0u, all ? kGo : kStop);
    }
  }
  if (threadIdx.x == 0) {
    unsigned long long w;
    uint32_t polls = 0;
    while ((w = meet_word(b)) == 0 && ++polls <= kMaxPolls)
      if (polls > 64) __nanosleep(100);
    if (polls > kMaxPolls) atomicOr(b.err, kErrBarrier);
    __threadfence();
    ms.arrivals = 0;
    ms.value = (uint32_t)w & 1u;
  }
  __syncthreads();
  const bool go = ms.value != 0;
  __syncthreads();
  return go;
}

// Meeting point of all blocks.  With `work`, block 0 (always the same: its instructions stay in that
// SM's cache; run by whichever block came last they cost 10 us of fetches a round) runs it when all
// have arrived and lets the others go on, and the value (kStop, kGo, kGoCut) that its thread 0
// returned comes back to every thread.  The waits are bounded: a block that gives up reports kErrBarrier and gets 0, as
// then do the others.
template <typename F>
__device__ uint32_t grid_meet(const BatchDev& b, MeetState& ms, bool work, F f) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(b.meet + kMeetArrived, 1u);
    const uint32_t all = ms.arrivals + gridDim.x;
    uint32_t polls = 0, v = kGo;
    if (work && blockIdx.x != 0) {
      unsigned long long w;
      while ((uint32_t)((w = meet_word(b)) >> 2) <= all && ++polls <= kMaxPolls)
        if (polls > 64) __nanosleep(100);
      v = (uint32_t)w & 3u;
    } else {
      volatile uint32_t* arrived = b.meet + kMeetArrived;
      while (*arrived < all && ++polls <= kMaxPolls)
        if (polls > 64) __nanosleep(100);
    }
    if (polls > kMaxPolls) {
      atomicOr(b.err, kErrBarrier);
      v = kStop;
    }
    ms.arrivals = all;
    ms.value = v;
    __threadfence();
  }
  __syncthreads();
  uint32_t v = ms.value;
  if (work && blockIdx.x == 0 && v != kStop) {
    v = f();
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      write_meet_word(b, ms.arrivals, v);
      ms.value = v;
    }
    __syncthreads();
    v = ms.value;
  }
  __syncthreads();
  return v;
}

template <int G>
union PushShared {
  TakeStage<G> take[kPushWarps];
  SpreadStage<G> spread[kPushWarps];
};

// Units per SM below which a batch is small: fewer than two for each of the 32 warps of 4 blocks.
// (One query of a 2^14-node graph: 0.49 ms of push with whole units, 0.39 with quarters; from
// two units a warp on the two differ by less than a percent.)
constexpr unsigned long long kSmallUnits = 64;
// 4 resident blocks (64 registers): 3 (no spilled register) took 130.4 ms where 4 take 121.5, 5
// 138 (256 sources of a 2^20-node R-MAT graph).
constexpr int kPushBlocks = 4;
// With kParts the launch runs a part of the push (PushPart).  (A template parameter: with the clock
// and the host's words a launch for one source of a small graph spills more.)
template <int G, int L, bool kParts, bool kFar = false>
__global__ void __launch_bounds__(kPushThreads, kPushBlocks)
    k_push(const __grid_constant__ GraphDev g, const __grid_constant__ BatchDev b,
           const __grid_constant__ PushPart part) {
  __shared__ PushShared<G> sh;
  __shared__ MeetState ms;
  __shared__ long long s_started;
  const PushState* ps = b.ps;
  const PushCtl* ctl = b.ctl;
  const uint32_t wid = threadIdx.x >> 5;
  const bool fresh = !(kParts && part.resume);
  const bool leads = blockIdx.x == 0 && threadIdx.x == 0;
  if (kParts && leads) {
    uint32_t* other = part.turn ? b.meet - kMeetWords : b.meet + kMeetWords;  // the next launch's
    other[kMeetArrived] = other[kMeetEntered] = other[kMeetReady] = 0;
    *(unsigned long long*)(other + kMeetWord) = 0;
  }
  if (!fresh) {
    const uint32_t state = __ldcg(&ps->go);
    if (state != 1u) {  // through, or not begun
      if (part.host && leads)
        *(volatile uint32_t*)&part.host->go[part.turn] = state ? kPushMissing : kPushDone;
      return;
    }
  }
  if (!all_enter<G>(g, b, fresh, part.sure != 0, ms)) {
    if (leads) {
      if (part.host)
        *(volatile uint32_t*)&part.host->go[part.turn] = kPushMissing;
      else
        atomicOr(b.err, kErrMissing);
    }
    return;
  }
  if (kParts && leads) s_started = clock64();
  uint32_t go = kGo;
  // Where the first round begins is kept in shared memory: seen by the compiler it makes a copy of
  // the loop, whose fetches cost a small push a microsecond a round.
  if (kParts) {
    if (threadIdx.x == 0) {
      uint32_t begin = kBeginTake;
      if (!fresh) {
        begin = (uint32_t)__ldcg(&ps->cur);
        if (__ldcg(&ctl->cut))
          begin ^= 1u;
        else
          begin |= kBeginSpread;
      }
      ms.begin = begin;
    }
    __syncthreads();
  }
  for (int nx = kParts ? (int)(ms.begin & 1u) : 0; go != kStop; nx ^= 1) {
    if (!kParts || !(ms.begin & kBeginSpread)) {
      take_phase<G, L, kFar>(g, b, nx, __ldcg(&ctl->nheavy), __ldcg(&ctl->nlist), sh.take[wid]);
      go = grid_meet(b, ms, true, [&] {
        bool stop = false;
        if (kParts && threadIdx.x == 0) {
          stop = part.slice != kNoSlice &&
                 (unsigned long long)(clock64() - s_started) >= kClocksPerUs * part.slice;
          if (part.stops) stop |= *(volatile uint32_t*)&part.host->stop != 0;
        }
        float us = 0.0f;
        const bool on = advance_phase<G>(g, b, nx, gridDim.x * kPushWarps, &us) && !stop;
        const bool cut = kParts && on && part.slice != kNoSlice && us >= (float)part.slice;
        if (kParts && threadIdx.x == 0) b.ctl->cut = cut ? 1u : 0u;
        return cut ? kGoCut : on ? kGo : kStop;
      });
      if (go == kStop) break;
    }
    spread_phase<G, G == 1 && L == 8>(g, b, nx, __ldcg(&ps->nhub), __ldcg(&ps->ngroups),
                                      __ldcg(&ctl->span), sh.spread[wid]);
    if (kParts) {
      if (threadIdx.x == 0) ms.begin = kBeginTake;
      if (go == kGoCut) break;
    }
    go = grid_meet(b, ms, false, [] { return kGo; });
  }
  const bool left = kParts && __ldcg(&ps->go);
  if (!left) finish_phase<G>(g, b);
  if (kParts && part.host && leads)
    *(volatile uint32_t*)&part.host->go[part.turn] =
        left && !(*(volatile uint32_t*)b.err & kErrBarrier) ? kPushLeft : kPushDone;
}

// The phases on their own.
template <int G>
__global__ void __launch_bounds__(kPushThreads) k_push_seed(const __grid_constant__ GraphDev g,
                                                            const __grid_constant__ BatchDev b) {
  seed_phase<G>(g, b);
}
__global__ void __launch_bounds__(kPushThreads) k_push_zero(const __grid_constant__ GraphDev g,
                                                            const __grid_constant__ BatchDev b) {
  zero_phase(g, b);
}
template <int G>
__global__ void __launch_bounds__(kPushThreads, kPushBlocks)
    k_push_spread(const __grid_constant__ GraphDev g, const __grid_constant__ BatchDev b) {
  __shared__ SpreadStage<G> stage[kPushWarps];
  if (b.ctl->cut) return;  // done by the launch before
  spread_phase<G, G == 1>(g, b, b.ps->cur, b.ps->nhub, b.ps->ngroups,
                  b.ctl->span, stage[threadIdx.x >> 5]);
}
template <int G>
__global__ void __launch_bounds__(kPushThreads, kPushBlocks)
    k_push_take(const __grid_constant__ GraphDev g, const __grid_constant__ BatchDev b) {
  __shared__ TakeStage<G> stage[kPushWarps];
  take_phase<G, 8, false>(g, b, b.ps->cur ^ 1, b.ctl->nheavy,
                          b.ctl->nlist, stage[threadIdx.x >> 5]);
}
template <int G>
__global__ void __launch_bounds__(kPushThreads) k_push_advance(const __grid_constant__ GraphDev g,
                                                               const __grid_constant__ BatchDev b) {
  const int nx = b.ps->cur ^ 1;
  __syncthreads();
  float us;
  advance_phase<G>(g, b, nx, 0u, &us);
  if (threadIdx.x == 0) b.ctl->cut = 0;
}
template <int G>
__global__ void __launch_bounds__(kPushThreads) k_push_finish(const __grid_constant__ GraphDev g,
                                                              const __grid_constant__ BatchDev b) {
  finish_phase<G>(g, b);
}

// Sources joining a batch between two push rounds (serving): slots [first, first + k) (their
// sources and r_max already in place, the places of their residues zeroed with the batch's) get
// r(s) = 1; their groups enter the next take, scanned whole, and the prefixes are extended over
// groups that are new.  One block.  The push of a source depends only on its own residues, so a
// source that joins later runs the same rounds as it would from the start.
template <int G>
__global__ void __launch_bounds__(kPushThreads) k_push_join(const __grid_constant__ GraphDev g,
                                                            const __grid_constant__ BatchDev b,
                                                            int first, int k) {
  PushState* ps = b.ps;
  const int old_groups = (first + G - 1) / G;
  const unsigned long long gtot = ps->ngroups, htot = ps->nhub;
  for (int i = threadIdx.x; i < k; i += blockDim.x) {
    const int slot = first + i;
    const uint32_t src = (uint32_t)b.sources[slot], gr = (uint32_t)slot / G;
    b.r[(unsigned long long)gr * G * (unsigned long long)g.n +
        (unsigned long long)src * width_of<G>(b, gr) + slot % G] = 1.0;
  }
  for (int gr = old_groups + (int)threadIdx.x; gr < b.ngrp; gr += blockDim.x) {
    b.gpre[gr + 1] = gtot;
    b.hpre[gr + 1] = htot;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t nheavy = b.ctl->nheavy;
    for (int gr = first / G; gr < b.ngrp; ++gr) {
      const uint32_t s = gr < old_groups ? b.light[gr] : 0u;
      if (!(s & kGroupActive) || (s & kGroupLight)) b.alist[nheavy++] = (uint32_t)gr;
      b.light[gr] = kGroupActive;
    }
    b.ctl->nheavy = nheavy;
    ps->go = 1;
  }
}

// The frontier test of the take on given (r, r_max, d) triples.
__global__ void k_threshold_table(const double* r, const double* rm, const uint32_t* d,
                                  uint8_t* out, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const float rmf = __double2float_rn(rm[i]);
  const bool fast = rmf >= 0x1p-100f && rmf <= 0x1p60f;
  out[i] = above_threshold(r[i], rm[i], rmf, fast, d[i]) ? 1 : 0;
}

// [slot][n] arrays to and from the batch's grouped ones.
__global__ void k_regroup(double* grouped, double* rows, unsigned long long n, int lay, int gw,
                          int nsrc, int to_rows) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (int slot = blockIdx.y; slot < nsrc; slot += gridDim.y) {
    const int gr = slot / gw, w = min(gw, lay - gr * gw);
    double* p = grouped + (unsigned long long)gr * gw * n + slot % gw;
    double* q = rows + (unsigned long long)slot * n;
    for (unsigned long long v = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += stride) {
      if (to_rows) q[v] = p[v * w]; else p[v * w] = q[v];
    }
  }
}

template <int G, int L, bool kParts, bool kFar = false>
cudaError_t push_t(const GraphDev& g, const BatchDev& b, int num_sms, const PushPart& part,
                   cudaStream_t st) {
  const int per_sm = resident_blocks((const void*)k_push<G, L, kParts, kFar>, kPushThreads);
  if (per_sm == 0) return cudaErrorInvalidConfiguration;
  // every SM at least once; more blocks only where a full scan has work for them
  const unsigned long long parts = (unsigned long long)b.ngrp * b.tiles * (8 / L);
  const unsigned long long want = (parts + kPushWarps - 1) / kPushWarps;
  unsigned blocks = (unsigned)num_sms;
  while (blocks < want && blocks < (unsigned)(num_sms * per_sm)) blocks += (unsigned)num_sms;
  BatchDev bd = b;
  bd.meet += part.turn * kMeetWords;
  const void* kernel = (const void*)k_push<G, L, kParts, kFar>;
  GraphDev gd = g;
  PushPart pt = part;
  void* args[] = {&gd, &bd, &pt};
  if (part.sure) return cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(kPushThreads), args, 0, st);
  return cudaLaunchKernel(kernel, dim3(blocks), dim3(kPushThreads), args, 0, st);
}

template <int G>
cudaError_t push_any(const GraphDev& g, const BatchDev& b, int num_sms, const PushPart* part,
                     cudaStream_t st) {
  // a small batch's full scan has few units: a warp reads a quarter of one, which shortens a round
  const unsigned long long units = (unsigned long long)b.ngrp * b.tiles;
  const bool small = units < kSmallUnits * (unsigned)num_sms;
  if (part->slice == kNoSlice && !part->resume)
    return small ? push_t<G, 2, false>(g, b, num_sms, *part, st)
                 : push_t<G, 8, false>(g, b, num_sms, *part, st);
  if (small) return push_t<G, 2, true>(g, b, num_sms, *part, st);
  if (G == 1 && units >= kFarUnits * (unsigned)num_sms * kPushBlocks * kPushWarps)
    return push_t<G, 8, true, G == 1>(g, b, num_sms, *part, st);
  return push_t<G, 8, true>(g, b, num_sms, *part, st);
}

template <int G>
cudaError_t push_round_t(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st) {
  const int spread_per_sm = resident_blocks((const void*)k_push_spread<G>, kPushThreads);
  const int take_per_sm = resident_blocks((const void*)k_push_take<G>, kPushThreads);
  if (spread_per_sm == 0 || take_per_sm == 0) return cudaErrorInvalidConfiguration;
  k_push_spread<G><<<num_sms * spread_per_sm, kPushThreads, 0, st>>>(g, b);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_push_take<G><<<num_sms * take_per_sm, kPushThreads, 0, st>>>(g, b);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_push_advance<G><<<1, kPushThreads, 0, st>>>(g, b);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_threshold_table(const double* r, const double* rm, const uint32_t* d,
                                   uint8_t* out, int count, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  k_threshold_table<<<(count + 255) / 256, 256, 0, st>>>(r, rm, d, out, count);
  return cudaGetLastError();
}

cudaError_t launch_push(const GraphDev& g, const BatchDev& b, int num_sms, const PushPart* part,
                        cudaStream_t st) {
  return b.gw == 1 ? push_any<1>(g, b, num_sms, part, st) : push_any<4>(g, b, num_sms, part, st);
}

template <int G>
cudaError_t load_phases() {
  cudaFuncAttributes a;
  for (const void* k : {(const void*)k_push_seed<G>, (const void*)k_push_spread<G>,
                        (const void*)k_push_take<G>, (const void*)k_push_advance<G>,
                        (const void*)k_push_finish<G>, (const void*)k_push_join<G>}) {
    const cudaError_t e = cudaFuncGetAttributes(&a, k);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t load_push_phases() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, (const void*)k_push_zero);
  if (e == cudaSuccess) e = load_phases<1>();
  return e == cudaSuccess ? load_phases<4>() : e;
}

cudaError_t launch_push_start(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st) {
  k_push_zero<<<num_sms * 8, kPushThreads, 0, st>>>(g, b);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (b.gw == 1)
    k_push_seed<1><<<1, kPushThreads, 0, st>>>(g, b);
  else
    k_push_seed<4><<<1, kPushThreads, 0, st>>>(g, b);
  return cudaGetLastError();
}

cudaError_t launch_push_round(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st) {
  return b.gw == 1 ? push_round_t<1>(g, b, num_sms, st) : push_round_t<4>(g, b, num_sms, st);
}

cudaError_t launch_push_finish(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st) {
  if (b.gw == 1)
    k_push_finish<1><<<num_sms, kPushThreads, 0, st>>>(g, b);
  else
    k_push_finish<4><<<num_sms, kPushThreads, 0, st>>>(g, b);
  return cudaGetLastError();
}

cudaError_t launch_push_join(const GraphDev& g, const BatchDev& b, int first, int k,
                             cudaStream_t st) {
  if (k <= 0) return cudaSuccess;
  if (b.gw == 1)
    k_push_join<1><<<1, kPushThreads, 0, st>>>(g, b, first, k);
  else
    k_push_join<4><<<1, kPushThreads, 0, st>>>(g, b, first, k);
  return cudaGetLastError();
}

cudaError_t launch_regroup(double* grouped, double* rows, const BatchDev& b, int64_t n,
                           bool to_rows, int num_sms, cudaStream_t st) {
  uint64_t bx = ((uint64_t)n + 255) / 256;
  const uint64_t most = ((uint64_t)num_sms * 32 + b.nsrc - 1) / b.nsrc;
  if (bx > most) bx = most;
  k_regroup<<<dim3((unsigned)bx, (unsigned)b.nsrc), 256, 0, st>>>(
      grouped, rows, (unsigned long long)n, b.lay, b.gw, b.nsrc, to_rows ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace fora
