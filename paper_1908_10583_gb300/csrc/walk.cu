// Walk phase of Alg. 2 over a batch of sources.
//
//   k_residual_count / k_residual_scan / k_residual_emit:
//     R = {(slot, v) : r(v) > 0} in ascending slot; omega_v = ceil(r(v) * C) with
//     C = omega / r_sum (Alg. 2); exclusive offsets of omega_v over R (one flat
//     walk index space for all sources) and the fixed-point weight
//     W_v = rint(r(v)/omega_v * 2^63) of every walk from v (Alg. 2: a_v r_sum/omega).
//   k_walks:
//     walk g in [0, W) belongs to the entry i with offset[i] <= g < offset[i+1] and is
//     walk j = g - offset[i] of node v; it reads its own Philox4x32-10 stream with
//     counter (c, j, v, s) and stops with probability alpha at every node
//     (Section 2.1); count[end] += 1 and acc[end] += W_v.
#include <algorithm>

#include "fora_engine.cuh"

namespace fora {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kResidualThreads = 256;

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// Philox4x32-10 with its ten round keys given (BatchDev::round_key, kernel parameters, so
// the key schedule costs no instruction per round).
__device__ __forceinline__ uint4 philox_rk(uint4 c, const uint2* rk) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ rk[i].x, lo1, hi0 ^ c.w ^ rk[i].y, lo0);
  }
  return c;
}

// omega_v = ceil(RN64(r * C)); W_v = rint((r / omega_v) * 2^63)
__device__ __noinline__ unsigned long long walks_exact(double r, double C) {
  return (unsigned long long)ceil(__dmul_rn(r, C));
}
__device__ __forceinline__ unsigned long long weight_of(double r, double omega) {
  return __double2ull_rn(__dmul_rn(__ddiv_rn(r, omega), 0x1p63));
}

constexpr uint32_t kOmegaUndecided = 0xFFFFFFFFu;

// omega_v for r > 0 without FP64 arithmetic where FP32 decides it (this GPU issues about
// two FP64 operations per clock per SM).  rf = r truncated to 23 mantissa bits (rf <= r
// < rf (1 + 2^-23)) and cf = RN32(C) give P = RN32(rf * cf) within 2^-22 of V = r * C,
// and T = RN64(V) is within 2^-53 of V; so T lies strictly inside (P (1 - 2^-20),
// P (1 + 2^-20)), and when that band holds no integer, ceil(T) = floor(band) + 1.
// Returns kOmegaUndecided otherwise (an integer in the band, P >= 2^22, r outside FP32's
// normal range, or C outside [1, 2^100], which `fast` excludes).
__device__ __forceinline__ uint32_t walks_fast(double r, float cf, bool fast) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(r);
  const uint32_t hi = (uint32_t)(bits >> 32);
  const uint32_t ex = hi >> 20;  // r > 0: no sign bit
  if (!fast || ex < 897u || ex > 1150u) return kOmegaUndecided;
  const float rf =
      __uint_as_float(((ex - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | ((uint32_t)bits >> 29));
  const float pr = rf * cf;
  if (!(pr < 0x1p22f)) return kOmegaUndecided;
  const float lo = pr * (1.0f - 0x1p-20f), up = pr * (1.0f + 0x1p-20f);
  const float fl = floorf(lo);
  if (floorf(up) != fl || fl == lo) return kOmegaUndecided;
  return (uint32_t)fl + 1u;
}

// omega_v of this lane's residue (0 when r = 0); every lane of the warp must call it.
__device__ __forceinline__ unsigned long long walks_of(double r, double C, float cf, bool fast) {
  const bool live = __double_as_longlong(r) != 0;  // residues are >= 0, never -0
  const uint32_t f = live ? walks_fast(r, cf, fast) : 0u;
  unsigned long long w = f;
  const bool undecided = f == kOmegaUndecided;
  if (__any_sync(kFull, undecided)) {  // rare: r * C within 2^-20 of an integer
    if (undecided) w = walks_exact(r, C);
  }
  return w;
}

// The residue the walks sample: r, or (1 - alpha) r with zero-hop pruning (Section 4.1).
__device__ __forceinline__ double sampled(const BatchDev& b, double r) {
  return b.zero_hop ? __dmul_rn(__dadd_rn(1.0, -b.alpha), r) : r;
}

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const T t = __shfl_up_sync(kFull, x, off);
    if ((int)(threadIdx.x & 31) >= off) x += t;
  }
  return x;
}

// Block-wide exclusive scan of (count, walks) pairs; also returns the block totals.
// Every thread of the block must call it.
__device__ __forceinline__ void block_excl_scan2(unsigned long long c, unsigned long long w,
                                                 unsigned long long* ce, unsigned long long* we,
                                                 unsigned long long* ct, unsigned long long* wt) {
  __shared__ unsigned long long sc[32], sw[32];
  __shared__ unsigned long long tc, tw;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned long long ci = warp_incl_scan(c), wi = warp_incl_scan(w);
  if (lane == 31) { sc[wid] = ci; sw[wid] = wi; }
  __syncthreads();
  if (wid == 0) {
    const unsigned long long a = lane < nw ? sc[lane] : 0, bb = lane < nw ? sw[lane] : 0;
    const unsigned long long ai = warp_incl_scan(a), bi = warp_incl_scan(bb);
    if (lane < nw) { sc[lane] = ai - a; sw[lane] = bi - bb; }
    if (lane == 31) { tc = ai; tw = bi; }
  }
  __syncthreads();
  *ce = sc[wid] + ci - c;
  *we = sw[wid] + wi - w;
  *ct = tc;
  *wt = tw;
  __syncthreads();
}

// The residual list in three kernels.  A warp's unit is a share of the nodes of one group of
// sources (G side by side, as the push leaves them; lane % G is the source), so neither pass
// over the residues needs a block barrier: k_residual_count counts each source's entries and
// walks per unit, k_residual_scan turns them into offsets (one block), k_residual_emit writes
// the entries, computing the weights (an FP64 division each) on packed lanes.
struct UnitRange {
  uint32_t gr, k, w;          // group, share, sources side by side
  uint32_t beg, end;          // its nodes
  unsigned long long g0;      // of the group's residues
};
template <int G>
__device__ __forceinline__ bool unit_range(const GraphDev& g, const BatchDev& b, UnitRange* u) {
  const unsigned long long warp =
      ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (warp >= (unsigned long long)b.ngrp * b.units) return false;
  u->gr = (uint32_t)(warp / b.units);
  u->k = (uint32_t)(warp - (unsigned long long)u->gr * b.units);
  u->w = min((uint32_t)G, (uint32_t)b.lay - u->gr * G);
  u->beg = (uint32_t)((unsigned long long)g.n * u->k / b.units);
  u->end = (uint32_t)((unsigned long long)g.n * (u->k + 1) / b.units);
  u->g0 = (unsigned long long)u->gr * G * (unsigned long long)g.n;
  return true;
}

constexpr int kResidualLoads = 4;  // residues a lane reads before it uses any

template <int G>
__global__ void __launch_bounds__(kResidualThreads) k_residual_count(GraphDev g, BatchDev b) {
  UnitRange u;
  if (!unit_range<G>(g, b, &u)) return;  // whole warps
  constexpr uint32_t kStep = 32 / G;
  const uint32_t lane = threadIdx.x & 31, j = lane % G, slot = u.gr * G + j;
  const bool mine = j < u.w && slot < (uint32_t)b.nsrc;
  const float cf = __double2float_rn(b.walk_scale);
  const bool fast = cf >= 1.0f && cf <= 0x1p100f;
  unsigned long long walks = 0;
  uint32_t cnt = 0, some = 0;  // entries (at least one walk), residues above 0
  double sum = 0.0;
  for (uint32_t v0 = u.beg; v0 < u.end; v0 += kStep * kResidualLoads) {
    double r[kResidualLoads];
#pragma unroll
    for (int k = 0; k < kResidualLoads; ++k) {
      const uint32_t v = v0 + k * kStep + lane / G;
      r[k] = mine && v < u.end ? b.r[u.g0 + (unsigned long long)v * u.w + j] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kResidualLoads; ++k) {
      // an entry of R needs at least one walk (omega_v = 0 only if r * C underflows)
      const unsigned long long w = walks_of(sampled(b, r[k]), b.walk_scale, cf, fast);
      if (__double_as_longlong(r[k]) != 0) {
        cnt += w > 0 ? 1u : 0u;
        walks += w;
        ++some;
        sum += r[k];
      }
    }
  }
#pragma unroll
  for (int o = 16; o >= G; o >>= 1) {
    cnt += __shfl_xor_sync(kFull, cnt, o);
    some += __shfl_xor_sync(kFull, some, o);
    walks += __shfl_xor_sync(kFull, walks, o);
    sum += __shfl_xor_sync(kFull, sum, o);
  }
  if (lane < (uint32_t)G && mine) {
    const size_t at = (size_t)slot * b.units + u.k;
    b.unit_cnt[at] = cnt;
    b.unit_walks[at] = walks;
    if (some) {
      atomicAdd(&b.stats[slot].residual_nodes, (unsigned long long)some);
      atomicAdd(&b.stats[slot].walks, walks);
      atomicAdd(&b.stats[slot].rsum, sum);
    }
  }
}

// One block: exclusive scan of the units' counts, slot after slot; totals; per-source walk limit.
// A thread scans consecutive units.
__global__ void __launch_bounds__(1024) k_residual_scan(BatchDev b) {
  const uint32_t total = (uint32_t)b.nsrc * (uint32_t)b.units;
  const uint32_t per = (total + blockDim.x - 1) / blockDim.x;
  const uint32_t beg = min(threadIdx.x * per, total), end = min(beg + per, total);
  unsigned long long c = 0, w = 0;
  for (uint32_t i = beg; i < end; ++i) {
    c += b.unit_cnt[i];
    w += b.unit_walks[i];
  }
  unsigned long long ce, we, ct, wt;
  block_excl_scan2(c, w, &ce, &we, &ct, &wt);
  for (uint32_t i = beg; i < end; ++i) {
    const unsigned long long ci = b.unit_cnt[i], wi = b.unit_walks[i];
    b.unit_cnt[i] = ce;
    b.unit_walks[i] = we;
    ce += ci;
    we += wi;
  }
  if (threadIdx.x == 0) {
    b.totals[0] = ct;
    b.totals[1] = wt;
    b.wr_offset[ct] = wt;
  }
  for (int s = threadIdx.x; s < b.nsrc; s += blockDim.x)
    if (b.stats[s].walks > 0xFFFFFFFFull) atomicOr(b.err, kErrWalkOverflow);
}

// The entries of up to 32 * kResidualLoads residues of a warp's unit, packed.
struct ResidualStage {
  double r[32 * kResidualLoads];
  uint32_t omega[32 * kResidualLoads];
  uint32_t pos[32 * kResidualLoads];   // place and walk offset within the unit's entries of
  uint32_t woff[32 * kResidualLoads];  // the source
  uint32_t v[32 * kResidualLoads];     // node - first node of the unit, times G, plus lane % G
};

template <int G>
__global__ void __launch_bounds__(kResidualThreads) k_residual_emit(GraphDev g, BatchDev b) {
  __shared__ ResidualStage stages[kResidualThreads / 32];
  UnitRange u;
  if (!unit_range<G>(g, b, &u)) return;  // whole warps
  ResidualStage& st = stages[threadIdx.x >> 5];
  constexpr uint32_t kStep = 32 / G;
  const uint32_t lane = threadIdx.x & 31, j = lane % G, slot = u.gr * G + j;
  const bool mine = j < u.w && slot < (uint32_t)b.nsrc;
  const unsigned long long base_c = mine ? b.unit_cnt[(size_t)slot * b.units + u.k] : 0ull;
  const unsigned long long base_w = mine ? b.unit_walks[(size_t)slot * b.units + u.k] : 0ull;
  const float cf = __double2float_rn(b.walk_scale);
  const bool fast = cf >= 1.0f && cf <= 0x1p100f;
  constexpr uint32_t kSame = (uint32_t)(0xFFFFFFFFull / ((1ull << G) - 1));  // lanes of source 0
  uint32_t done_c = 0, done_w = 0;  // entries and walks of this lane's source so far
  for (uint32_t v0 = u.beg; v0 < u.end; v0 += kStep * kResidualLoads) {
    double r[kResidualLoads];
#pragma unroll
    for (int k = 0; k < kResidualLoads; ++k) {
      const uint32_t v = v0 + k * kStep + lane / G;
      r[k] = mine && v < u.end ? b.r[u.g0 + (unsigned long long)v * u.w + j] : 0.0;
    }
    uint32_t staged = 0;
#pragma unroll
    for (int k = 0; k < kResidualLoads; ++k) {
      const double x = sampled(b, r[k]);
      const uint32_t omega = (uint32_t)walks_of(x, b.walk_scale, cf, fast);  // below 2^32 (scan)
      const bool live = omega > 0;
      const uint32_t m = __ballot_sync(kFull, live);
      if (m == 0) continue;  // warp-uniform
      const uint32_t same = m & (kSame << j);  // this source's
      uint32_t incl = omega;                   // its walks up to this lane
#pragma unroll
      for (int o = G; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, o);
        if ((int)lane >= o) incl += t;
      }
      if (live) {
        const uint32_t at = staged + __popc(m & ((1u << lane) - 1u));
        st.r[at] = x;
        st.omega[at] = omega;
        st.pos[at] = done_c + __popc(same & ((1u << lane) - 1u));
        st.woff[at] = done_w + incl - omega;
        st.v[at] = (v0 - u.beg + k * kStep) * G + lane;
      }
      staged += __popc(m);
      done_c += __popc(same);
      done_w += __shfl_sync(kFull, incl, 32 - G + j);
    }
    __syncwarp();
    for (uint32_t e0 = 0; e0 < staged; e0 += 32) {
      const uint32_t e = e0 + lane;
      const bool have = e < staged;
      const uint32_t vj = have ? st.v[e] : 0u;
      const unsigned long long pos = __shfl_sync(kFull, base_c, vj % G) + (have ? st.pos[e] : 0u);
      const unsigned long long off = __shfl_sync(kFull, base_w, vj % G) + (have ? st.woff[e] : 0u);
      if (have && FORA_IN_RANGE(b.err, pos, (unsigned long long)b.nsrc * g.n)) {
        b.wr_entry[pos] =
            ((unsigned long long)(u.gr * G + vj % G) << 32) | (unsigned long long)(u.beg + vj / G);
        b.wr_offset[pos] = off;
        b.wr_weight[pos] = weight_of(st.r[e], (double)st.omega[e]);
      }
    }
    __syncwarp();
  }
}

constexpr int kWalkThreads = 384;
constexpr int kWalkWarps = kWalkThreads / 32;
constexpr int kIndexedThreads = 256;
constexpr uint32_t kMaxSteps = 16384u;

// Largest i in [0, nR) with off[i] <= g (off non-decreasing, off[0] = 0 <= g);
// warp-cooperative 32-ary search, every lane gets the answer.
__device__ __forceinline__ unsigned long long warp_find_entry(const unsigned long long* off,
                                                              unsigned long long nR,
                                                              unsigned long long g) {
  const unsigned lane = threadIdx.x & 31;
  unsigned long long lo = 0, hi = nR;
  while (hi - lo > 32) {
    const unsigned long long step = (hi - lo + 31) / 32;
    const unsigned long long p = lo + lane * step;
    const unsigned bal = __ballot_sync(kFull, p < hi && off[p] <= g);
    lo += (unsigned long long)(31 - __clz(bal)) * step;
    hi = min(lo + step, hi);
  }
  const unsigned long long p = lo + lane;
  const unsigned bal = __ballot_sync(kFull, p < hi && off[p] <= g);
  return lo + (unsigned long long)(31 - __clz(bal));
}

// Walks a warp takes from the flat walk range at a time: fewer when the walks would not
// give every warp several such shares, so that a small query still uses every warp.
__device__ __forceinline__ uint32_t share_walks(unsigned long long W, unsigned long long nwarps,
                                                uint32_t most) {
  const unsigned long long share = (W + nwarps - 1) / nwarps / 6;
  return share >= most ? most : (uint32_t)((share + 32) / 32 * 32);
}

// The walk kernels' copy of the degree classes (GraphDev::wcls) in shared memory.
__device__ __forceinline__ void load_classes(const GraphDev& g, uint2* cls) {
  for (int c = threadIdx.x; c < g.ncls; c += blockDim.x) cls[c] = g.wcls[c];
}

// {first edge, out-degree} of the node of a record: from its class, without a load from
// global memory, or (when `need`) from the list of the nodes without a class.  cls has an
// entry at ncls too.
__device__ __forceinline__ uint2 node_row(const GraphDev& g, const uint2* cls, uint32_t rec,
                                          bool need) {
  const uint32_t c = rec >> g.wbits, id = walk_id(g, rec);
  const uint2 k = cls[c];
  uint2 r = make_uint2(k.x + id * k.y, k.y);
  if (c >= (uint32_t)g.ncls && need) r = g.wesc[id];
  return r;
}

constexpr uint32_t kCapped = 0x80000000u;

// The rest of a walk whose neighbour draw at x came out with a low word below d on its first
// try, word `pos - 1` of its Philox block cb - 1 (Lemire's method rejects the try when the
// low word is below 2^32 mod d, probability below d / 2^32): the words are taken one at a
// time from there, tries, stop tests and moves in stream order.  It evaluates the block again
// rather than keep its words alive.  Returns the record of the end node (low word) and the walk's moves (high word), with kCapped set in the latter when
// the walk reaches the step cap (or, never in practice, 64 rejected tries in a row).
__device__ __forceinline__ unsigned long long walk_rest(const uint32_t* wcol, const uint2* wesc,
                                                     const uint2* cls, uint32_t ncls,
                                                     uint32_t wbits, int pos, uint32_t cb,
                                                     uint32_t j, uint32_t v, uint32_t s, uint2 key,
                                                     uint32_t t_alpha, uint32_t x, uint32_t steps) {
  uint4 blk = philox4x32_10(make_uint4(cb - 1, j, v, s), key);
  auto next = [&]() -> uint32_t {
    if (pos == 4) {
      blk = philox4x32_10(make_uint4(cb, j, v, s), key);
      ++cb;
      pos = 0;
    }
    const uint32_t w = pos == 0 ? blk.x : pos == 1 ? blk.y : pos == 2 ? blk.z : blk.w;
    ++pos;
    return w;
  };
  --pos;  // the move at x takes its first try again
  for (bool first = true;; first = false) {
    if (!first) {
      if (next() < t_alpha) break;
      if (steps >= kMaxSteps) { steps |= kCapped; break; }
    }
    const uint32_t c = x >> wbits, id = x & ((1u << wbits) - 1u);
    uint2 r;
    if (c >= ncls) {
      r = wesc[id];
    } else {
      const uint2 k = cls[c];
      r = make_uint2(k.x + id * k.y, k.y);
    }
    const uint32_t reject_below = (0u - r.y) % r.y;
    unsigned long long m = (unsigned long long)next() * r.y;
    int tries = 0;
    while ((uint32_t)m < reject_below && ++tries <= 64) m = (unsigned long long)next() * r.y;
    if (tries > 64) { steps |= kCapped; break; }
    x = wcol[r.x + (uint32_t)(m >> 32)];
    ++steps;
  }
  return ((unsigned long long)steps << 32) | x;
}

// A warp's window on the residual entries: the data of up to 32 consecutive entries, twice
// (walks of the window before are still running while the next one's are started), and the
// entry of each of the window's walks.
constexpr uint32_t kWindowWalks = 512;
constexpr uint32_t kWalkShare = 4096;
struct WalkWindow {
  uint4 walk[64];  // node v, source, record of v, low word of the entry's walk offset
  uint4 end[64];   // weight (low, high), slot
  unsigned long long pos, stop;  // the warp's share of the walk range that is still to start
  unsigned long long entry;      // the entry of walk pos
  unsigned long long next;       // the warp's next share
  uint8_t map[kWindowWalks];
};

// The next window of the warp's share (or of its next share) into half `half` of the window:
// its number of walks, 0 when no walk is left.
__device__ __forceinline__ uint32_t next_window(const GraphDev& g, const BatchDev& b,
                                                WalkWindow& w, uint32_t half) {
  const uint32_t lane = threadIdx.x & 31;
  const unsigned long long W = b.totals[1], nR = b.totals[0];
  unsigned long long pos = w.pos, stop = w.stop, entry = w.entry;
  if (pos >= stop) {
    const unsigned long long nwarps = (unsigned long long)gridDim.x * kWalkWarps;
    const uint32_t share = share_walks(W, nwarps, kWalkShare);
    const unsigned long long mine = w.next;
    pos = mine * share;
    if (pos >= W) return 0;
    __syncwarp();
    if (lane == 0) w.next = nwarps + atomicAdd(b.walk_next, 1ull);
    stop = min(pos + share, W);
    entry = warp_find_entry(b.wr_offset, nR, pos);
  }
  const unsigned long long i = entry + lane;
  const bool live = i < nR;
  // offsets relative to pos; the entry of walk pos has offset 0, the others follow
  const unsigned long long o = live ? b.wr_offset[i] : ~0ull;
  const unsigned long long past = entry + 32 < nR ? b.wr_offset[entry + 32] : W;
  const uint32_t rel = o <= pos ? 0u : (uint32_t)min(o - pos, 0x7FFFFFFFull);
  if (live) {
    const unsigned long long ent = b.wr_entry[i], wgt = b.wr_weight[i];
    const uint32_t slot = (uint32_t)(ent >> 32), v = (uint32_t)ent;
    w.walk[half * 32 + lane] = make_uint4(v, (uint32_t)b.sources[slot], g.wid[v], (uint32_t)o);
    w.end[half * 32 + lane] = make_uint4((uint32_t)wgt, (uint32_t)(wgt >> 32), slot, 0u);
  }
  const uint32_t cnt =
      (uint32_t)min(min(stop, past) - pos, (unsigned long long)kWindowWalks);
  for (uint32_t k = lane; k < cnt + lane; k += 32) {  // every lane takes part in every step
    int lo = 0, hi = 31;  // largest entry whose offset is at most k
#pragma unroll
    for (int t = 0; t < 5; ++t) {
      const int mid = (lo + hi + 1) >> 1;
      if (__shfl_sync(kFull, rel, mid) <= k) lo = mid; else hi = mid - 1;
    }
    if (k < cnt) w.map[k] = (uint8_t)lo;
  }
  const uint32_t passed = (uint32_t)__popc(__ballot_sync(kFull, rel <= cnt));  // entries begun
  __syncwarp();
  if (lane == 0) {
    w.pos = pos + cnt;
    w.stop = stop;
    w.entry = pos + cnt == past ? entry + 32 : entry + passed - 1;
  }
  __syncwarp();
  return cnt;
}

// Adds the moves of the lanes with `due` to the counters of their sources (every lane of the
// warp calls it): one atomic when they are of one source.  (One per lane queued 2 * 10^5
// atomics on the counter of a single-source query, 0.1 ms.)
__device__ __forceinline__ void flush_moves(const BatchDev& b, bool due, uint32_t& moves,
                                            uint32_t slot) {
  const uint32_t some = __ballot_sync(kFull, due && moves > 0);
  if (some == 0) return;
  const uint32_t first = __shfl_sync(kFull, slot, __ffs(some) - 1);
  if (__all_sync(kFull, !due || moves == 0 || slot == first)) {
    const uint32_t sum = __reduce_add_sync(kFull, due ? moves : 0u);  // each below 2^26
    if ((threadIdx.x & 31) == 0) atomicAdd(&b.stats[first].walk_steps, (unsigned long long)sum);
  } else if (due && moves) {
    atomicAdd(&b.stats[slot].walk_steps, (unsigned long long)moves);
  }
  if (due) moves = 0;
}

// The walk kernel.  The flat walk range goes to the warps in shares, in order, so the walks in
// flight at any time are a narrow window of the source-major walk space and their end sums
// stay in L2.  A warp goes through its share in windows of up to 32 residual entries, staged in
// shared memory with the entry of each walk; each lane runs one walk and takes the window's
// next unstarted walk when it ends (walk lengths are geometric: with a fixed share of walks per
// lane a warp would wait for its longest share).  A walk's registers are its record x, number j
// and state st = (block << 6 | place of its entry in the window); the entry's data stay in the
// window, whose other half takes the next entries once no running walk needs it, so no lane
// waits for the last walk of a window.
//
// One loop iteration consumes exactly one Philox block of every walk, so the ten rounds run on
// full warps: a plain walk takes the words as stop test, move, stop test, move, a zero-hop
// walk as move, stop test, move, stop test (its first move has no stop test).  A walk that
// stops inside a block leaves the block's remaining words unused, as its stream definition
// does; every block before took two moves, so a walk at block c has made 2 c moves.  A
// neighbour try that Lemire's method may reject moves the walk off this block alignment:
// walk_rest finishes it.
//
// Bounds: one gathered sector per move at 3.0e11 a second (one per clock and SM) and one
// reduction per walk at 2.0e11; the latency of an iteration's two dependent gathers (the
// slowest of 32 lanes' sectors) and instruction issue keep it above them.  Hence one record
// per move, the tests and moves without branches, and little state in registers: 40, for 4
// blocks of 384 threads.  Measured against a kernel with two lookups per move, an 18-register
// walk state, one counter atomic per lane and source, and chunks whose last walks the warp
// waited for: 256 sources of a 2^20-node R-MAT graph (0.35 of the rule's r_max) 119.3 -> 63.2
// ms, 1.75e11 moves/s; 64 of 2^18 14.5 -> 8.1 ms; 100 of a 200003-node graph without hubs 13.9
// -> 7.1 ms; one of 2^20 0.99 -> 0.63 ms.  Two walks per lane (54 registers) took 70.4 ms of
// the first, 320 or 448 threads 75 and 68, shares of 1024, 2048 or 8192 walks 71, 65.5, 65.6.
//
// kTally: the end of walk g is summed into b.acc; otherwise it is stored in b.walk_dest[g]
// (a walk index) or summed and counted (b.wcount).
constexpr uint32_t kIdle = 0xFFFFFFFFu;
template <int kMinBlocks, bool kZeroHop, bool kTally>
__global__ void __launch_bounds__(kWalkThreads, kMinBlocks) k_walks(GraphDev g, BatchDev b) {
  __shared__ WalkWindow windows[kWalkWarps];
  __shared__ uint2 cls[kMaxWalkClasses + 1];
  if (*b.err) return;
  load_classes(g, cls);
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t t_alpha = b.alpha_threshold;
  WalkWindow& win = windows[wid];
  if (lane == 0) {
    win.pos = win.stop = 0;
    win.next = (unsigned long long)blockIdx.x * kWalkWarps + wid;
  }
  __syncwarp();

  uint32_t half = 0;                // the half of the window whose walks are being started
  uint32_t cnt = 0, next_walk = 0;  // next_walk of the window's cnt walks are started
  bool more = true;
  uint32_t x = 0, j = 0, st = kIdle;
  uint32_t moves = 0, mslot = 0xFFFFFFFFu;  // moves of this lane's walks of slot mslot
  for (;;) {
    if (next_walk >= cnt && more) {  // warp-uniform
      // does a running walk need the other half?
      if (!__any_sync(kFull, st != kIdle && ((st >> 5) & 1u) != half)) {
        half ^= 1u;
        cnt = next_window(g, b, win, half);
        next_walk = 0;
        more = cnt > 0;
      }
    }
    const uint32_t idle = __ballot_sync(kFull, st == kIdle);
    const uint32_t i = next_walk + (uint32_t)__popc(idle & ((1u << lane) - 1u));
    if (st == kIdle && i < cnt) {
      const uint32_t e = half * 32 + win.map[i];
      const uint4 w = win.walk[e];
      x = w.z;
      j = (uint32_t)win.pos - cnt + i - w.w;
      st = e;
    }
    next_walk = min(next_walk + (uint32_t)__popc(idle), cnt);
    if (!__any_sync(kFull, st != kIdle)) {
      if (!more) break;
      continue;
    }

    const uint4 w = win.walk[st & 63u];
    const uint4 o = philox_rk(make_uint4(st >> 6, j, w.x, w.y), b.round_key);
    static_assert(kMaxSteps % 2 == 0, "the cap is met before a block's first move");
    uint32_t steps = 2u * (st >> 6);
    bool have = st != kIdle;
    bool go = have && (kZeroHop || o.x >= t_alpha);  // makes the block's first move
    if (go && steps >= kMaxSteps) {
      atomicOr(b.err, kErrWalkCap);
      have = go = false;
    }
    if (!FORA_IN_RANGE(b.err, walk_id(g, x), g.n)) have = go = false;
    uint2 r = node_row(g, cls, x, go);
    unsigned long long m = (unsigned long long)(kZeroHop ? o.x : o.y) * r.y;
    bool again = go && (uint32_t)m < r.y;  // a try that may be rejected
    const bool one = go && !again;
    uint32_t e = r.x + (uint32_t)(m >> 32);
    if (one && FORA_IN_RANGE(b.err, e, g.m)) x = g.wcol[e];
    go = one && (kZeroHop ? o.y : o.z) >= t_alpha;  // makes the second
    r = node_row(g, cls, x, go);
    m = (unsigned long long)(kZeroHop ? o.z : o.w) * r.y;
    const bool retry = go && (uint32_t)m < r.y;
    const bool two = go && !retry;
    again |= retry;
    e = r.x + (uint32_t)(m >> 32);
    if (two && FORA_IN_RANGE(b.err, e, g.m)) x = g.wcol[e];
    steps += (one ? 1u : 0u) + (two ? 1u : 0u);
    bool stop = have && !(kZeroHop ? two && o.w >= t_alpha : two);
    if (__any_sync(kFull, again)) {  // rare
      if (again) {
        const unsigned long long end =
            walk_rest(g.wcol, g.wesc, cls, (uint32_t)g.ncls, (uint32_t)g.wbits,
                      (one ? 4 : 2) - (kZeroHop ? 1 : 0), (st >> 6) + 1, j, win.walk[st & 63u].x,
                      win.walk[st & 63u].y, b.round_key[0], t_alpha, x, steps);
        x = (uint32_t)end;
        steps = (uint32_t)(end >> 32);
        stop = (steps & kCapped) == 0;
        if (!stop) {
          atomicOr(b.err, kErrWalkCap);
          have = false;
        }
      }
    }
    uint32_t slot = 0;
    if (stop) {
      // the walk stops at x (Section 2.1): its weight is added there (Alg. 2), or its end is
      // recorded in a walk index (Section 3.3); its moves count for its source
      const uint32_t id = walk_id(g, x);
      const uint4 end = win.end[st & 63u];
      slot = end.z;
      const unsigned long long at = (unsigned long long)slot * b.ends + end_place(g, id);
      if (!kTally && b.walk_dest) {
        b.walk_dest[j + win.walk[st & 63u].w] = id;  // an index has fewer than 2^32 walks
      } else if (FORA_IN_RANGE(b.err, id, g.n) && FORA_IN_RANGE(b.err, slot, b.nsrc)) {
        if (!kTally) atomicAdd(&b.wcount[at], 1u);
        atomicAdd(&b.acc[at], ((unsigned long long)end.y << 32) | end.x);
      }
    }
    const bool due = stop && (slot != mslot || moves >= 1u << 25);
    if (__any_sync(kFull, due)) flush_moves(b, due, moves, mslot);
    if (stop) {
      mslot = slot;
      moves += steps;
    }
    st = have && !stop ? st + 64u : kIdle;
  }
  flush_moves(b, true, moves, mslot);
}

// Edge records of the walks (GraphDev::wcol), one warp per node.
__global__ void k_walk_records(GraphDev g, uint32_t* wcol) {
  const unsigned long long warp = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  for (unsigned long long v = warp; v < (unsigned long long)g.n; v += nwarps) {
    const uint32_t rec = g.wid[v], c = rec >> g.wbits, id = walk_id(g, rec);
    const uint32_t rb = g.row[v], d = g.row[v + 1] - rb;
    const uint32_t to = c < (uint32_t)g.ncls ? g.wcls[c].x + id * d : g.wesc[id].x;
    for (uint32_t k = lane; k < d; k += 32) wcol[to + k] = g.wid[g.col[rb + k]];
  }
}

// FORA+ (Section 3.3): the residue whose walk count is the index's omega_max(v).
__global__ void k_index_residue(GraphDev g, double* r, double rmax) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long v = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
       v < (unsigned long long)g.n; v += stride)
    r[v] = __dmul_rn(rmax, (double)(g.row[v + 1] - g.row[v]));
}

// The walk phase served from a walk index: walk j of the residue (slot, v) ends at
// idx_dest[idx_off[v] + j] (the j-th stored walk from v) instead of being simulated.  The sources
// of a group that hold a residue at v share its first walks, so the kernels go through the
// residues by node and a warp adds, for each of 32 / G walks, the weights of the G sources to
// their sums, which lie side by side (BatchDev::side_by_side): one sector takes all four.  The
// additions bound it: 7.2 ms for 64 sources of a 2^20-node graph, 1.57e9 walks, 2.2e11 a second.
// (Source by source, from a list of entries, they took 11.2 ms: 1.4e11 a second, what scattered
// 8-byte atomics with this graph's skew reach; the list took 0.9 ms more.)
// k_indexed_nodes takes the nodes of up to kIndexedMost walks and lists the others, whose walks
// k_indexed_hubs takes in chunks of kIndexedMost; a list serves as many groups as it can count
// (index_list_groups), so large batches take the two kernels more than once.
// A residue of more walks than are stored (above the index's r_max) sets kErrIndexRange; only the
// stored ones are taken.
constexpr int kIndexedPer = 4;    // steps of a warp (of 32 / G walks) whose loads are in flight
constexpr int kIndexedLoads = 8;  // residues a lane reads before it uses any

// This lane's source of group gr: its residue's walks and weight at node v, at most the stored
// ones.  Every lane of the warp must call it.
template <int G>
__device__ __forceinline__ void indexed_entry(const BatchDev& b, double r, uint32_t stored,
                                              uint32_t* omega, unsigned long long* weight) {
  const float cf = __double2float_rn(b.walk_scale);
  const bool fast = cf >= 1.0f && cf <= 0x1p100f;
  const double x = sampled(b, r);
  const uint32_t w = (uint32_t)walks_of(x, b.walk_scale, cf, fast);  // below 2^32 (scan)
  *weight = w ? weight_of(x, (double)w) : 0ull;
  if (w > stored) atomicOr(b.err, kErrIndexRange);
  *omega = min(w, stored);
}

// Adds the walk that ends at dest to this lane's source's sum (source j of w in the group).
__device__ __forceinline__ void add_end(const GraphDev& g, const BatchDev& b,
                                        unsigned long long base, uint32_t w, uint32_t j,
                                        uint32_t dest, unsigned long long weight) {
  const unsigned long long at = base + (unsigned long long)end_place(g, dest) * w + j;
  if (b.want_count) atomicAdd(&b.wcount[at], 1u);
  atomicAdd(&b.acc[at], weight);
}

template <int G>
__global__ void __launch_bounds__(kIndexedThreads) k_indexed_nodes(
    GraphDev g, BatchDev b, const unsigned long long* idx_off, const uint32_t* idx_dest) {
  if (__any_sync(kFull, *b.err != 0)) return;  // whole warps
  constexpr uint32_t kPer = 32 / G;                // nodes of a batch, walks of a step
  constexpr uint32_t kNodes = kPer * kIndexedLoads;  // of a warp
  const uint32_t lane = threadIdx.x & 31, j = lane % G, q = lane / G;
  const unsigned long long n = (unsigned long long)g.n, units = (n + kNodes - 1) / kNodes;
  const unsigned long long warp =
      ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (warp >= units * (unsigned long long)(b.end_grp - b.first_grp)) return;  // whole warps
  const uint32_t gr = (uint32_t)b.first_grp + (uint32_t)(warp / units);
  const uint32_t v0 = (uint32_t)(warp % units * kNodes);
  const uint32_t w = min((uint32_t)G, (uint32_t)b.lay - gr * G);
  const bool mine = j < w && gr * G + j < (uint32_t)b.nsrc;
  const unsigned long long g0 = (unsigned long long)gr * G * n;
  const unsigned long long base = (unsigned long long)gr * G * b.ends;
  double r[kIndexedLoads];
#pragma unroll
  for (int k = 0; k < kIndexedLoads; ++k) {
    const unsigned long long v = v0 + k * kPer + q;
    r[k] = mine && v < n ? b.r[g0 + v * w + j] : 0.0;
  }
#pragma unroll
  for (int k = 0; k < kIndexedLoads; ++k) {
    if (!__any_sync(kFull, __double_as_longlong(r[k]) != 0)) continue;
    const uint32_t v = (uint32_t)min((unsigned long long)(v0 + k * kPer + q), n - 1);
    const unsigned long long off = idx_off[v];
    uint32_t omega;
    unsigned long long weight;
    indexed_entry<G>(b, r[k], (uint32_t)(idx_off[v + 1] - off), &omega, &weight);
    uint32_t most = omega;  // of the node's sources
#pragma unroll
    for (int o = 1; o < G; o <<= 1) most = max(most, __shfl_xor_sync(kFull, most, o));
    if (most > kIndexedMost) {
      if (j == 0) {
        const unsigned long long chunks = (most - 1) / kIndexedMost + 1;
        const unsigned long long at = atomicAdd(b.walk_next, (1ull << kListBits) | chunks);
        const unsigned long long i = at >> kListBits;
        if (FORA_IN_RANGE(b.err, i, (unsigned long long)b.nsrc * n)) {
          b.wr_entry[i] = (unsigned long long)gr << 32 | v;
          b.wr_offset[i] = at & ((1ull << kListBits) - 1ull);
        }
      }
      most = 0;
    }
    // the batch's nodes have ceil(most / kPer) steps each, one after the other
    const uint32_t steps = (most + kPer - 1) / kPer;
    uint32_t incl = steps;
#pragma unroll
    for (int o = G; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, incl, o);
      if ((int)lane >= o) incl += t;
    }
    const uint32_t total = __shfl_sync(kFull, incl, 31);
    for (uint32_t t0 = 0; t0 < total; t0 += kIndexedPer) {
      uint32_t dest[kIndexedPer];
      unsigned long long add[kIndexedPer];
      bool have[kIndexedPer];
#pragma unroll
      for (int u = 0; u < kIndexedPer; ++u) {
        const uint32_t t = min(t0 + u, total - 1u);
        const uint32_t node = __popc(__ballot_sync(kFull, j == 0 && incl <= t));
        const uint32_t first = __shfl_sync(kFull, incl - steps, node * G);
        const uint32_t walk = (t - first) * kPer + q;
        const unsigned long long at = __shfl_sync(kFull, off, node * G) + walk;
        add[u] = __shfl_sync(kFull, weight, node * G + j);
        have[u] = walk < __shfl_sync(kFull, omega, node * G + j) && t0 + u < total;
        dest[u] = have[u] ? idx_dest[at] : 0u;
      }
#pragma unroll
      for (int u = 0; u < kIndexedPer; ++u)
        if (have[u]) add_end(g, b, base, w, j, dest[u], add[u]);
    }
  }
}

template <int G>
__global__ void __launch_bounds__(kIndexedThreads) k_indexed_hubs(
    GraphDev g, BatchDev b, const unsigned long long* idx_off, const uint32_t* idx_dest) {
  if (__any_sync(kFull, *b.err != 0)) return;  // whole warps
  constexpr uint32_t kPer = 32 / G;
  const uint32_t lane = threadIdx.x & 31, j = lane % G, q = lane / G;
  const unsigned long long listed = *b.walk_next;
  const unsigned long long nodes = listed >> kListBits;
  const unsigned long long chunks = listed & ((1ull << kListBits) - 1ull);
  const unsigned long long nwarps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
  for (unsigned long long x = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
       x < chunks; x += nwarps) {
    const unsigned long long i = warp_find_entry(b.wr_offset, nodes, x);
    const unsigned long long entry = b.wr_entry[i];
    const uint32_t gr = (uint32_t)(entry >> 32), v = (uint32_t)entry;
    const uint32_t w = min((uint32_t)G, (uint32_t)b.lay - gr * G);
    const bool mine = j < w && gr * G + j < (uint32_t)b.nsrc;
    const unsigned long long base = (unsigned long long)gr * G * b.ends;
    const double r =
        mine ? b.r[(unsigned long long)gr * G * g.n + (unsigned long long)v * w + j] : 0.0;
    const unsigned long long off = idx_off[v];
    uint32_t omega;
    unsigned long long weight;
    indexed_entry<G>(b, r, (uint32_t)(idx_off[v + 1] - off), &omega, &weight);
    const uint32_t beg = (uint32_t)(x - b.wr_offset[i]) * kIndexedMost;  // below 2^32
    const uint32_t end = omega - min(omega, beg) < kIndexedMost ? omega : beg + kIndexedMost;
#pragma unroll 1
    for (uint32_t s = 0; s < kIndexedMost; s += kPer * kIndexedPer) {
      const uint32_t k = beg + s;  // the chunk's last walk is below 2^32, the next chunk need not be
      if (!__any_sync(kFull, k < end)) break;
      uint32_t dest[kIndexedPer];
#pragma unroll
      for (int u = 0; u < kIndexedPer; ++u) {
        const uint32_t walk = k + u * kPer + q;
        dest[u] = walk < end ? idx_dest[off + walk] : 0u;
      }
#pragma unroll
      for (int u = 0; u < kIndexedPer; ++u)
        if (k + u * kPer + q < end) add_end(g, b, base, w, j, dest[u], weight);
    }
  }
}

__global__ void k_unpack_ends(GraphDev g, BatchDev b, uint32_t* cnt, unsigned long long* acc) {
  const unsigned long long n = (unsigned long long)g.n;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (int slot = blockIdx.y; slot < b.nsrc; slot += gridDim.y) {
    const unsigned long long g0 = (unsigned long long)slot * n;
    const EndSums sums = end_sums(b, slot);
    for (unsigned long long v = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += stride) {
      const unsigned long long at = sums.at(end_place(g, walk_id(g, g.wid[v])));
      if (cnt) cnt[g0 + v] = b.wcount[at];
      if (acc) acc[g0 + v] = b.acc[at];
    }
  }
}

__global__ void k_philox_table(const uint32_t* ck, uint32_t* out, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const uint4 o = philox4x32_10(make_uint4(ck[6 * i], ck[6 * i + 1], ck[6 * i + 2], ck[6 * i + 3]),
                                make_uint2(ck[6 * i + 4], ck[6 * i + 5]));
  out[4 * i] = o.x; out[4 * i + 1] = o.y; out[4 * i + 2] = o.z; out[4 * i + 3] = o.w;
}

}  // namespace

int residual_units(int64_t n, int nsrc) {
  int64_t units = kMaxUnits / nsrc;
  units = std::min<int64_t>(units, (n + 511) / 512);
  units = std::min<int64_t>(units, kMaxSlotUnits);
  return (int)std::max<int64_t>(units, 1);
}

template <int G>
cudaError_t residuals_t(const GraphDev& g, const BatchDev& b, cudaStream_t st) {
  const unsigned long long warps = (unsigned long long)b.ngrp * b.units;
  const unsigned blocks = (unsigned)((warps * 32 + kResidualThreads - 1) / kResidualThreads);
  k_residual_count<G><<<blocks, kResidualThreads, 0, st>>>(g, b);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_residual_scan<<<1, 1024, 0, st>>>(b);
  e = cudaGetLastError();
  if (e != cudaSuccess || b.side_by_side) return e;  // indexed walks need no list
  k_residual_emit<G><<<blocks, kResidualThreads, 0, st>>>(g, b);
  return cudaGetLastError();
}

cudaError_t launch_residuals(const GraphDev& g, const BatchDev& b, cudaStream_t st) {
  return b.gw == 1 ? residuals_t<1>(g, b, st) : residuals_t<4>(g, b, st);
}

// Walk kernel instances for 3, 4 or 5 resident blocks per SM (the register budget the
// compiler gets); b.walk_blocks picks one (launch shape only).
template <int kMinBlocks, bool kZeroHop, bool kTally>
cudaError_t launch_walks_t(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st) {
  const int per_sm =
      resident_blocks((const void*)k_walks<kMinBlocks, kZeroHop, kTally>, kWalkThreads);
  if (per_sm == 0) return cudaErrorInvalidConfiguration;
  k_walks<kMinBlocks, kZeroHop, kTally><<<num_sms * per_sm, kWalkThreads, 0, st>>>(g, b);
  return cudaGetLastError();
}

template <bool kZeroHop>
cudaError_t launch_walks_zh(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st) {
  const bool tally = !b.walk_dest && !b.want_count;
  switch (b.walk_blocks) {
    case 3:
      return tally ? launch_walks_t<3, kZeroHop, true>(g, b, num_sms, st)
                   : launch_walks_t<3, kZeroHop, false>(g, b, num_sms, st);
    case 5:
      return tally ? launch_walks_t<5, kZeroHop, true>(g, b, num_sms, st)
                   : launch_walks_t<5, kZeroHop, false>(g, b, num_sms, st);
    default:
      return tally ? launch_walks_t<4, kZeroHop, true>(g, b, num_sms, st)
                   : launch_walks_t<4, kZeroHop, false>(g, b, num_sms, st);
  }
}

cudaError_t launch_walks(const GraphDev& g, const BatchDev& b, int num_sms, cudaStream_t st) {
  return b.zero_hop ? launch_walks_zh<true>(g, b, num_sms, st)
                    : launch_walks_zh<false>(g, b, num_sms, st);
}

cudaError_t launch_index_residue(const GraphDev& g, double* r, double rmax, cudaStream_t st) {
  k_index_residue<<<1024, 256, 0, st>>>(g, r, rmax);
  return cudaGetLastError();
}

template <int G>
cudaError_t walks_indexed_t(const GraphDev& g, BatchDev b, int num_sms, int groups,
                            const unsigned long long* idx_off, const uint32_t* idx_dest,
                            cudaStream_t st) {
  constexpr unsigned long long kNodes = 32 / G * kIndexedLoads, kWarps = kIndexedThreads / 32;
  const int per_sm = resident_blocks((const void*)k_indexed_hubs<G>, kIndexedThreads);
  if (per_sm == 0) return cudaErrorInvalidConfiguration;
  for (int first = 0; first < b.ngrp; first = b.end_grp) {
    cudaError_t e = cudaSuccess;
    if (first > 0) e = cudaMemsetAsync(b.walk_next, 0, sizeof(*b.walk_next), st);
    if (e != cudaSuccess) return e;
    b.first_grp = first;
    b.end_grp = groups < b.ngrp - first ? first + groups : b.ngrp;
    const unsigned long long warps = ((unsigned long long)g.n + kNodes - 1) / kNodes *
                                     (unsigned long long)(b.end_grp - first);
    k_indexed_nodes<G><<<(unsigned)((warps + kWarps - 1) / kWarps), kIndexedThreads, 0, st>>>(
        g, b, idx_off, idx_dest);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_indexed_hubs<G><<<num_sms * per_sm, kIndexedThreads, 0, st>>>(g, b, idx_off, idx_dest);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_walks_indexed(const GraphDev& g, const BatchDev& b, int num_sms, int groups,
                                 const unsigned long long* idx_off, const uint32_t* idx_dest,
                                 cudaStream_t st) {
  const int64_t most = index_list_groups(g.n, b.gw);
  if (groups < 1 || groups > most) groups = (int)std::min<int64_t>(most, b.ngrp);
  return b.gw == 1 ? walks_indexed_t<1>(g, b, num_sms, groups, idx_off, idx_dest, st)
                   : walks_indexed_t<4>(g, b, num_sms, groups, idx_off, idx_dest, st);
}

cudaError_t launch_unpack_ends(const GraphDev& g, const BatchDev& b, uint32_t* cnt,
                               unsigned long long* acc, int num_sms, cudaStream_t st) {
  uint64_t bx = ((uint64_t)g.n + 255) / 256;
  const uint64_t most = ((uint64_t)num_sms * 32 + b.nsrc - 1) / b.nsrc;
  if (bx > most) bx = most;
  k_unpack_ends<<<dim3((unsigned)bx, (unsigned)b.nsrc), 256, 0, st>>>(g, b, cnt, acc);
  return cudaGetLastError();
}

cudaError_t launch_walk_records(const GraphDev& g, uint32_t* wcol, int num_sms, cudaStream_t st) {
  k_walk_records<<<num_sms * 8, 256, 0, st>>>(g, wcol);
  return cudaGetLastError();
}

cudaError_t launch_philox_table(const uint32_t* ctr_key, uint32_t* out, int count,
                                cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  k_philox_table<<<(count + 127) / 128, 128, 0, st>>>(ctr_key, out, count);
  return cudaGetLastError();
}

}  // namespace fora
