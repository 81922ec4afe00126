// Estimate and top-k select (the query returns the k nodes with the largest
// estimated PPR, Section 2.1; ties go to the smaller id).
//
// Every element t of a row gets the 96-bit key  Z = bits(pi_hat(t)) : ~t.  pi_hat >= 0,
// so its IEEE bits order like its value, and ~t orders equal values by ascending id;
// keys are unique, so the k largest keys are exactly the answer.
//   k_topk_first    histogram of the upper 18 bits of the estimate (sign, exponent, 6 bits of
//                   mantissa), clamped to the 4096 bins from 2^-63 to 2: estimates crowd into
//                   few exponents, so a digit of the exponent alone would not separate them.  A
//                   row's last block picks the bin that holds the k-th largest key as the row's
//                   prefix; the row is done once the keys above the bin and its own fit the sort.
//   k_topk_levels   for rows that are not (more equal or near-equal values than the sort takes,
//                   or a k-th value outside the bins): the next 12 bits of the keys with the
//                   row's prefix, and so on.  The blocks of a row take its parts as they come,
//                   and whichever finishes a level's last part picks its digit.
//   k_topk_collect  every key from the prefix on goes to the candidate list; a row's last block
//                   sorts it (bitonic, in shared memory) and writes the first k.
// Two passes over the rows; HBM bounds large ones, the launches and the sort small ones.
// 24 rows of 10^6 estimates: 40 us, 4 us where no level is left, 50 us (the two passes at the
// measured copy rate: 58); fora_topk 522 -> 128 us.  (As 19 launches:
// eight levels of 12 bits from the top, whether a row had use for them or not, then collect and
// sort.)  fora_topk of rows whose k-th value is 0 (eight levels): one row of 2^25 values 0.92 ms,
// 24 of 2^20 0.88, 256 of 2^14 0.48.  With eight blocks of a cluster for each row's levels, however
// long the row, they took 10.9, 1.06 and 1.03, as 19 launches 1.26, 1.28 and 0.74.
#include <algorithm>

#include "fora_engine.cuh"

namespace fora {

namespace {

typedef unsigned __int128 u128;

__device__ __forceinline__ u128 key_of(double e, uint32_t t) {
  return ((u128)(unsigned long long)__double_as_longlong(e) << 32) | (u128)(~t);
}

// One row of the grid per group of sources, kEstValues values per block: the walk ends are
// gathered (by walk id), so few groups at a time keep their sectors in L2 until all four sums
// of each are used.  (64 sources in flight: 5.3 ms for 256 sources of 2^20 nodes.)
constexpr int kEstThreads = 256;
constexpr int kEstPer = 8;
constexpr int kEstValues = kEstThreads * kEstPer;
template <int G>
__global__ void __launch_bounds__(kEstThreads) k_estimate(GraphDev g, BatchDev b, double* est) {
  const unsigned long long n = (unsigned long long)g.n;
  const uint32_t j = threadIdx.x % G;
  const unsigned long long v0 =
      (unsigned long long)blockIdx.x * (kEstValues / G) + threadIdx.x / G;
  for (int gr = blockIdx.y; gr < b.ngrp; gr += gridDim.y) {
    const int slot = gr * G + (int)j;
    const unsigned long long w = min(G, b.lay - gr * G);
    if (slot >= b.nsrc) continue;
    const unsigned long long g0 = (unsigned long long)gr * G * n;
    const EndSums sums = end_sums(b, slot);
    unsigned long long acc[kEstPer];
#pragma unroll
    for (int k = 0; k < kEstPer; ++k) {
      const unsigned long long v = v0 + k * (kEstThreads / G);
      acc[k] = v < n ? b.acc[sums.at(end_place(g, walk_id(g, g.wid[v])))] : 0ull;
    }
#pragma unroll
    for (int k = 0; k < kEstPer; ++k) {
      const unsigned long long v = v0 + k * (kEstThreads / G);
      if (v >= n) break;
      // pi_hat = reserve (+ alpha r with zero-hop pruning) + acc * 2^-63 (exact scaling)
      const unsigned long long at = g0 + v * w + j;
      const double res = b.res[at];
      const double base = b.zero_hop ? __dadd_rn(res, __dmul_rn(b.alpha, b.r[at])) : res;
      est[(unsigned long long)slot * n + v] =
          __dadd_rn(base, __dmul_rn(__ull2double_rn(acc[k]), 0x1p-63));
    }
  }
}

constexpr int kTopkThreads = 1024;
constexpr int kTopkLoads = 4;   // elements a thread reads before it uses any

struct TopkRun {
  const double* est;
  int64_t n;
  uint32_t k;
  int32_t* out_ids;
  double* out_vals;
  TopkScratch s;
};

// The first digit: bits of the estimate from kFirstShift on (with the sign), less kFirstBase.
constexpr int kFirstShift = 46;
constexpr uint32_t kFirstBase = 960u << 6;  // 2^-63
__device__ __forceinline__ uint32_t first_bin(double e) {
  const unsigned long long top = (unsigned long long)__double_as_longlong(e) >> kFirstShift;
  if (top < kFirstBase) return 0u;
  return (uint32_t)min(top - kFirstBase, (unsigned long long)(kBins - 1));
}

__device__ __forceinline__ TopkSlot load_slot(const TopkSlot* p) {
  TopkSlot s;
  s.pa = __ldcg(&p->pa);
  s.pb = __ldcg(&p->pb);
  s.plen = __ldcg(&p->plen);
  s.kk = __ldcg(&p->kk);
  s.done = __ldcg(&p->done);
  s.ncand = __ldcg(&p->ncand);
  s.arrived = 0;
  return s;
}

// Elements [beg, end) of part `part` of `parts` of a row of n.
__device__ __forceinline__ void row_range(int64_t n, int part, int parts, int64_t* beg,
                                          int64_t* end) {
  *beg = n * (int64_t)part / parts;
  *end = n * (int64_t)(part + 1) / parts;
}

// Counts one part of a row in sh: the first digit (s == nullptr), else the next digit of the keys
// with s's prefix.  Bin 0 of the first digit
// (zeros and values below 2^-63, most of many rows) is not counted: what is asked of it is the
// keys above the bins.
__device__ void topk_hist(const TopkRun& t, int row, int part, int parts, const TopkSlot* s,
                          uint32_t* sh) {
  int64_t beg, end;
  row_range(t.n, part, parts, &beg, &end);
  const double* e = t.est + (size_t)row * (size_t)t.n;
  const uint32_t width = s ? min((uint32_t)kDigitBits, 96u - s->plen) : 0u;
  const u128 p = s && s->plen ? (((u128)s->pa << 32) | s->pb) >> (96 - s->plen) : 0;
  // block-uniform trip count
  for (int64_t top = beg; top < end; top += (int64_t)blockDim.x * kTopkLoads) {
    const int64_t base = top + threadIdx.x;
    double v[kTopkLoads];
#pragma unroll
    for (int q = 0; q < kTopkLoads; ++q) {
      const int64_t i = base + (int64_t)q * blockDim.x;
      v[q] = i < end ? e[i] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kTopkLoads; ++q) {
      const int64_t i = base + (int64_t)q * blockDim.x;
      if (!s) {
        const uint32_t bin = first_bin(v[q]);
        if (bin) atomicAdd(&sh[bin], 1u);
      } else {
        const u128 z = key_of(v[q], (uint32_t)i);
        const bool in = i < end && (s->plen == 0 || (z >> (96 - s->plen)) == p);
        const unsigned members = __ballot_sync(0xFFFFFFFFu, in);
        if (in) {
          // equal values share every digit but the ids': lanes of one bin add their count once
          const uint32_t bin = (uint32_t)(z >> (96 - s->plen - width)) & ((1u << width) - 1u);
          const unsigned grp = __match_any_sync(members, bin);
          if ((threadIdx.x & 31) == (uint32_t)(__ffs(grp) - 1))
            atomicAdd(&sh[bin], (uint32_t)__popc(grp));
        }
      }
    }
  }
}

// Clears sh; adds it to the row's histogram h.  By the whole block.
__device__ __forceinline__ void topk_clear(uint32_t* sh) {
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) sh[i] = 0;
  __syncthreads();
}
__device__ __forceinline__ void topk_flush(const uint32_t* sh, uint32_t* h) {
  __syncthreads();
  for (int i = threadIdx.x; i < kBins; i += blockDim.x)
    if (sh[i]) atomicAdd(&h[i], sh[i]);
}

// The digit of one row from its histogram (1024 threads; thread th owns bins 4095 - 4 th ..
// 4092 - 4 th, descending), which is cleared for the next.
__device__ void topk_select(const TopkRun& t, int row, bool first) {
  __shared__ uint32_t wsum[32];
  __shared__ uint32_t s_found;
  uint32_t* h = t.s.hist + (size_t)row * kBins;
  TopkSlot s = load_slot(&t.s.slots[row]);
  if (first) s.kk = t.k;
  const int th = threadIdx.x, lane = th & 31, wid = th >> 5;
  uint32_t c[4];
  uint32_t local = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c[q] = __ldcg(&h[kBins - 1 - (4 * th + q)]);
    local += c[q];
  }
  // exclusive scan of `local` over the block (descending bin order)
  uint32_t incl = local;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
    if (lane >= off) incl += v;
  }
  if (th == 0) s_found = 0;
  if (lane == 31) wsum[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const uint32_t a = wsum[lane];
    uint32_t ai = a;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, ai, off);
      if (lane >= off) ai += v;
    }
    wsum[lane] = ai - a;
  }
  __syncthreads();
  uint32_t above = wsum[wid] + incl - local;  // keys in bins above this thread's bins
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int bin = kBins - 1 - (4 * th + q);
    // the clamped bins of the first digit are no prefix
    if (above < s.kk && s.kk <= above + c[q] && !(first && (bin == 0 || bin == kBins - 1))) {
      if (first) {
        s.pa = (unsigned long long)(kFirstBase + (uint32_t)bin) << kFirstShift;
        s.plen = 64 - kFirstShift;
      } else {
        const uint32_t width = min((uint32_t)kDigitBits, 96u - s.plen);
        const u128 p = (((u128)s.pa << 32) | s.pb) | ((u128)(uint32_t)bin << (96 - s.plen - width));
        s.pa = (unsigned long long)(p >> 32);
        s.pb = (uint32_t)p;
        s.plen += width;
      }
      s.kk -= above;
      const uint32_t sure = t.k - s.kk;  // keys strictly above the bucket
      s.done = (sure + c[q] <= kSortCap) || (s.plen >= 96);
      t.s.slots[row] = s;
      s_found = 1;
    }
    above += c[q];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) h[kBins - 1 - (4 * th + q)] = 0;
  __syncthreads();
  if (th == 0 && s_found == 0) t.s.slots[row] = s;  // the k-th key lies outside the first bins
}

// A row's levels: how many have been picked, and of each the parts that blocks have taken and
// finished.  It lies at the start of the row's candidates, which k_topk_collect writes later.
constexpr int kMaxLevels = 8;  // of 12 bits (the last, fewer)
struct LevelWork {
  uint32_t level;
  uint32_t taken[kMaxLevels], done[kMaxLevels];
};
__device__ __forceinline__ LevelWork* level_work(const TopkRun& t, int row) {
  return (LevelWork*)(t.s.cand_key + (size_t)row * kSortCap);
}

// Whether this block is the last of its row's to get here; what the others wrote is then visible.
__device__ bool last_of_row(TopkSlot* slot) {
  __shared__ uint32_t s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&slot->arrived, 1u) == gridDim.x - 1 ? 1u : 0u;
  __syncthreads();
  __threadfence();
  return s_last != 0;
}

// Grid (parts of a row, rows); histograms and slots are zero.
__global__ void __launch_bounds__(kTopkThreads, 2) k_topk_first(TopkRun t) {
  __shared__ uint32_t sh[kBins];
  const int row = blockIdx.y;
  topk_clear(sh);
  topk_hist(t, row, blockIdx.x, gridDim.x, nullptr, sh);
  topk_flush(sh, t.s.hist + (size_t)row * kBins);
  if (!last_of_row(&t.s.slots[row])) return;
  topk_select(t, row, true);
  LevelWork* lw = level_work(t, row);
  for (int i = threadIdx.x; i < (int)(sizeof(LevelWork) / sizeof(uint32_t)); i += blockDim.x)
    ((uint32_t*)lw)[i] = 0;
}

// Grid (parts of a row, rows).  A block takes parts of the row's level until none is left, adds its
// counts, and waits for the blocks that hold the others; the one that finishes the last picks the
// digit, clears the histogram and lets the row go on.  Only parts that a running block has taken
// are waited for, so blocks that have not started hold nobody up, and a block that has waited too
// long can leave: the block that finishes a level takes the next one's parts itself.
constexpr uint32_t kLevelPolls = 1u << 20;
__global__ void __launch_bounds__(kTopkThreads, 2) k_topk_levels(TopkRun t) {
  __shared__ uint32_t sh[kBins];
  __shared__ uint32_t s_x;
  const int row = blockIdx.y;
  if (__ldcg(&t.s.slots[row].done)) return;
  LevelWork* lw = level_work(t, row);
  if (threadIdx.x == 0) s_x = *(volatile uint32_t*)&lw->level;
  __syncthreads();
  for (uint32_t level = s_x; level < (uint32_t)kMaxLevels;) {
    __threadfence();
    // of this level for certain only once a part of it is taken (a level ends with its last part)
    const TopkSlot s = load_slot(&t.s.slots[row]);
    if (__syncthreads_or(s.done != 0)) return;
    topk_clear(sh);
    uint32_t mine = 0;
    for (;;) {
      if (threadIdx.x == 0) s_x = atomicAdd(&lw->taken[level], 1u);
      __syncthreads();
      const uint32_t part = s_x;
      __syncthreads();
      if (part >= gridDim.x) break;
      topk_hist(t, row, (int)part, (int)gridDim.x, &s, sh);
      ++mine;
    }
    bool last = false;
    if (mine) {  // block-uniform
      topk_flush(sh, t.s.hist + (size_t)row * kBins);
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) s_x = atomicAdd(&lw->done[level], mine) + mine;
      __syncthreads();
      last = s_x == gridDim.x;
      __syncthreads();
    }
    if (last) {
      __threadfence();
      topk_select(t, row, false);
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) *(volatile uint32_t*)&lw->level = level + 1;
      ++level;
    } else {
      if (threadIdx.x == 0) {
        uint32_t now, polls = 0;
        while ((now = *(volatile uint32_t*)&lw->level) <= level && ++polls <= kLevelPolls)
          if (polls > 64) __nanosleep(50);
        s_x = now;
      }
      __syncthreads();
      if (s_x <= level) return;
      level = s_x;
      __syncthreads();
    }
  }
}

// Bitonic sort (descending by key) of one row's candidates; writes the first k.
__device__ void topk_sort(const TopkRun& t, int row, unsigned char* smem) {
  unsigned long long* ka = (unsigned long long*)smem;
  uint32_t* kb = (uint32_t*)(ka + kSortCap);
  const uint32_t nc = min(__ldcg(&t.s.slots[row].ncand), kSortCap);
  uint32_t size = 1;
  while (size < nc) size <<= 1;
  for (uint32_t i = threadIdx.x; i < size; i += blockDim.x) {
    if (i < nc) {
      ka[i] = __ldcg(&t.s.cand_key[(size_t)row * kSortCap + i]);
      kb[i] = ~__ldcg(&t.s.cand_id[(size_t)row * kSortCap + i]);
    } else {
      ka[i] = 0;  // below every real key (a real key has ~id > 0)
      kb[i] = 0;
    }
  }
  __syncthreads();
  for (uint32_t len = 2; len <= size; len <<= 1) {
    for (uint32_t j = len >> 1; j > 0; j >>= 1) {
      for (uint32_t q = threadIdx.x; q < size / 2; q += blockDim.x) {
        const uint32_t i = 2 * q - (q & (j - 1)), pr = i + j;  // the q-th pair at distance j
        const bool desc = (i & len) == 0;
        const unsigned long long ai = ka[i], ap = ka[pr];
        const uint32_t bi = kb[i], bp = kb[pr];
        const bool less = ai < ap || (ai == ap && bi < bp);
        const bool more = ai > ap || (ai == ap && bi > bp);
        if (desc ? less : more) {
          ka[i] = ap; ka[pr] = ai;
          kb[i] = bp; kb[pr] = bi;
        }
      }
      __syncthreads();
    }
  }
  for (uint32_t i = threadIdx.x; i < t.k; i += blockDim.x) {
    t.out_ids[(size_t)row * t.k + i] = (int32_t)(~kb[i]);
    t.out_vals[(size_t)row * t.k + i] = __longlong_as_double((long long)ka[i]);
  }
}

// Grid (parts of a row, rows).  A part is read from its end: k_topk_first has read that last.
__global__ void __launch_bounds__(kTopkThreads, 2) k_topk_collect(TopkRun t) {
  extern __shared__ unsigned char smem[];
  const int row = blockIdx.y;
  const unsigned long long pa = __ldcg(&t.s.slots[row].pa);
  const uint32_t pb = __ldcg(&t.s.slots[row].pb);  // (pa, pb): the least key of the prefix
  int64_t beg, end;
  row_range(t.n, blockIdx.x, gridDim.x, &beg, &end);
  const double* e = t.est + (size_t)row * (size_t)t.n;
  const unsigned lane = threadIdx.x & 31;
  // block-uniform trip count, descending
  for (int64_t top = end; top > beg; top -= (int64_t)kTopkThreads * kTopkLoads) {
    double v[kTopkLoads];
#pragma unroll
    for (int q = 0; q < kTopkLoads; ++q) {
      const int64_t i = top - 1 - (int64_t)q * kTopkThreads - threadIdx.x;
      v[q] = i >= beg ? e[i] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kTopkLoads; ++q) {
      const int64_t i = top - 1 - (int64_t)q * kTopkThreads - threadIdx.x;
      const unsigned long long bits = (unsigned long long)__double_as_longlong(v[q]);
      const bool take = i >= beg && (bits > pa || (bits == pa && ~(uint32_t)i >= pb));
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, take);
      if (bal) {
        uint32_t pos = 0;
        if (lane == 0) pos = atomicAdd(&t.s.slots[row].ncand, (uint32_t)__popc(bal));
        pos = __shfl_sync(0xFFFFFFFFu, pos, 0) + __popc(bal & ((1u << lane) - 1u));
        if (take && pos < kSortCap) {
          t.s.cand_key[(size_t)row * kSortCap + pos] = bits;
          t.s.cand_id[(size_t)row * kSortCap + pos] = (uint32_t)i;
        }
      }
    }
  }
  if (last_of_row(&t.s.slots[row])) topk_sort(t, row, smem);
}

}  // namespace

size_t topk_scratch_bytes(int nrows) {
  const size_t r = (size_t)nrows;
  return r * kBins * sizeof(uint32_t) + r * sizeof(TopkSlot) +
         r * kSortCap * (sizeof(unsigned long long) + sizeof(uint32_t)) + 256;
}

TopkScratch topk_scratch_carve(void* base, int nrows) {
  const size_t r = (size_t)nrows;
  TopkScratch s;
  unsigned char* p = (unsigned char*)base;
  s.cand_key = (unsigned long long*)p;  p += r * kSortCap * sizeof(unsigned long long);
  s.slots = (TopkSlot*)p;               p += r * sizeof(TopkSlot);
  s.hist = (uint32_t*)p;                p += r * kBins * sizeof(uint32_t);
  s.cand_id = (uint32_t*)p;
  return s;
}

cudaError_t launch_estimate(const GraphDev& g, const BatchDev& b, double* est, cudaStream_t st) {
  const unsigned per = (unsigned)(kEstValues / b.gw);
  const dim3 grid((unsigned)(((uint64_t)g.n + per - 1) / per), (unsigned)b.ngrp);
  if (b.gw == 1)
    k_estimate<1><<<grid, kEstThreads, 0, st>>>(g, b, est);
  else
    k_estimate<4><<<grid, kEstThreads, 0, st>>>(g, b, est);
  return cudaGetLastError();
}

cudaError_t launch_topk(const double* est, int64_t n, int nrows, uint32_t k, int32_t* out_ids,
                        double* out_vals, const TopkScratch& s, int num_sms, cudaStream_t st) {
  if (nrows <= 0 || k == 0) return cudaSuccess;
  const size_t smem = kSortCap * (sizeof(unsigned long long) + sizeof(uint32_t));
  cudaError_t e = cudaFuncSetAttribute(k_topk_collect, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  // slots and histograms lie side by side
  e = cudaMemsetAsync(s.slots, 0, (size_t)nrows * (sizeof(TopkSlot) + kBins * sizeof(uint32_t)), st);
  if (e != cudaSuccess) return e;
  // Parts of at least 4096 elements: for few rows one wave of two blocks per SM, for more (which
  // might fill half a last wave) about four.
  int64_t bpr = nrows <= 32 ? (int64_t)num_sms * 2 / nrows
                            : ((int64_t)num_sms * 8 + nrows - 1) / nrows;
  bpr = std::max<int64_t>(1, std::min<int64_t>(bpr, (n + 4095) / 4096));
  const dim3 grid((unsigned)bpr, (unsigned)nrows);
  const TopkRun t{est, n, k, out_ids, out_vals, s};
  k_topk_first<<<grid, kTopkThreads, 0, st>>>(t);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // a level's hand-over costs more than a short part's pass, so its parts are of 8192 or more
  const dim3 level_grid((unsigned)std::min<int64_t>(bpr, (n + 8191) / 8192), (unsigned)nrows);
  k_topk_levels<<<level_grid, kTopkThreads, 0, st>>>(t);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_topk_collect<<<grid, kTopkThreads, smem, st>>>(t);
  return cudaGetLastError();
}

}  // namespace fora
