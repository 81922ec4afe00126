// Learned r_max: per-source features and a 16-64-64-1 MLP with BF16 weights and
// activations and FP32 accumulation, with hand-written forward, backward and Adam
// kernels.  The network predicts log2(r_max / r_rule) for a source; the query then uses
// r_max = r_rule * 2^prediction.  Any r_max keeps the accuracy guarantee of Lemma
// (layerppr-conc) (omega scales with r_sum), so the network only trades push work
// against walk work, as the balancing of Section 4.2 does with timing.
//
// Parameter vector (FP32 masters, kNumParams floats):
//   W1 [64][16] | b1 [64] | W2 [64][64] | b2 [64] | W3 [64] | b3
// Forward for one sample (every product accumulated in FP32):
//   x  = bf16((f - mu) / sigma)
//   z1 = bf16(W1) x + bf16(b1),  h1 = bf16(relu(z1))
//   z2 = bf16(W2) h1 + bf16(b2), h2 = bf16(relu(z2))
//   y  = bf16(W3) . h2 + bf16(b3)
// Loss 0.5 * mean (y - t)^2; gradients w.r.t. the BF16 weights are applied to the
// FP32 masters (Adam).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fora.h"
#include "fora_engine.cuh"

namespace fora {

namespace {

constexpr int kIn = FORA_NUM_FEATURES;
constexpr int kHid = 64;
constexpr int kOffW1 = 0;
constexpr int kOffB1 = kOffW1 + kHid * kIn;
constexpr int kOffW2 = kOffB1 + kHid;
constexpr int kOffB2 = kOffW2 + kHid * kHid;
constexpr int kOffW3 = kOffB2 + kHid;
constexpr int kOffB3 = kOffW3 + kHid;
constexpr int kNumParams = kOffB3 + 1;
static_assert(kNumParams == FORA_MODEL_PARAMS, "parameter count");
constexpr int kTile = 64;  // samples per block

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ---------------------------------------------------------------- features

// Warp per source.  Sums of integer degrees are exact in FP64.
__global__ void k_features(GraphDev g, const uint32_t* __restrict__ indeg,
                           const int32_t* __restrict__ sources, int nsrc, double alpha,
                           double rmax_rule, float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= nsrc) return;
  const uint32_t s = (uint32_t)sources[w];
  const uint32_t rb = g.row[s], d = g.row[s + 1] - rb;
  const double inc = (1.0 - alpha) / (double)d;  // residue one edge carries in round 1
  double sum_out = 0.0, sum_in = 0.0, f1 = 0.0, f1_edges = 0.0;
  for (uint32_t e = lane; e < d; e += 32) {
    const uint32_t u = (uint32_t)g.col[rb + e];
    const uint32_t du = g.row[u + 1] - g.row[u];
    sum_out += (double)du;
    sum_in += (double)indeg[u];
    if (inc > rmax_rule * (double)du) {
      f1 += 1.0;
      f1_edges += (double)du;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum_out += __shfl_down_sync(0xFFFFFFFFu, sum_out, o);
    sum_in += __shfl_down_sync(0xFFFFFFFFu, sum_in, o);
    f1 += __shfl_down_sync(0xFFFFFFFFu, f1, o);
    f1_edges += __shfl_down_sync(0xFFFFFFFFu, f1_edges, o);
  }
  if (lane == 0) {
    float* f = out + (size_t)w * kIn;
    f[0] = (float)log1p((double)d);
    f[1] = (float)log1p((double)indeg[s]);
    f[2] = (float)log1p(sum_out);
    f[3] = (float)log1p(sum_in);
    f[4] = (float)log1p(f1);
    f[5] = (float)log1p(f1_edges);
    f[6] = (float)log(rmax_rule * (double)g.m);
    f[7] = (float)log((double)g.m / (double)g.n);
    for (int i = 8; i < kIn; ++i) f[i] = 0.0f;
  }
}

__global__ void k_indegree(GraphDev g, uint32_t* indeg) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
       e < (unsigned long long)g.m; e += stride)
    atomicAdd(&indeg[g.col[e]], 1u);
}

// ---------------------------------------------------------------- network

// One tile of kTile samples by one block of kNetThreads threads.  A thread computes 4 x 4 outputs
// of a layer (4 neurons of 4 samples), each as the chain of FMAs over the layer's inputs in
// ascending order; a gradient is the chain over the tile's samples, a parameter per thread and
// step, 4 x 4 of W2's at a time.  So 16 chains are in flight per thread and two 16-byte shared
// loads feed 16 FMAs.  A tile takes about 16 us, bound by latency: 12300 instructions per SM
// partition in 33000 clocks (the FMAs of the three 64 x 64 x 64 products are 6100 clocks of an
// SM, the shared loads 15000).  (With a thread per sample, 64 of 256 busy in the passes over the
// layers and one chain in each, a tile took about 50 us.)
constexpr int kNetThreads = 256;
constexpr int kRow = kHid + 4;  // row of 64 values in shared memory: rows begin 4 banks apart
constexpr int kRowX = kIn + 4;

// BF16-rounded parameters held as floats; W1 with the input index first.
struct NetParams {
  float w1t[kIn][kRow];
  float w2[kHid][kRow];
  float b1[kHid], b2[kHid], w3[kHid];
  float b3;
  float pad[3];
};

struct TileState {
  float x[kTile][kRowX];
  float h1[kTile][kRow], h2[kTile][kRow];  // activations (BF16-rounded)
  float d1[kTile][kRow], d2[kTile][kRow];  // dz1, dz2
  float y[kTile], dy[kTile];
};

__device__ __forceinline__ void put_param(NetParams& np, int p, float v) {
  if (p < kOffB1) {
    np.w1t[(p - kOffW1) % kIn][(p - kOffW1) / kIn] = v;
  } else if (p < kOffW2) {
    np.b1[p - kOffB1] = v;
  } else if (p < kOffB2) {
    np.w2[(p - kOffW2) / kHid][(p - kOffW2) % kHid] = v;
  } else if (p < kOffW3) {
    np.b2[p - kOffB2] = v;
  } else if (p < kOffB3) {
    np.w3[p - kOffW3] = v;
  } else {
    np.b3 = v;
  }
}

__device__ __forceinline__ void load_params(const float* __restrict__ master, NetParams& np) {
  for (int p = threadIdx.x; p < kNumParams; p += kNetThreads) put_param(np, p, bf(master[p]));
}

__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ void st4(float* p, const float* v) {
  *(float4*)p = make_float4(v[0], v[1], v[2], v[3]);
}

__device__ __forceinline__ void fma4(float* acc, float a, const float* c) {
#pragma unroll
  for (int o = 0; o < 4; ++o) acc[o] = __fmaf_rn(c[o], a, acc[o]);
}
__device__ __forceinline__ void unpack(float4 v, float* out) {
  out[0] = v.x;
  out[1] = v.y;
  out[2] = v.z;
  out[3] = v.w;
}

// acc[s][o] += sum over i of w[i][o0 + o] * in[s0 + s][i]: weights with the input index first.
template <int kInputs, int kInRow>
__device__ __forceinline__ void layer_in(const float (*w)[kRow], const float (*in)[kInRow], int o0,
                                         int s0, float (&acc)[4][4]) {
#pragma unroll 4
  for (int i = 0; i < kInputs; i += 4) {
    float a[4][4];
#pragma unroll
    for (int s = 0; s < 4; ++s) unpack(ld4(&in[s0 + s][i]), a[s]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float c[4];
      unpack(ld4(&w[i + q][o0]), c);
#pragma unroll
      for (int s = 0; s < 4; ++s) fma4(acc[s], a[s][q], c);
    }
  }
}

// acc[s][o] += sum over i of w[o0 + 16 o][i] * in[s0 + s][i]: weights with the output index first
// (outputs 16 apart, so that the rows of a warp's loads lie in different banks).
__device__ __forceinline__ void layer_out(const float (*w)[kRow], const float (*in)[kRow], int o0,
                                          int s0, float (&acc)[4][4]) {
#pragma unroll 4
  for (int i = 0; i < kHid; i += 4) {
    float a[4][4], c[4][4];
#pragma unroll
    for (int s = 0; s < 4; ++s) unpack(ld4(&in[s0 + s][i]), a[s]);
#pragma unroll
    for (int o = 0; o < 4; ++o) unpack(ld4(&w[o0 + 16 * o][i]), c[o]);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[s][o] = __fmaf_rn(c[o][q], a[s][q], acc[s][o]);
  }
}

// Thread t's part of a [samples][64] array: samples from sample0(), and outputs from out0() on or
// every 16th from out0s().
__device__ __forceinline__ int out0() { return 4 * (threadIdx.x % 16); }
__device__ __forceinline__ int out0s() { return threadIdx.x % 16; }
__device__ __forceinline__ int sample0() { return 4 * (threadIdx.x / 16); }

// 4 of the 16 inputs of a sample (thread t: sample t / 4, inputs from 4 (t % 4)).
__device__ __forceinline__ float4 load_x(const float* __restrict__ X, int row) {
  return *(const float4*)(X + (size_t)row * kIn + 4 * (threadIdx.x % 4));
}

// Normalised inputs of the tile; zeros from sample cnt on.
__device__ __forceinline__ void put_x(TileState& ts, float4 f, const float* __restrict__ norm,
                                      int cnt) {
  const int s = threadIdx.x / 4, i0 = 4 * (threadIdx.x % 4);
  const float v[4] = {f.x, f.y, f.z, f.w};
  float x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    x[q] = s < cnt ? bf(__fdiv_rn(__fsub_rn(v[q], norm[i0 + q]), norm[kIn + i0 + q])) : 0.0f;
  st4(&ts.x[s][i0], x);
}

// Forward of the tile's cnt samples (activations of the others are 0): y, h1, h2, and the signs
// of this thread's z1 (outputs from out0()) and z2 (every 16th from out0s()): bit 4 s + o.
__device__ __forceinline__ void forward_tile(const NetParams& np, TileState& ts, int cnt,
                                             uint32_t* pos1, uint32_t* pos2) {
  const int o1 = out0(), o2 = out0s(), s0 = sample0();
  float acc[4][4];
#pragma unroll
  for (int s = 0; s < 4; ++s) unpack(ld4(&np.b1[o1]), acc[s]);
  layer_in<kIn, kRowX>(np.w1t, ts.x, o1, s0, acc);
  *pos1 = *pos2 = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    float h[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const bool in = s0 + s < cnt;
      h[o] = in ? bf(fmaxf(acc[s][o], 0.0f)) : 0.0f;
      if (in && acc[s][o] > 0.0f) *pos1 |= 1u << (4 * s + o);
    }
    st4(&ts.h1[s0 + s][o1], h);
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int o = 0; o < 4; ++o) acc[s][o] = np.b2[o2 + 16 * o];
  layer_out(np.w2, ts.h1, o2, s0, acc);
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const bool in = s0 + s < cnt;
      ts.h2[s0 + s][o2 + 16 * o] = in ? bf(fmaxf(acc[s][o], 0.0f)) : 0.0f;
      if (in && acc[s][o] > 0.0f) *pos2 |= 1u << (4 * s + o);
    }
  __syncthreads();
  if (threadIdx.x < kTile) {
    const float* h = ts.h2[threadIdx.x];
    float y = np.b3;
#pragma unroll 4
    for (int i = 0; i < kHid; i += 4) {
      const float4 v = ld4(h + i), w = ld4(&np.w3[i]);
      y = __fmaf_rn(w.x, v.x, y);
      y = __fmaf_rn(w.y, v.y, y);
      y = __fmaf_rn(w.z, v.z, y);
      y = __fmaf_rn(w.w, v.w, y);
    }
    ts.y[threadIdx.x] = y;
  }
}

// Forward and backward of the tile whose inputs are in ts.x: the tile's gradient goes to
// out[kNumParams].  target: this thread's sample's (threads 0 .. cnt - 1); the sample's loss goes
// to *loss.  ts is still being read at the end.
__device__ __forceinline__ void gradient_tile(const NetParams& np, TileState& ts, int cnt,
                                              float target, float inv_batch, float* loss,
                                              float* out) {
  const int t = threadIdx.x, o0 = out0(), s0 = sample0();
  uint32_t pos1, pos2;
  forward_tile(np, ts, cnt, &pos1, &pos2);
  if (t < kTile) {
    float dy = 0.0f;
    if (t < cnt) {
      const float err = __fsub_rn(ts.y[t], target);
      dy = __fmul_rn(err, inv_batch);
      *loss = __fmul_rn(0.5f, __fmul_rn(err, err));
    }
    ts.dy[t] = dy;
  }
  __syncthreads();
  // dz2 = dy * W3 * [z2 > 0]; dz1 = (W2^T dz2) * [z1 > 0]
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const float dy = ts.dy[s0 + s];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const int j = out0s() + 16 * o;
      ts.d2[s0 + s][j] = pos2 >> (4 * s + o) & 1u ? __fmul_rn(dy, np.w3[j]) : 0.0f;
    }
  }
  __syncthreads();
  {
    float acc[4][4] = {};
    layer_in<kHid, kRow>(np.w2, ts.d2, o0, s0, acc);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
#pragma unroll
      for (int o = 0; o < 4; ++o)
        if (!(pos1 >> (4 * s + o) & 1u)) acc[s][o] = 0.0f;
      st4(&ts.d1[s0 + s][o0], acc[s]);
    }
  }
  __syncthreads();
  // gradients summed over the tile, samples in order
  {
    const int j0 = s0, i0 = o0;  // W2[j][i] += dz2[j] h1[i]
    float acc[4][4] = {};
#pragma unroll 4
    for (int b = 0; b < kTile; ++b) {
      float d[4], h[4];
      unpack(ld4(&ts.d2[b][j0]), d);
      unpack(ld4(&ts.h1[b][i0]), h);
#pragma unroll
      for (int j = 0; j < 4; ++j) fma4(acc[j], d[j], h);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) st4(&out[kOffW2 + (j0 + j) * kHid + i0], acc[j]);
  }
  {
    const int j = t / 4, i0 = 4 * (t % 4);  // W1[j][i] += dz1[j] x[i]
    float acc[4] = {};
#pragma unroll 8
    for (int b = 0; b < kTile; ++b) {
      float x[4];
      unpack(ld4(&ts.x[b][i0]), x);
      fma4(acc, ts.d1[b][j], x);
    }
    st4(&out[kOffW1 + j * kIn + i0], acc);
  }
  const int j = t % kHid;
  float a = 0.0f;
  if (t < kHid) {  // b1
#pragma unroll 8
    for (int b = 0; b < kTile; ++b) a = __fadd_rn(a, ts.d1[b][j]);
    out[kOffB1 + j] = a;
  } else if (t < 2 * kHid) {  // b2
#pragma unroll 8
    for (int b = 0; b < kTile; ++b) a = __fadd_rn(a, ts.d2[b][j]);
    out[kOffB2 + j] = a;
  } else if (t < 3 * kHid) {  // W3[j] += dy h2[j]
#pragma unroll 8
    for (int b = 0; b < kTile; ++b) a = __fmaf_rn(ts.dy[b], ts.h2[b][j], a);
    out[kOffW3 + j] = a;
  } else if (j == 0) {  // b3
#pragma unroll 8
    for (int b = 0; b < kTile; ++b) a = __fadd_rn(a, ts.dy[b]);
    out[kOffB3] = a;
  }
}

struct NetShared {
  NetParams np;
  TileState ts;
};

// Block per tile.
__global__ void __launch_bounds__(kNetThreads) k_mlp_forward(const float* __restrict__ master,
                                                             const float* __restrict__ norm,
                                                             const float* __restrict__ X, int n,
                                                             float* __restrict__ Y) {
  extern __shared__ float4 net_smem[];
  NetShared& sh = *(NetShared*)net_smem;
  const int first = blockIdx.x * kTile, cnt = min(kTile, n - first);
  const int s = (int)threadIdx.x / 4;
  const float4 f = s < cnt ? load_x(X, first + s) : make_float4(0, 0, 0, 0);
  load_params(master, sh.np);
  put_x(sh.ts, f, norm, cnt);
  __syncthreads();
  uint32_t pos1, pos2;
  forward_tile(sh.np, sh.ts, cnt, &pos1, &pos2);
  if ((int)threadIdx.x < cnt) Y[first + threadIdx.x] = sh.ts.y[threadIdx.x];
}

// Forward and backward of one tile (rows idx[tile*kTile ...] of X, T) per block; the tile's
// gradient goes to partial[tile] (kPartialStride floats each).
constexpr int kPartialStride = (kNumParams + 3) / 4 * 4;
__global__ void __launch_bounds__(kNetThreads) k_mlp_backward(const float* __restrict__ master,
                                                              const float* __restrict__ norm,
                                                              const float* __restrict__ X,
                                                              const float* __restrict__ T,
                                                              const int32_t* __restrict__ idx,
                                                              int n, float inv_batch,
                                                              float* __restrict__ partial,
                                                              float* __restrict__ loss_partial) {
  extern __shared__ float4 net_smem[];
  NetShared& sh = *(NetShared*)net_smem;
  const int first = blockIdx.x * kTile, cnt = min(kTile, n - first);
  const int t = threadIdx.x, s = t / 4;
  float4 f = make_float4(0, 0, 0, 0);
  float target = 0.0f;
  if (s < cnt) f = load_x(X, idx ? idx[first + s] : first + s);
  if (t < cnt) target = T[idx ? idx[first + t] : first + t];
  load_params(master, sh.np);
  put_x(sh.ts, f, norm, cnt);
  __syncthreads();
  gradient_tile(sh.np, sh.ts, cnt, target, inv_batch, &loss_partial[first + t],
                partial + (size_t)blockIdx.x * kPartialStride);
}

// grad[p] = sum over tiles (in tile order) of partial[tile][p]
__global__ void k_mlp_reduce(const float* __restrict__ partial, int tiles, float* __restrict__ grad) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kNumParams) return;
  float a = 0.0f;
  for (int t = 0; t < tiles; ++t) a = __fadd_rn(a, partial[(size_t)t * kPartialStride + p]);
  grad[p] = a;
}

// Adam on one parameter; c1, c2: 1 - b1^step, 1 - b2^step.
struct AdamStep {
  float lr, b1, b2, eps;
};
__device__ __forceinline__ void adam_one(const AdamStep& a, float c1, float c2, float gr,
                                         float* master, float* m, float* v) {
  const float mp = __fmaf_rn(1.0f - a.b1, gr, __fmul_rn(a.b1, *m));
  const float vp = __fmaf_rn(__fmul_rn(1.0f - a.b2, gr), gr, __fmul_rn(a.b2, *v));
  *m = mp;
  *v = vp;
  *master -= a.lr * (mp / c1) / (sqrtf(vp / c2) + a.eps);
}

__global__ void k_adam(float* __restrict__ master, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ grad, AdamStep a, float c1, float c2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kNumParams) return;
  adam_one(a, c1, c2, grad[p], &master[p], &m[p], &v[p]);
}

// An epoch in one launch, for batches of up to kMaxCluster tiles: a cluster with a block per tile.
// The parameters stay in shared memory (each block has all of them, and the masters and moments
// of every ntiles-th).  A step: each block its tile's gradient, the cluster meets, each block adds
// the tiles' partial sums (in tile order) of the parameters it keeps, steps them and writes the
// rounded values to every block, the cluster meets.  Bound by the chain of a step, of which the
// tile's gradient is most; the next step's inputs are on their way meanwhile.  A step of 256
// samples takes 18 us (three launches of one tile per block: 34 us); 10000 samples, 2 epochs of
// batches of 256: 5.03 -> 2.02 ms, with the same bits.
constexpr int kMaxCluster = 8;
constexpr int kAdamPer = 6;  // 5313 parameters over 4 blocks of 256 threads
struct TrainShared {
  NetShared net;
  float part[kPartialStride];
  float master[kNumParams], m[kNumParams], v[kNumParams];  // first kNumParams / ntiles used
};
struct TrainArgs {
  float *master, *m, *v;
  const float *norm, *X, *T;
  const int32_t* idx;  // [n] the epoch's order
  const float2* c;     // [steps] Adam's (c1, c2)
  int n, batch;
  AdamStep adam;
  float* loss;  // [n]
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_meet() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The generic address of p's counterpart in block `rank` of the cluster.
template <typename V>
__device__ __forceinline__ V* peer(V* p, uint32_t rank) {
  unsigned long long out;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"((unsigned long long)p), "r"(rank));
  return (V*)out;
}

__global__ void __launch_bounds__(kNetThreads, 1) k_mlp_train(const __grid_constant__ TrainArgs a) {
  extern __shared__ float4 net_smem[];
  TrainShared& sh = *(TrainShared*)net_smem;
  const int t = threadIdx.x, s = t / 4;
  const int rank = (int)cluster_rank(), nblk = (int)gridDim.x;  // one cluster
  // parameter p is kept by block p % nblk, at p / nblk
  for (int p = rank + nblk * t, k = t; p < kNumParams; p += nblk * kNetThreads, k += kNetThreads) {
    sh.master[k] = a.master[p];
    sh.m[k] = a.m[p];
    sh.v[k] = a.v[p];
  }
  load_params(a.master, sh.net.np);
  // The rows of this thread's inputs (x) and target (t) of the batch at off: -1 where it has none.
  struct Rows {
    int x, t;
  };
  auto rows = [&](int off) {
    const int first = off + rank * kTile;
    const int cnt = min(min(kTile, a.batch - rank * kTile), a.n - first);
    return Rows{s < cnt ? a.idx[first + s] : -1, t < cnt ? a.idx[first + t] : -1};
  };
  auto inputs = [&](const Rows& r, float4* f, float* target) {
    *f = r.x >= 0 ? load_x(a.X, r.x) : make_float4(0, 0, 0, 0);
    *target = r.t >= 0 ? a.T[r.t] : 0.0f;
  };
  float4 f;
  float target;
  inputs(rows(0), &f, &target);
  Rows next = rows(a.batch);
  for (int off = 0, step = 0; off < a.n; off += a.batch, ++step) {
    const int size = min(a.batch, a.n - off), tiles = (size + kTile - 1) / kTile;
    const int cnt = min(kTile, size - rank * kTile);
    const float2 c = a.c[step];
    // what the next steps need is on its way meanwhile: inputs, and the rows of the step after
    float4 next_f;
    float next_target;
    inputs(next, &next_f, &next_target);
    next = rows(off + 2 * a.batch);
    if (rank < tiles) {
      put_x(sh.net.ts, f, a.norm, cnt);
      __syncthreads();
      gradient_tile(sh.net.np, sh.net.ts, cnt, target, 1.0f / (float)size,
                    &a.loss[off + rank * kTile + t], sh.part);
    }
    cluster_meet();
    // kAdamPer parameters of a thread at a time, so that the reads of other blocks overlap
    const int mine = (kNumParams - rank + nblk - 1) / nblk;  // parameters kept here
    for (int k0 = t; k0 < mine; k0 += kNetThreads * kAdamPer) {
      float g[kAdamPer] = {};
      for (int b = 0; b < tiles; ++b) {
        const float* part = peer(sh.part, b);
#pragma unroll
        for (int q = 0; q < kAdamPer; ++q) {
          const int k = k0 + q * kNetThreads;
          if (k < mine) g[q] = __fadd_rn(g[q], part[rank + nblk * k]);
        }
      }
#pragma unroll
      for (int q = 0; q < kAdamPer; ++q) {
        const int k = k0 + q * kNetThreads;
        if (k >= mine) break;
        adam_one(a.adam, c.x, c.y, g[q], &sh.master[k], &sh.m[k], &sh.v[k]);
        const float w = bf(sh.master[k]);
        for (int b = 0; b < nblk; ++b) put_param(*peer(&sh.net.np, b), rank + nblk * k, w);
      }
    }
    cluster_meet();
    f = next_f;
    target = next_target;
  }
  for (int p = rank + nblk * t, k = t; p < kNumParams; p += nblk * kNetThreads, k += kNetThreads) {
    a.master[p] = sh.master[k];
    a.m[p] = sh.m[k];
    a.v[p] = sh.v[k];
  }
}

__global__ void k_pred_to_rmax(const float* __restrict__ pred, int n, double rmax_rule, float lo,
                               float hi, double* __restrict__ rmax) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float p = fminf(fmaxf(pred[i], lo), hi);
  rmax[i] = rmax_rule * exp2((double)p);
}

constexpr float kBeta1 = 0.9f, kBeta2 = 0.999f, kAdamEps = 1e-8f;

template <typename K>
cudaError_t allow_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

cudaError_t launch_indegree(const GraphDev& g, uint32_t* indeg, int num_sms, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(indeg, 0, (size_t)g.n * sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  k_indegree<<<num_sms * 8, 256, 0, st>>>(g, indeg);
  return cudaGetLastError();
}

cudaError_t launch_features(const GraphDev& g, const uint32_t* indeg, const int32_t* sources,
                            int nsrc, double alpha, double rmax_rule, float* out, cudaStream_t st) {
  if (nsrc <= 0) return cudaSuccess;
  const int warps_per_block = 8;
  k_features<<<(nsrc + warps_per_block - 1) / warps_per_block, 32 * warps_per_block, 0, st>>>(
      g, indeg, sources, nsrc, alpha, rmax_rule, out);
  return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const float* master, const float* norm, const float* X, int n,
                               float* Y, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const cudaError_t e = allow_smem(k_mlp_forward, sizeof(NetShared));
  if (e != cudaSuccess) return e;
  k_mlp_forward<<<(n + kTile - 1) / kTile, kNetThreads, sizeof(NetShared), st>>>(master, norm, X, n,
                                                                               Y);
  return cudaGetLastError();
}

cudaError_t launch_mlp_grad(const float* master, const float* norm, const float* X,
                            const float* T, const int32_t* idx, int n, float* partial,
                            float* loss_partial, float* grad, cudaStream_t st) {
  cudaError_t e = allow_smem(k_mlp_backward, sizeof(NetShared));
  if (e != cudaSuccess) return e;
  const int tiles = (n + kTile - 1) / kTile;
  k_mlp_backward<<<tiles, kNetThreads, sizeof(NetShared), st>>>(
      master, norm, X, T, idx, n, 1.0f / (float)n, partial, loss_partial);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_mlp_reduce<<<(kNumParams + 255) / 256, 256, 0, st>>>(partial, tiles, grad);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* master, float* m, float* v, const float* grad, int step, float lr,
                        cudaStream_t st) {
  const float2 c = adam_correction(step);
  k_adam<<<(kNumParams + 255) / 256, 256, 0, st>>>(master, m, v, grad,
                                                   AdamStep{lr, kBeta1, kBeta2, kAdamEps}, c.x, c.y);
  return cudaGetLastError();
}

float2 adam_correction(int step) {
  return make_float2(1.0f - powf(kBeta1, (float)step), 1.0f - powf(kBeta2, (float)step));
}

// A cluster takes one tile per block, so larger batches go step by step.
bool mlp_train_fits(int batch) { return batch <= kMaxCluster * kTile; }

cudaError_t launch_mlp_epoch(float* master, float* m, float* v, const float* norm, const float* X,
                             const float* T, const int32_t* idx, const float2* corrections, int n,
                             int batch, float lr, float* loss, cudaStream_t st) {
  cudaError_t e = allow_smem(k_mlp_train, sizeof(TrainShared));
  if (e != cudaSuccess) return e;
  const unsigned tiles = (unsigned)((std::min(batch, n) + kTile - 1) / kTile);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = tiles;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles);
  cfg.blockDim = dim3(kNetThreads);
  cfg.dynamicSmemBytes = sizeof(TrainShared);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const TrainArgs a{master, m, v, norm, X, T, idx, corrections, n, batch,
                    AdamStep{lr, kBeta1, kBeta2, kAdamEps}, loss};
  return cudaLaunchKernelEx(&cfg, k_mlp_train, a);
}

cudaError_t launch_pred_to_rmax(const float* pred, int n, double rmax_rule, float lo, float hi,
                                double* rmax, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_pred_to_rmax<<<(n + 255) / 256, 256, 0, st>>>(pred, n, rmax_rule, lo, hi, rmax);
  return cudaGetLastError();
}

size_t mlp_partial_floats(int n) { return (size_t)((n + kTile - 1) / kTile) * kPartialStride; }

}  // namespace fora
