// Learned tau: the FP32 network x(65) -> Linear(65,64) -> GELU -> Linear(64,64)
// -> GELU -> Linear(64,1) -> y = log10(tau / (||A||_F ||B||_F)), with x the
// 64-bin histogram of log2 relative norm products (each bin a fraction of
// all bm * bk * bn triples) followed by log10 of the target relative error.  The
// paper chooses tau by a valid-ratio search (Section 3.5.2); the network
// replaces that search with one forward pass, and plain bisection on the
// achieved error stays the fallback.
//
// Parameters: one flat FP32 array, W1 (64 x 65, row-major out x in), b1,
// W2 (64 x 64), b2, W3 (1 x 64), b3: 8449 values.  GELU is the exact
// 0.5 z (1 + erf(z / sqrt 2)).
//
// Kernels: a batched forward (one thread per sample, weights in shared
// memory), the prediction from a histogram (one CTA per instance), one Adam
// step, and the gradient and the training loop, both on one cluster of up to
// 16 CTAs: every CTA keeps the weights in its shared memory and takes every
// 16th chunk of 16 samples.  In the training loop each CTA sends every other
// its sixteenth of the partial gradient (one bulk copy into that CTA's shared
// memory, completion counted on its mbarrier), sums the sixteen parts of its own
// share in a fixed order, updates those weights (Adam, the moments in registers)
// and sends them to every CTA.  A 256-sample step is 13 MFLOP: on one SM that
// alone is 25 us.  Waits are bounded as in the multiply: one that runs out ends the
// training of every CTA, leaves NaN in all weights and latches SPAMM_ERR_TIMEOUT.
#include <atomic>
#include <cmath>

#include <cooperative_groups.h>

#include "plan.cuh"
#include "tc_common.cuh"

namespace spamm {
namespace mlp {

constexpr int kIn = 65, kH = 64;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH,
              kOffB2 = kOffW2 + kH * kH, kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH;
constexpr int kParams = kOffB3 + 1;   // 8449
static_assert(kParams == 8449, "parameter count");

__device__ __forceinline__ float gelu(float z) {
  return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) +
         z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// y for one sample x[65] with the weights W (shared or global).
__device__ float forward_one(const float* __restrict__ W, const float* __restrict__ x) {
  float h1[kH];
#pragma unroll 4
  for (int o = 0; o < kH; ++o) {
    float z = W[kOffB1 + o];
    for (int i = 0; i < kIn; ++i) z = fmaf(W[kOffW1 + o * kIn + i], x[i], z);
    h1[o] = gelu(z);
  }
  float y = W[kOffB3];
  for (int o = 0; o < kH; ++o) {
    float z = W[kOffB2 + o];
#pragma unroll 8
    for (int i = 0; i < kH; ++i) z = fmaf(W[kOffW2 + o * kH + i], h1[i], z);
    y = fmaf(W[kOffW3 + o], gelu(z), y);
  }
  return y;
}

__global__ void __launch_bounds__(128) forward_kernel(const float* __restrict__ Wg,
                                                      const float* __restrict__ X, int count,
                                                      float* __restrict__ Y) {
  extern __shared__ float W[];
  for (int q = threadIdx.x; q < kParams; q += blockDim.x) W[q] = Wg[q];
  __syncthreads();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= count) return;
  float x[kIn];
  for (int i = 0; i < kIn; ++i) x[i] = X[(int64_t)s * kIn + i];
  Y[s] = forward_one(W, x);
}

// Adam with bias-corrected moments (beta1 0.9, beta2 0.999, eps 1e-8).  Zero moments
// (weights of features that never occur, padding) are kept out of the divisions and
// the square root: a zero operand there takes a slow path, for the whole warp.
__device__ __forceinline__ void adam_update(float& w, float g, float& m, float& v, float lr,
                                            float c1, float c2) {
  m = 0.9f * m + 0.1f * g;
  v = 0.999f * v + 0.001f * g * g;
  const bool m0 = m == 0.0f, v0 = v == 0.0f;
  const float mhat = (m0 ? 1.0f : m) / c1, root = sqrtf((v0 ? 1.0f : v) / c2);
  const float step = lr * mhat / ((v0 ? 0.0f : root) + 1e-8f);
  w -= m0 ? 0.0f * lr : step;   // (an infinite rate gives NaN, as in the formula)
}

__global__ void adam_kernel(float* __restrict__ W, const float* __restrict__ grad,
                            float* __restrict__ m, float* __restrict__ v, int t, float lr) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kParams) return;
  const float c1 = 1.0f - powf(0.9f, (float)t), c2 = 1.0f - powf(0.999f, (float)t);
  float w = W[p], mm = m[p], vv = v[p];
  adam_update(w, grad[p], mm, vv, lr, c1, c2);
  W[p] = w;
  m[p] = mm;
  v[p] = vv;
}

constexpr int kThreads = 512;
constexpr int kChunk = 16;    // samples per chunk: 2 per warp pair
constexpr int kLd = 68;       // row stride in shared memory: 16-byte rows, conflict-free columns

// The parameters as the cluster holds them: padded rows, whole 16-byte groups.  The
// partial gradients and the exchange use the same layout; the padding stays zero,
// but for b3[1], where the gradient carries the loss.
struct Params {
  float w1[kH * kLd], w2[kH * kLd], b1[kH], b2[kH], w3[kH], b3[4];
  float pad[60];              // to equal shares of 16 (or 8) CTAs
};
constexpr int kGroups = sizeof(Params) / 16;                  // float4 groups
constexpr int kLossSlot = 2 * kH * kLd + 3 * kH + 1;
static_assert(sizeof(Params) % (16 * 16) == 0, "equal shares of whole groups");

// Shared memory of one CTA of the gradient cluster.
struct Net {
  Params w, part;             // weights; this CTA's partial gradient
  float x[2][kChunk * kLd];   // the chunk's samples, and the next chunk's on their way
  float h1[kChunk * kLd], h2[kChunk * kLd], g1[kChunk * kLd], g2[kChunk * kLd];
  float y[2][kChunk], g3[kChunk], loss[kThreads / 32], gb3[kThreads / 32], half[4 * kH];
  Params recv;                // this CTA's share of every CTA's partial gradient, by rank
  uint64_t bar[2];            // all shares / all weights have arrived
  int abort_flag;             // a wait of some CTA of the cluster ran out
};

// Status word of the training loop: static, so that a call needs no allocation (it may be
// captured); spamm_last_device_status reads and clears it with the library's own.
static __device__ int32_t g_train_status;

// Place of parameter p (the flat order of the weights) in Params, in floats.
__device__ __forceinline__ int place(int p) {
  constexpr int kW2 = kH * kLd, kB1 = 2 * kH * kLd;
  if (p < kOffB1) return p / kIn * kLd + p % kIn;
  if (p < kOffW2) return kB1 + p - kOffB1;
  if (p < kOffB2) return kW2 + (p - kOffW2) / kH * kLd + (p - kOffW2) % kH;
  return kB1 + kH + p - kOffB2;   // b2, w3, b3 follow each other
}

// Row of this warp's sample of the chunk at c0: -1 past `count`.
__device__ __forceinline__ int sample_row(const int* __restrict__ idx, int c0, int count) {
  const int s = c0 + (int)(threadIdx.x >> 5);
  return s < count ? (idx ? idx[s] : s) : -1;
}

// Starts the copies of a chunk's samples, one row per warp (-1: zeros).
__device__ __forceinline__ void fetch(Net& n, int buf, const float* __restrict__ Xg,
                                      const float* __restrict__ Yg, int row) {
  static_assert(kChunk == kThreads / 32, "a row per warp");
  const int s = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* dst = n.x[buf] + s * kLd;
  if (row >= 0) {
    const float* src = Xg + (int64_t)row * kIn;
    tc::copy4(dst + lane, src + lane);
    tc::copy4(dst + lane + 32, src + lane + 32);
    if (lane == 0) tc::copy4(dst + 64, src + 64);
    if (lane == 1) tc::copy4(&n.y[buf][s], Yg + row);
  } else {
    dst[lane] = 0.0f;
    dst[lane + 32] = 0.0f;
    if (lane == 0) dst[64] = 0.0f;
    if (lane == 1) n.y[buf][s] = 0.0f;
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// A layer's products are cut into tiles of 4 units x 4 samples, the sum of a tile's
// 16 values over eight neighbouring lanes (8 of the 64 terms each): 8 shared-memory
// loads feed 64 FMAs, where a thread per unit and two samples needs 24 and is bound
// by shared memory.  fold leaves each lane two of the values, all eight lanes' terms
// summed in a fixed tree: unit lane / 2 of the tile, samples 2 (lane % 2) and the next.
__device__ __forceinline__ void fold(float (&v)[16], int lane, float (&out)[2]) {
#pragma unroll
  for (int half = 8, bit = 4; half >= 2; half >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int q = 0; q < half; ++q) {
      const float keep = up ? v[q + half] : v[q], send = up ? v[q] : v[q + half];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
  }
  out[0] = v[0];
  out[1] = v[1];
}

// Sums over 64 columns of W's rows u4 .. u4 + 3 times H's rows s4 .. s4 + 3.
__device__ __forceinline__ void layer(const float* __restrict__ W, const float* __restrict__ H,
                                      int lane, float (&out)[2]) {
  float v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = 0.0f;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int k = (lane & 7) * 4 + 32 * i;
    float4 w[4], h[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      w[a] = *reinterpret_cast<const float4*>(W + a * kLd + k);
      h[a] = *reinterpret_cast<const float4*>(H + a * kLd + k);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b)
        v[a * 4 + b] = fmaf(w[a].w, h[b].w,
                            fmaf(w[a].z, h[b].z, fmaf(w[a].y, h[b].y, fmaf(w[a].x, h[b].x, v[a * 4 + b]))));
  }
  fold(v, lane, out);
}

// The same with W's transpose: sums over 64 rows of W's columns u4 .. u4 + 3 (W points at
// the first) times H's rows s4 .. s4 + 3.
__device__ __forceinline__ void layer_t(const float* __restrict__ W, const float* __restrict__ H,
                                        int lane, float (&out)[2]) {
  float v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = (lane & 7) + 8 * i;
    const float4 w = *reinterpret_cast<const float4*>(W + k * kLd);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float h = H[b * kLd + k];
      v[b] = fmaf(w.x, h, v[b]);
      v[4 + b] = fmaf(w.y, h, v[4 + b]);
      v[8 + b] = fmaf(w.z, h, v[8 + b]);
      v[12 + b] = fmaf(w.w, h, v[12 + b]);
    }
  }
  fold(v, lane, out);
}

// acc[4][4] += outer products of four columns of G and of H over the chunk.
__device__ __forceinline__ void outer(const float* __restrict__ G, const float* __restrict__ H,
                                      float (&acc)[4][4]) {
#pragma unroll 8
  for (int s = 0; s < kChunk; ++s) {
    const float4 g = *reinterpret_cast<const float4*>(G + s * kLd);
    const float4 h = *reinterpret_cast<const float4*>(H + s * kLd);
    const float gv[4] = {g.x, g.y, g.z, g.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(gv[a], hv[b], acc[a][b]);
  }
}

// This CTA's share of a gradient: the chunks first, first + stride, ... of `count`
// samples (idx: their rows, or null), divided by norm, into n.part (with the
// loss in part.b3[1]).  The first chunk is in buffer 0 or on its way (fetch);
// then(): called once the last chunk's samples have been read, to fetch the
// next call's first chunk into buffer 0.  Every thread of the CTA calls it.
template <typename Then>
__device__ __forceinline__ void cta_gradient(Net& n, const float* __restrict__ Xg,
                                             const float* __restrict__ Yg,
                                             const int* __restrict__ idx, int count, float norm,
                                             float q, int first, int stride, Then then) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  // this thread's lanes' tile of 4 units x 4 samples, and its own unit and two samples
  const int u4 = ((warp & 7) * 2 + ((lane >> 3) & 1)) * 4, s4 = ((warp >> 3) * 2 + (lane >> 4)) * 4;
  const int o = u4 + ((lane >> 1) & 3), s0 = s4 + (lane & 1) * 2;
  // 4 x 4 entries of d W1 (the lower half of the CTA) or d W2
  const int upper = t >> 8, ty = ((t >> 4) & 15) * 4, tx = (t & 15) * 4;
  // and, over half of the chunk: column 64 of W1, b1, b2, W3 (one unit each)
  const int part = (t >> 6) & 3, pu = t & 63;
  float acc[4][4], ax = 0.0f, ab3 = 0.0f, loss = 0.0f;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
  const int chunks = (count + kChunk - 1) / kChunk;
  int buf = 0;
  for (int c = first; c < chunks; c += stride) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();   // the chunk is here, and the previous one has been read
    if (c + stride < chunks)
      fetch(n, buf ^ 1, Xg, Yg, sample_row(idx, (c + stride) * kChunk, count));
    const float* x = n.x[buf];
    float z1[2], z2[2], g[2];
    layer(n.w.w1 + u4 * kLd, x + s4 * kLd, lane, z1);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      z1[j] += fmaf(n.w.w1[o * kLd + 64], x[(s0 + j) * kLd + 64], n.w.b1[o]);
      n.h1[(s0 + j) * kLd + o] = gelu(z1[j]);
    }
    __syncthreads();
    layer(n.w.w2 + u4 * kLd, n.h1 + s4 * kLd, lane, z2);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      z2[j] += n.w.b2[o];
      n.h2[(s0 + j) * kLd + o] = gelu(z2[j]);
    }
    __syncthreads();
    // output and d loss / d y (pinball slope q for r > 0, q - 1 otherwise): a sample per warp
    {
      const int s = warp;
      float y = fmaf(n.w.w3[lane], n.h2[s * kLd + lane], n.w.w3[lane + 32] * n.h2[s * kLd + lane + 32]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) y += __shfl_xor_sync(0xffffffffu, y, off);
      if (lane == 0) {
        float g = 0.0f;
        if (c * kChunk + s < count) {
          const float r = n.y[buf][s] - (y + n.w.b3[0]);
          g = -(r > 0.0f ? q : q - 1.0f) / norm;
          loss += fmaxf(q * r, (q - 1.0f) * r) / norm;
        }
        n.g3[s] = g;
        ab3 += g;
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 2; ++j)
      n.g2[(s0 + j) * kLd + o] = n.g3[s0 + j] * n.w.w3[o] * gelu_grad(z2[j]);
    __syncthreads();
    layer_t(n.w.w2 + u4, n.g2 + s4 * kLd, lane, g);
#pragma unroll
    for (int j = 0; j < 2; ++j) n.g1[(s0 + j) * kLd + o] = g[j] * gelu_grad(z1[j]);
    __syncthreads();
    outer((upper ? n.g2 : n.g1) + ty, (upper ? n.h1 : x) + tx, acc);
    {
      const float* gs = part < 2 ? n.g1 : (part == 2 ? n.g2 : n.h2);
#pragma unroll
      for (int z = 0; z < kChunk / 2; ++z) {
        const int s = upper * (kChunk / 2) + z;
        const float f = part == 0 ? x[s * kLd + 64] : (part == 3 ? n.g3[s] : 1.0f);
        ax = fmaf(f, gs[s * kLd + pu], ax);
      }
    }
    buf ^= 1;
  }
  if (lane == 0) {
    n.loss[warp] = loss;
    n.gb3[warp] = ab3;
  }
  if (upper) n.half[t & 255] = ax;
  __syncthreads();   // every thread has read the last chunk
  then();
  float* own = (upper ? n.part.w2 : n.part.w1) + ty * kLd + tx;
#pragma unroll
  for (int a = 0; a < 4; ++a)
    *reinterpret_cast<float4*>(own + a * kLd) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
  if (!upper) {
    ax += n.half[t];
    if (part == 0) n.part.w1[pu * kLd + 64] = ax;
    else (part == 1 ? n.part.b1 : (part == 2 ? n.part.b2 : n.part.w3))[pu] = ax;
  } else if (t >= kThreads - 32) {   // the warps' sums of d loss / d y and of the loss
    float sums[2] = {lane < kThreads / 32 ? n.gb3[lane] : 0.0f, lane < kThreads / 32 ? n.loss[lane] : 0.0f};
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      sums[0] += __shfl_xor_sync(0xffffffffu, sums[0], off);
      sums[1] += __shfl_xor_sync(0xffffffffu, sums[1], off);
    }
    if (lane == 0) {
      n.part.b3[0] = sums[0];
      n.part.b3[1] = sums[1];
    }
  }
}

// Groups of each CTA of a cluster of CL: one per thread.
template <int CL>
constexpr int slice() {
  static_assert(kGroups / CL <= kThreads, "a group per thread");
  return kGroups / CL;
}

// Sum of a group's partial values over the cluster, in rank order.
template <int CL>
__device__ __forceinline__ float4 cluster_total(cooperative_groups::cluster_group& cl, Net& n, int g) {
  float4 v[CL];
#pragma unroll
  for (int r = 0; r < CL; ++r) v[r] = *cl.map_shared_rank(reinterpret_cast<float4*>(&n.part) + g, r);
  float4 s = v[0];
#pragma unroll
  for (int r = 1; r < CL; ++r) {
    s.x += v[r].x;
    s.y += v[r].y;
    s.z += v[r].z;
    s.w += v[r].w;
  }
  return s;
}

// Weights into shared memory, the padding of weights and partial gradient cleared.
__device__ __forceinline__ void load_weights(Net& n, const float* __restrict__ Wg) {
  for (int q = threadIdx.x; q < 2 * kGroups; q += kThreads)
    reinterpret_cast<float4*>(&n.w)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  for (int p = threadIdx.x; p < kParams; p += kThreads) reinterpret_cast<float*>(&n.w)[place(p)] = Wg[p];
}

// One cluster: `steps` Adam steps; step s uses the samples idx[s * batch .. (s + 1) *
// batch).  A thread whose wait runs out latches SPAMM_ERR_TIMEOUT in g_train_status and
// raises the abort flag of its CTA and of the others; from then on it neither sends nor
// arrives, and its waits return after a few polls, so that the remaining steps end quickly
// (leaving the loop in its middle, or reading the flag before every send, costs 8 to 12 us
// in 64 steps).  With the flag up, all weights and losses end as NaN, and m and v keep what they held.  WITHHOLD (self-test):
// nothing is sent, so the first wait runs out after limit_ns; elapsed receives the longest
// time a thread of the cluster waited.
// 64 steps of 256 samples: 516 us, 8 us a step.  Of a step's 16 thousand cycles (clock
// stamps in a copy of the kernel) each
// layer takes 1.6 to 2.0 (shared memory and latency), the outer products 2.3 (shared
// memory), Adam 1.2, the two exchanges 5 (35 KB each way per CTA at the ~20 bytes per
// clock of the cluster's network).  Before: one CTA, W2 read with 32-way bank conflicts,
// 15.1 ms; the cluster with a thread per unit and four samples, and the exchange by
// remote loads and stores, 746 us.
template <int CL, bool WITHHOLD>
__global__ void __launch_bounds__(kThreads, 1)
    train_kernel(float* __restrict__ Wg, float* __restrict__ mg, float* __restrict__ vg, int t0,
                 const float* __restrict__ X, const float* __restrict__ Y,
                 const int* __restrict__ idx, int steps, int batch, float lr, float q,
                 float* __restrict__ loss_hist, uint64_t limit_ns, long long* elapsed) {
  extern __shared__ __align__(16) unsigned char smem[];
  Net& n = *reinterpret_cast<Net*>(smem);
  auto cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank(), t = threadIdx.x;
  constexpr int kSlice = slice<CL>();
  constexpr uint32_t kBytes = kSlice * 16;
  const int g = rank * kSlice + t;           // this thread's group
  const bool mine = t < kSlice;
  // a copy per warp: their issue is serial within one (CL: none)
  int to = (t & 31) ? CL : t >> 5;
  if (t == 0) {
    tc::mbar_init(&n.bar[0], 1);
    tc::mbar_init(&n.bar[1], 1);
    n.abort_flag = 0;
    tc::fence_mbarrier_init();
  }
  load_weights(n, Wg);
  // the moments of this thread's group, through the (still unused) partial gradient
  float4 m, v;
  for (int pass = 0; pass < 2; ++pass) {
    __syncthreads();
    for (int p = t; p < kParams; p += kThreads)
      reinterpret_cast<float*>(&n.part)[place(p)] = (pass ? vg : mg)[p];
    __syncthreads();
    const float4 x = mine ? reinterpret_cast<float4*>(&n.part)[g] : make_float4(0.f, 0.f, 0.f, 0.f);
    if (pass) v = x;
    else m = x;
  }
  __syncthreads();
  // the padding of the partial gradient stays zero
  for (int q = t; q < kGroups; q += kThreads)
    reinterpret_cast<float4*>(&n.part)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  fetch(n, 0, X, Y, sample_row(idx, rank * kChunk, batch));
  cl.sync();   // every CTA's barriers are initialised
  uint32_t phase = 0;
  auto wait = [&](uint64_t* bar) {
    if (wait_ab(bar, phase, &n.abort_flag, &g_train_status, WITHHOLD ? limit_ns : kWaitLimitNs)) return;
    if (to < CL) *cl.map_shared_rank(&n.abort_flag, to) = 1;
    to = CL;
  };
  for (int s = 0; s < steps; ++s, phase ^= 1u) {
    const int* now = idx + (int64_t)s * batch;
    const int row = s + 1 < steps ? sample_row(now + batch, rank * kChunk, batch) : -1;
    cta_gradient(n, X, Y, now, batch, (float)batch, q, rank, CL, [&] { fetch(n, 0, X, Y, row); });
    tc::fence_proxy_async_smem();
    __syncthreads();
    // send every CTA its share; a share's place in the receiver is free: it sent the
    // weights this step started from after it had summed the previous shares
    if (t == 0 && to < CL) tc::mbar_arrive_expect_tx(&n.bar[0], CL * kBytes);
    if (!WITHHOLD && to < CL)
      tc::bulk_s2peer(tc::peer_addr(reinterpret_cast<float4*>(&n.recv) + rank * kSlice, to),
                      reinterpret_cast<float4*>(&n.part) + to * kSlice, kBytes,
                      tc::peer_addr(&n.bar[0], to));
    const int step = t0 + s + 1;
    const float c1 = 1.0f - powf(0.9f, (float)step), c2 = 1.0f - powf(0.999f, (float)step);
    const uint64_t since = WITHHOLD ? tc::globaltimer_ns() : 0;
    wait(&n.bar[0]);
    if (WITHHOLD) atomicMax(elapsed, (long long)(tc::globaltimer_ns() - since));
    if (mine) {
      const float4* r4 = reinterpret_cast<const float4*>(&n.recv) + t;
      float4 d = r4[0];
#pragma unroll
      for (int r = 1; r < CL; ++r) {
        const float4 x = r4[r * kSlice];
        d.x += x.x;
        d.y += x.y;
        d.z += x.z;
        d.w += x.w;
      }
      if (g == kLossSlot / 4) {   // b3, the loss beside it
        if (loss_hist) loss_hist[s] = d.y;
        d.y = 0.0f;
      }
      float4 w = reinterpret_cast<float4*>(&n.w)[g];
      adam_update(w.x, d.x, m.x, v.x, lr, c1, c2);
      adam_update(w.y, d.y, m.y, v.y, lr, c1, c2);
      adam_update(w.z, d.z, m.z, v.z, lr, c1, c2);
      adam_update(w.w, d.w, m.w, v.w, lr, c1, c2);
      reinterpret_cast<float4*>(&n.w)[g] = w;
      tc::fence_proxy_async_smem();
    }
    __syncthreads();
    // send the new weights to the others (which have all finished this step's
    // gradient: their shares are here)
    if (t == 0 && to < CL) tc::mbar_arrive_expect_tx(&n.bar[1], (CL - 1) * kBytes);
    if (to < CL && to != rank)
      tc::bulk_s2peer(tc::peer_addr(reinterpret_cast<float4*>(&n.w) + rank * kSlice, to),
                      reinterpret_cast<float4*>(&n.w) + rank * kSlice, kBytes,
                      tc::peer_addr(&n.bar[1], to));
    wait(&n.bar[1]);
  }
  cl.sync();   // no CTA leaves while another sends to it
  if (*const_cast<volatile int*>(&n.abort_flag)) {   // the same in every CTA
    asm volatile("cp.async.wait_all;" ::: "memory");   // the next samples' copies
    // copies sent before the barrier may still be on their way (35 KB in all, microseconds)
    const uint64_t since = tc::globaltimer_ns(), drain = min(limit_ns, kDrainLimitNs);
    while (tc::globaltimer_ns() - since < drain) __nanosleep(1000);
    for (int p = t; p < kParams; p += kThreads)
      if (place(p) / 4 / kSlice == rank) Wg[p] = NAN;
    if (loss_hist && rank == 0)
      for (int s = t; s < steps; s += kThreads) loss_hist[s] = NAN;
    cl.sync();
    return;
  }
  // weights and moments back, each CTA its own groups
  for (int pass = 0; pass < 2; ++pass) {
    __syncthreads();
    if (mine) reinterpret_cast<float4*>(&n.part)[g] = pass ? v : m;
    __syncthreads();
    for (int p = t; p < kParams; p += kThreads) {
      const int at = place(p);
      if (at / 4 / kSlice != rank) continue;
      (pass ? vg : mg)[p] = reinterpret_cast<float*>(&n.part)[at];
      if (!pass) Wg[p] = reinterpret_cast<float*>(&n.w)[at];
    }
  }
}

// One cluster: the gradient and the loss over `count` samples.
template <int CL>
__global__ void __launch_bounds__(kThreads, 1)
    grad_kernel(const float* __restrict__ Wg, const float* __restrict__ X,
                const float* __restrict__ Y, int count, float q, float* __restrict__ grad,
                float* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smem[];
  Net& n = *reinterpret_cast<Net*>(smem);
  auto cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank();
  load_weights(n, Wg);
  fetch(n, 0, X, Y, sample_row(nullptr, rank * kChunk, count));
  __syncthreads();
  cta_gradient(n, X, Y, nullptr, count, (float)count, q, rank, CL, [] {});
  cl.sync();
  // this CTA's groups into its (then unused) weights, from there to the flat order
  for (int l = threadIdx.x; l < slice<CL>(); l += kThreads) {
    const int g = rank * slice<CL>() + l;
    if (g < kGroups) reinterpret_cast<float4*>(&n.w)[g] = cluster_total<CL>(cl, n, g);
  }
  __syncthreads();
  for (int p = threadIdx.x; p < kParams; p += kThreads) {
    const int at = place(p);
    if (at / 4 / slice<CL>() == rank) grad[p] = reinterpret_cast<float*>(&n.w)[at];
  }
  if (threadIdx.x == 0 && kLossSlot / 4 / slice<CL>() == rank) *loss = n.w.b3[1];
  cl.sync();   // no CTA leaves while its shared memory is read
}

// Features of an instance from its histogram and the network's tau: tau = 10^y *
// ||A||_F ||B||_F, target relative error in Inst::target_rel.  One CTA per
// instance, one thread per unit of a layer, every unit's sum in index order (the
// batched forward's order).  Bound by latency: the weights' 34 KB and three
// chains of 64 FMAs; one thread per instance took 88 us, this about 7.
constexpr int kTauThreads = 256;

__global__ void __launch_bounds__(kTauThreads) tau_kernel(InstRef R, const float* __restrict__ Wg,
                                                          float* __restrict__ feats,
                                                          double* __restrict__ tau) {
  extern __shared__ float W[];   // rows of 65 (W2 padded: conflict-free columns)
  __shared__ float x[kIn], h1[kH], h2[kH];
  const int t = threadIdx.x, i = blockIdx.x;
  const Inst& in = R.at(i);
  constexpr int kPadW2 = kOffW2, kPadB2 = kPadW2 + kH * (kH + 1), kShift = kPadB2 - kOffB2;
#pragma unroll 8
  for (int q = t; q < kParams; q += kTauThreads) {
    const float w = Wg[q];
    if (q < kOffW2) W[q] = w;
    else if (q < kOffB2) W[kPadW2 + (q - kOffW2) / kH * (kH + 1) + (q - kOffW2) % kH] = w;
    else W[q + kShift] = w;
  }
  if (t < kHistBins) {
    const double cube = (double)in.bm * (double)in.bk * (double)in.bn;
    x[t] = (float)((double)in.pd->hist[t] / cube);
  } else if (t == kHistBins) {
    x[t] = (float)log10(in.target_rel);
  }
  __syncthreads();
  if (feats && t < kIn) feats[(int64_t)i * kIn + t] = x[t];
  if (t < kH) {
    float z = W[kOffB1 + t];
#pragma unroll 13
    for (int q = 0; q < kIn; ++q) z = fmaf(W[kOffW1 + t * kIn + q], x[q], z);
    h1[t] = gelu(z);
  }
  __syncthreads();
  if (t < kH) {
    float z = W[kPadB2 + t];
#pragma unroll 16
    for (int q = 0; q < kH; ++q) z = fmaf(W[kPadW2 + t * (kH + 1) + q], h1[q], z);
    h2[t] = gelu(z);
  }
  __syncthreads();
  if (t == 0) {
    float y = W[kOffB3 + kShift];
#pragma unroll 16
    for (int q = 0; q < kH; ++q) y = fmaf(W[kOffW3 + kShift + q], h2[q], y);
    tau[i] = exp10((double)y) * (in.pd->norm_a * in.pd->norm_b);
  }
}

// Launches a kernel as one cluster: 16 CTAs where the device can place them (a
// non-portable size), else 8.
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*k16)(KArgs...), void (*k8)(KArgs...), cudaStream_t s,
                           Args... args) {
  static int size[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {16, 1, 1};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sizeof(Net);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  for (auto* k : {k16, k8}) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Net));
    if (e != cudaSuccess) return e;
  }
  if (size[dev] == 0) {
    int fit = 0;
    if (cudaFuncSetAttribute(k16, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&fit, k16, &cfg) != cudaSuccess)
      fit = 0;
    (void)cudaGetLastError();
    size[dev] = fit > 0 ? 16 : 8;
  }
  if (size[dev] == 16) {
    e = cudaFuncSetAttribute(k16, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, k16, args...) : e;
  }
  attr[0].val.clusterDim = {8, 1, 1};
  cfg.gridDim = dim3(8);
  return cudaLaunchKernelEx(&cfg, k8, args...);
}

}  // namespace mlp

namespace {
std::atomic<bool> g_train_ran[64];   // per device: the status word may hold something
}

int mlp_param_count() { return mlp::kParams; }

cudaError_t launch_mlp_forward(const float* W, const float* X, int count, float* Y,
                               cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  const size_t smem = mlp::kParams * sizeof(float);
  cudaFuncSetAttribute(mlp::forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  mlp::forward_kernel<<<(count + 127) / 128, 128, smem, s>>>(W, X, count, Y);
  return cudaPeekAtLastError();
}

cudaError_t launch_mlp_grad(const float* W, const float* X, const float* Y, int count, float q,
                            float* grad, float* loss, cudaStream_t s) {
  return mlp::launch_cluster(mlp::grad_kernel<16>, mlp::grad_kernel<8>, s, W, X, Y, count, q, grad,
                             loss);
}

cudaError_t launch_mlp_adam(float* W, const float* grad, float* m, float* v, int t, float lr,
                            cudaStream_t s) {
  mlp::adam_kernel<<<(mlp::kParams + 255) / 256, 256, 0, s>>>(W, grad, m, v, t, lr);
  return cudaPeekAtLastError();
}

cudaError_t launch_mlp_train(float* W, float* m, float* v, int t0, const float* X, const float* Y,
                             const int* idx, int steps, int batch, float lr, float q,
                             float* loss_hist, cudaStream_t s) {
  if (steps <= 0) return cudaSuccess;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64) g_train_ran[dev].store(true, std::memory_order_relaxed);
  return mlp::launch_cluster(mlp::train_kernel<16, false>, mlp::train_kernel<8, false>, s, W, m, v, t0,
                             X, Y, idx, steps, batch, lr, q, loss_hist, kWaitLimitNs,
                             (long long*)nullptr);
}

cudaError_t mlp_take_status(cudaStream_t s, int32_t* code) {
  *code = 0;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !g_train_ran[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  void* w = nullptr;
  e = cudaGetSymbolAddress(&w, mlp::g_train_status);
  if (e == cudaSuccess) e = cudaMemcpyAsync(code, w, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w, 0, sizeof(int32_t), s);
  return e;
}

namespace {
constexpr int kSelftestSteps = 64;
}

int mlp_wait_selftest_results() { return mlp::kParams + kSelftestSteps; }
int mlp_wait_selftest_floats() {
  return 3 * mlp::kParams + mlp::kIn + 1 + 2 * kSelftestSteps;
}

cudaError_t launch_mlp_wait_selftest(float* buf, uint64_t limit_ns, long long* elapsed,
                                     cudaStream_t s) {
  // steps of one sample each: W, losses, m, v, the sample's features and target, the steps'
  // indexes (all zero)
  cudaError_t e = cudaMemsetAsync(buf, 0, mlp_wait_selftest_floats() * sizeof(float), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(elapsed, 0, sizeof(long long), s);
  int dev = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64) g_train_ran[dev].store(true, std::memory_order_relaxed);
  float *W = buf, *loss = W + mlp::kParams, *m = loss + kSelftestSteps, *v = m + mlp::kParams;
  float *X = v + mlp::kParams, *Y = X + mlp::kIn;
  return mlp::launch_cluster(mlp::train_kernel<16, true>, mlp::train_kernel<8, true>, s, W, m, v, 0, X, Y,
                             reinterpret_cast<const int*>(Y + 1), kSelftestSteps, 1, 1e-3f, 0.5f,
                             loss, limit_ns, elapsed);
}

cudaError_t launch_tau_from_hist(const InstRef& ref, const float* W, float* feats, double* tau,
                                 cudaStream_t s) {
  const size_t smem = (mlp::kParams + mlp::kH) * sizeof(float);
  mlp::tau_kernel<<<ref.count, mlp::kTauThreads, smem, s>>>(ref, W, feats, tau);
  return cudaPeekAtLastError();
}

}  // namespace spamm
