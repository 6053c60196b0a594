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
// 16th chunk of 16 samples; the partial gradients are summed in a fixed order
// through distributed shared memory, each CTA taking 1/16 of the parameters,
// updating them (Adam, the moments in registers) and writing them back to
// every CTA's weights.  A 256-sample step is 13 MFLOP: on one SM that alone is
// 25 us, and the exchange (8449 values per CTA, two cluster barriers) costs
// about 2 us.
#include <cmath>

#include <cooperative_groups.h>

#include "plan.cuh"

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

// Adam with bias-corrected moments (beta1 0.9, beta2 0.999, eps 1e-8).
__device__ __forceinline__ void adam_update(float& w, float g, float& m, float& v, float lr,
                                            float c1, float c2) {
  m = 0.9f * m + 0.1f * g;
  v = 0.999f * v + 0.001f * g * g;
  const float mhat = m / c1, vhat = v / c2;
  w -= lr * mhat / (sqrtf(vhat) + 1e-8f);
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

constexpr int kThreads = 256;
constexpr int kChunk = 16;    // samples per chunk: 4 per warp pair
constexpr int kLd = 68;       // row stride in shared memory: 16-byte rows, conflict-free columns

// Shared memory of one CTA of the gradient cluster.
struct Net {
  float w1[kH * kLd], w2[kH * kLd], b1[kH], b2[kH], w3[kH], b3[4];
  float x[2][kChunk * kLd];   // the chunk's samples, and the next chunk's on their way
  float h1[kChunk * kLd], h2[kChunk * kLd], g1[kChunk * kLd], g2[kChunk * kLd];
  float y[2][kChunk], g3[kChunk], loss[kThreads / 32];
  float part[kParams + 3];    // this CTA's partial gradient, then its partial loss
};

// Shared-memory slot of parameter p (the flat order of the weights).
__device__ __forceinline__ float& weight(Net& n, int p) {
  if (p < kOffB1) return n.w1[p / kIn * kLd + p % kIn];
  if (p < kOffW2) return n.b1[p - kOffB1];
  if (p < kOffB2) return n.w2[(p - kOffW2) / kH * kLd + (p - kOffW2) % kH];
  if (p < kOffW3) return n.b2[p - kOffB2];
  if (p < kOffB3) return n.w3[p - kOffW3];
  return n.b3[0];
}

__device__ __forceinline__ void copy4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

// Starts the copies of the samples c0 .. c0 + kChunk - 1 (zeros past `count`).
__device__ __forceinline__ void fetch(Net& n, int buf, const float* __restrict__ Xg,
                                      const float* __restrict__ Yg, const int* __restrict__ idx,
                                      int c0, int count) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < kChunk / 8; ++q) {   // a warp takes whole rows
    const int s = warp + 8 * q;
    float* dst = n.x[buf] + s * kLd;
    if (c0 + s < count) {
      const int row = idx ? idx[c0 + s] : c0 + s;
      const float* src = Xg + (int64_t)row * kIn;
      copy4(dst + lane, src + lane);
      copy4(dst + lane + 32, src + lane + 32);
      if (lane == 0) copy4(dst + 64, src + 64);
      if (lane == 1) copy4(&n.y[buf][s], Yg + row);
    } else {
      dst[lane] = 0.0f;
      dst[lane + 32] = 0.0f;
      if (lane == 0) dst[64] = 0.0f;
      if (lane == 1) n.y[buf][s] = 0.0f;
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// acc[4][4] += outer products of four columns of G and four of H over the chunk.
__device__ __forceinline__ void outer4(const float* __restrict__ G, const float* __restrict__ H,
                                       float (&acc)[4][4]) {
#pragma unroll 4
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
// loss in part[kParams]).  The first chunk is in buffer 0 or on its way (fetch);
// then(): called once the last chunk's samples have been read, to fetch the
// next call's first chunk into buffer 0.  Every thread of the CTA calls it.
template <typename Then>
__device__ __forceinline__ void cta_gradient(Net& n, const float* __restrict__ Xg,
                                             const float* __restrict__ Yg,
                                             const int* __restrict__ idx, int count, float norm,
                                             float q, int first, int stride, Then then) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int o = (warp & 1) * 32 + lane, s0 = (warp >> 1) * 4;   // one unit, four samples
  const int ty = (t >> 4) * 4, tx = (t & 15) * 4;               // 4 x 4 weights of each matrix
  const int part = t >> 6, pu = t & 63;   // and: column 64 of W1, b1, b2, W3 (one unit each)
  float a1[4][4], a2[4][4], ax = 0.0f, ab3 = 0.0f, loss = 0.0f;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) a1[a][b] = a2[a][b] = 0.0f;
  const int chunks = (count + kChunk - 1) / kChunk;
  int buf = 0;
  for (int c = first; c < chunks; c += stride) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();   // the chunk is here, and the previous one has been read
    if (c + stride < chunks) fetch(n, buf ^ 1, Xg, Yg, idx, (c + stride) * kChunk, count);
    const float* x = n.x[buf];
    float z1[4], z2[4];
    // layer 1
#pragma unroll
    for (int j = 0; j < 4; ++j) z1[j] = n.b1[o];
#pragma unroll 4
    for (int i = 0; i < 64; i += 4) {
      const float4 w = *reinterpret_cast<const float4*>(n.w1 + o * kLd + i);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = *reinterpret_cast<const float4*>(x + (s0 + j) * kLd + i);
        z1[j] = fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, z1[j]))));
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      z1[j] = fmaf(n.w1[o * kLd + 64], x[(s0 + j) * kLd + 64], z1[j]);
      n.h1[(s0 + j) * kLd + o] = gelu(z1[j]);
      z2[j] = n.b2[o];
    }
    __syncthreads();
    // layer 2
#pragma unroll 4
    for (int i = 0; i < kH; i += 4) {
      const float4 w = *reinterpret_cast<const float4*>(n.w2 + o * kLd + i);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = *reinterpret_cast<const float4*>(n.h1 + (s0 + j) * kLd + i);
        z2[j] = fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, z2[j]))));
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) n.h2[(s0 + j) * kLd + o] = gelu(z2[j]);
    __syncthreads();
    // output and d loss / d y (pinball slope q for r > 0, q - 1 otherwise): two samples per warp
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int s = warp * 2 + j;
      float y = fmaf(n.w3[lane], n.h2[s * kLd + lane], n.w3[lane + 32] * n.h2[s * kLd + lane + 32]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) y += __shfl_xor_sync(0xffffffffu, y, off);
      if (lane == 0) {
        float g = 0.0f;
        if (c * kChunk + s < count) {
          const float r = n.y[buf][s] - (y + n.b3[0]);
          g = -(r > 0.0f ? q : q - 1.0f) / norm;
          loss += fmaxf(q * r, (q - 1.0f) * r) / norm;
        }
        n.g3[s] = g;
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j)
      n.g2[(s0 + j) * kLd + o] = n.g3[s0 + j] * n.w3[o] * gelu_grad(z2[j]);
    __syncthreads();
    {
      float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
      for (int j0 = 0; j0 < kH; j0 += 4) {
        float w[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) w[b] = n.w2[(j0 + b) * kLd + o];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 v = *reinterpret_cast<const float4*>(n.g2 + (s0 + j) * kLd + j0);
          g[j] = fmaf(v.w, w[3], fmaf(v.z, w[2], fmaf(v.y, w[1], fmaf(v.x, w[0], g[j]))));
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) n.g1[(s0 + j) * kLd + o] = g[j] * gelu_grad(z1[j]);
    }
    __syncthreads();
    outer4(n.g1 + ty, x + tx, a1);
    outer4(n.g2 + ty, n.h1 + tx, a2);
    {
      const float* g = part < 2 ? n.g1 : (part == 2 ? n.g2 : n.h2);
#pragma unroll 4
      for (int s = 0; s < kChunk; ++s) {
        const float f = part == 0 ? x[s * kLd + 64] : (part == 3 ? n.g3[s] : 1.0f);
        ax = fmaf(f, g[s * kLd + pu], ax);
      }
      if (t == 0)
        for (int s = 0; s < kChunk; ++s) ab3 += n.g3[s];
    }
    buf ^= 1;
  }
  if (lane == 0) n.loss[warp] = loss;
  __syncthreads();   // every thread has read the last chunk
  then();
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      n.part[kOffW1 + (ty + a) * kIn + tx + b] = a1[a][b];
      n.part[kOffW2 + (ty + a) * kH + tx + b] = a2[a][b];
    }
  const int where[4] = {kOffW1 + pu * kIn + 64, kOffB1 + pu, kOffB2 + pu, kOffW3 + pu};
  n.part[where[part]] = ax;
  if (t == 0) {
    n.part[kOffB3] = ab3;
    float l = 0.0f;
    for (int w = 0; w < kThreads / 32; ++w) l += n.loss[w];
    n.part[kParams] = l;
  }
}

// Parameter slots (the loss counts as one) of each CTA of a cluster of CL.
template <int CL>
constexpr int slice() { return (kParams + 1 + CL - 1) / CL; }

// Sum of slot p's partial values over the cluster, in rank order.
template <int CL>
__device__ __forceinline__ float cluster_total(cooperative_groups::cluster_group& cl, Net& n, int p) {
  float v[CL];
#pragma unroll
  for (int r = 0; r < CL; ++r) v[r] = *cl.map_shared_rank(&n.part[p], r);
  float g = v[0];
#pragma unroll
  for (int r = 1; r < CL; ++r) g += v[r];
  return g;
}

// One cluster: `steps` Adam steps; step s uses the samples idx[s * batch .. (s + 1) *
// batch).  Before (one CTA, 32-sample chunks, W2 read with 32-way bank conflicts): 235
// us per 256-sample step; now 11.7 us.
template <int CL>
__global__ void __launch_bounds__(kThreads, 1)
    train_kernel(float* __restrict__ Wg, float* __restrict__ mg, float* __restrict__ vg, int t0,
                 const float* __restrict__ X, const float* __restrict__ Y,
                 const int* __restrict__ idx, int steps, int batch, float lr, float q,
                 float* __restrict__ loss_hist) {
  extern __shared__ __align__(16) unsigned char smem[];
  Net& n = *reinterpret_cast<Net*>(smem);
  auto cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank(), t = threadIdx.x;
  constexpr int kSlice = slice<CL>(), kOwn = (kSlice + kThreads - 1) / kThreads;
  for (int p = t; p < kParams; p += kThreads) weight(n, p) = Wg[p];
  float m[kOwn], v[kOwn];
#pragma unroll
  for (int r = 0; r < kOwn; ++r) {
    const int l = t + r * kThreads, p = rank * kSlice + l;
    const bool mine = l < kSlice && p < kParams;
    m[r] = mine ? mg[p] : 0.0f;
    v[r] = mine ? vg[p] : 0.0f;
  }
  fetch(n, 0, X, Y, idx, rank * kChunk, batch);
  __syncthreads();
  for (int s = 0; s < steps; ++s) {
    cta_gradient(n, X, Y, idx + (int64_t)s * batch, batch, (float)batch, q, rank, CL, [&] {
      if (s + 1 < steps)
        fetch(n, 0, X, Y, idx + (int64_t)(s + 1) * batch, rank * kChunk, batch);
    });
    cl.sync();   // every CTA's partial gradient is there
    const int step = t0 + s + 1;
    const float c1 = 1.0f - powf(0.9f, (float)step), c2 = 1.0f - powf(0.999f, (float)step);
#pragma unroll
    for (int r = 0; r < kOwn; ++r) {
      const int l = t + r * kThreads, p = rank * kSlice + l;
      if (l >= kSlice || p > kParams) continue;
      const float g = cluster_total<CL>(cl, n, p);
      if (p == kParams) {
        if (loss_hist) loss_hist[s] = g;
        continue;
      }
      float w = weight(n, p);
      adam_update(w, g, m[r], v[r], lr, c1, c2);
#pragma unroll
      for (int d = 0; d < CL; ++d) *cl.map_shared_rank(&weight(n, p), d) = w;
    }
    cl.sync();   // the new weights are everywhere, the partial gradients read
  }
#pragma unroll
  for (int r = 0; r < kOwn; ++r) {
    const int l = t + r * kThreads, p = rank * kSlice + l;
    if (l < kSlice && p < kParams) {
      Wg[p] = weight(n, p);
      mg[p] = m[r];
      vg[p] = v[r];
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
  for (int p = threadIdx.x; p < kParams; p += kThreads) weight(n, p) = Wg[p];
  fetch(n, 0, X, Y, nullptr, rank * kChunk, count);
  __syncthreads();
  cta_gradient(n, X, Y, nullptr, count, (float)count, q, rank, CL, [] {});
  cl.sync();
  for (int l = threadIdx.x; l < slice<CL>(); l += kThreads) {
    const int p = rank * slice<CL>() + l;
    if (p > kParams) continue;
    const float g = cluster_total<CL>(cl, n, p);
    if (p == kParams) *loss = g;
    else grad[p] = g;
  }
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
  return mlp::launch_cluster(mlp::train_kernel<16>, mlp::train_kernel<8>, s, W, m, v, t0, X, Y, idx,
                             steps, batch, lr, q, loss_hist);
}

cudaError_t launch_tau_from_hist(const InstRef& ref, const float* W, float* feats, double* tau,
                                 cudaStream_t s) {
  const size_t smem = (mlp::kParams + mlp::kH) * sizeof(float);
  mlp::tau_kernel<<<ref.count, mlp::kTauThreads, smem, s>>>(ref, W, feats, tau);
  return cudaPeekAtLastError();
}

}  // namespace spamm
