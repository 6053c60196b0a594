// Plain FP32 multiply on the SIMT cores (Section 3.3's FP32 multiplication
// kernel; the baseline the tensor-core modes are measured against).
//
// One persistent CTA per SM holds several independent groups of warps; a group
// multiplies one tile at a time: 1 warp at leaf 32, 2 at 64, 8 at 128, and 4 at leaf 32
// and 64 where there are few tiles (kWideTiles).  The
// non-empty tiles of all instances (most survivors first) are dealt over the SMs
// with a fixed stride; inside an SM its groups take them from a shared-memory
// counter, so a group that met short tiles takes more of them (a fixed deal to
// every group left a third of the warps idle on average).  A warp owns 32 x 64
// entries of the tile (32 x 32 at leaf 32), a thread 8 rows x 8 (4) columns: rows
// ty + 4 u, columns 4 tx .. 4 tx + 3 and 32 further on, so that the distinct
// addresses of every shared-memory read fall into different banks.
// The surviving k are streamed in slices of the inner dimension through a ring of
// stages filled by asynchronous copies (16 bytes where rows are
// aligned, else 4; entries outside the matrix are filled with zeros), A as rows,
// B as rows: neither is transposed.  The products accumulate in FP32 FMA over the
// surviving k in increasing order, two columns per instruction (packed
// fma.rn.f32x2: the same FP32 rate, half the issue slots).  Bound by the FP32 pipe
// on dense skip sets: 48, 49 and 44 TFLOP/s at leaf 32, 64 and 128 (n = 4096,
// 30% of the triples; 256 threads per tile with transposed A slices: 19, 30 and
// 29), 42 at leaf 64 with unaligned rows (26).  Slices of 32 in two stages instead of
// 16 in three give 45 -> 48 and 42 -> 44 at leaf 32 and 128; at leaf 64 49 -> 52, but
// lists of 2 to 3 blocks become 6% slower (the first slice is all that a tile has on its
// way at its start), so it keeps 16.
#include <algorithm>

#include "tc_common.cuh"

namespace spamm {
namespace {

// Outputs up to this size: the multiply writes the empty tiles itself.  A second kernel
// beside it (on a side stream) costs two events and a launch, but its stores overlap the
// multiply's latency.  Product on exponential decay (nearly all tiles empty), second
// kernel -> own stores: at 4 MB 21.0 -> 19.4, 27.1 -> 23.9 and 53.8 -> 50.7 us at leaf 32, 64
// and 128; at 31 MB 33.0 -> 30.0, 33.2 -> 28.6, 55.8 -> 57.7; at 64 MB 45.7 -> 45.2, 41.3 ->
// 34.8, 57.8 -> 64.6; at 127 MB 63.3 -> 87.6, 58.5 -> 56.9, 77.7 -> 95.9 (16 MB, leaf 128:
// 53.8 -> 52.1).  Leaf 128 has the fewest warps to store with.  Against a second kernel
// behind the multiply, in the same stream, own stores win at leaf 128 too (product without
// allocation, 64 MB: 123 -> 117 us).
constexpr int64_t own_zero_bytes(int leaf, bool beside) {
  return (int64_t)(leaf == 128 && beside ? 24 : 64) << 20;
}

// Up to this many non-empty tiles per SM, four warps share a tile, in three groups with a
// longer ring: with one or two warps per tile the other schedulers of an SM would idle
// through its list.  One tile per SM, lists of 256 blocks at leaf 32: 325 -> 217 us (256
// threads per tile, one group: 298), of 128 at leaf 64: 451 -> 301 (417); 32 tiles of 1024
// blocks at leaf 32: 954 -> 523 (848), 8 of 256 at leaf 64: 895 -> 590 (822).  Two per SM
// 254 -> 192 and 499 -> 496; three 263 -> 287 at leaf 32, and at leaf 64 757 -> 629 with
// equal lists, but the selection of tau (uneven ones) 800 -> 812: hence the limit.  With
// many empty tiles to write beside them the idle warps are not idle: only up to one tile per
// SM then (two per SM, 23 empty ones each, short lists at leaf 32: product 31.1 -> 33.5 us; one
// per SM at leaf 64, five empty ones: 39.2 -> 35.2).  The sums are in the same order in
// both forms.
constexpr int kWideTiles = 2;

// How a CTA is cut into groups of warps, a group's tile into warps and a warp's part
// into threads: thread (ty, tx) of a warp has the rows ty + kTy u (u < TM) and the columns
// 4 tx .. 4 tx + 3 and 4 kTx further on.
template <int LEAF_, bool WIDE>
struct SimtTile {
  static_assert(!WIDE || LEAF_ < 128, "leaf 128: one form");
  static constexpr int LEAF = LEAF_;
  static constexpr int kWarps = WIDE ? 4 : (LEAF == 128 ? 8 : (LEAF == 64 ? 2 : 1));
  static constexpr int kThreads = 32 * kWarps;
  // groups per CTA, one CTA per SM: 168 registers per thread at leaf 32 and 64 (8 and 16
  // groups at 128 registers spill: 37 and 42 TFLOP/s against 48 and 45)
  static constexpr int kGroups = WIDE ? 3 : (LEAF == 128 ? 1 : (LEAF == 64 ? 6 : 12));
  // slices of the inner dimension, stages of the ring
  static constexpr int kSlice = LEAF == 64 ? 16 : 32;
  static constexpr int kStages = (LEAF == 64 ? 3 : 2) * (WIDE ? 12 / (kGroups * (LEAF == 64 ? 2 : 1)) : 1);
  static constexpr int kLdA = kSlice + 4;   // floats per staged row of A: 16-byte rows, kTy
                                            // rows in different banks
  static constexpr bool kSmall = WIDE && LEAF == 32;   // 2 x 4 entries per thread
  static constexpr int kTy = kSmall ? 8 : 4, kTx = 32 / kTy;
  static constexpr int TM = kSmall ? 2 : 8;                          // rows per thread
  static constexpr int TN = LEAF == 32 || WIDE ? 4 : 8;              // columns per thread
  static constexpr int kWarpRows = kTy * TM, kWarpCols = kTx * TN;
  static_assert(kWarps * kWarpRows * kWarpCols == LEAF * LEAF, "the warps cover the tile");
  static constexpr int kStageFloats = LEAF * kLdA + kSlice * LEAF;   // A rows, then B rows
  static constexpr size_t kSmem = (size_t)kStages * kStageFloats * sizeof(float);
  static constexpr int kCtaThreads = kGroups * kThreads;
  static constexpr size_t kCtaSmem = kGroups * kSmem;
  static_assert(kCtaSmem <= 227 * 1024 && kCtaThreads <= 1024 && kGroups <= 15, "CTA shape");
};

// Stages rows [r, r + ROWS) x columns [c, c + COLS) of a rows x cols matrix with
// leading dimension ld as ROWS rows of LD floats.
template <int ROWS, int COLS, int LD, int THREADS>
__device__ __forceinline__ void stage(float* dst, const float* __restrict__ M, int64_t rows,
                                      int64_t cols, int64_t ld, int64_t r, int64_t c, bool vec) {
  constexpr int kPerRow = COLS / 4;
  const int tid = threadIdx.x % THREADS;
  if (vec) {
#pragma unroll
    for (int l = 0; l < ROWS * kPerRow / THREADS; ++l) {
      const int p = tid + l * THREADS, pr = p / kPerRow, pc = p % kPerRow * 4;
      const int64_t left = r + pr < rows ? cols - (c + pc) : 0;
      const int bytes = left >= 4 ? 16 : (left > 0 ? (int)left * 4 : 0);
      tc::copy16(dst + pr * LD + pc, bytes ? M + (r + pr) * ld + c + pc : M, bytes);
    }
  } else {
#pragma unroll 4
    for (int l = 0; l < ROWS * COLS / THREADS; ++l) {
      const int p = tid + l * THREADS, pr = p / COLS, pc = p % COLS;
      const bool in = r + pr < rows && c + pc < cols;
      tc::copy4(dst + pr * LD + pc, in ? M + (r + pr) * ld + c + pc : M, in ? 4 : 0);
    }
  }
}

// Two FP32 FMAs, each rounded to nearest.
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t pair(float x, float y) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ void unpair(uint64_t d, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(d));
}

// The barrier of one group (hardware barrier 1 + group).
template <class T>
__device__ __forceinline__ void tile_sync(int group) {
  if constexpr (T::kWarps == 1)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(T::kThreads) : "memory");
}

// An empty tile of an instance with beta = 0: zeros, and the tile's norm; by kThreads threads.
template <int LEAF, int kThreads>
__device__ __forceinline__ void zero_tile(const Inst& in, int64_t t, int tid) {
  const int i = (int)(t / in.bn), j = (int)(t - (int64_t)i * in.bn);
  const int64_t r0 = (int64_t)i * LEAF, c0 = (int64_t)j * LEAF;
  const int rows = (int)min((int64_t)LEAF, in.m - r0), cols = (int)min((int64_t)LEAF, in.n - c0);
  float* p = in.C + r0 * in.ldc + c0;
  if ((in.ldc & 3) == 0 && (cols & 3) == 0) {
    constexpr int kPerRow = LEAF / 4;
    for (int x = tid; x < rows * kPerRow; x += kThreads) {
      const int r = x / kPerRow, c = x % kPerRow * 4;
      if (c < cols)
        *reinterpret_cast<float4*>(p + r * in.ldc + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  } else {
    for (int x = tid; x < rows * LEAF; x += kThreads)
      if (x % LEAF < cols) p[x / LEAF * in.ldc + x % LEAF] = 0.0f;
  }
  if (in.nC && tid == 0) in.nC[t] = 0.0;
}

// The groups of one CTA multiply their tiles; zeros: they also write the tiles without
// survivors (every instance has beta = 0).
template <class T>
__device__ __forceinline__ void multiply_tiles(const InstRef& R, const PlanBuffers& Bf, int64_t ne,
                                               int dynamic, int zeros, int* s_taken, int* s_next,
                                               SumSq* s_norm, const int thread) {
  extern __shared__ __align__(16) float smem_all[];
  constexpr int LEAF = T::LEAF, TM = T::TM, TN = T::TN, kHalves = TN / 4;
  constexpr int kSlice = T::kSlice, kStages = T::kStages, kLdA = T::kLdA, kTy = T::kTy, kTx = T::kTx;
  const int group = thread / T::kThreads, tid = thread % T::kThreads;
  const int warp = tid >> 5, lane = tid & 31;
  const int tx = lane % kTx, ty = lane / kTx;
  constexpr int kWarpsAcross = LEAF / T::kWarpCols;
  const int wr = warp / kWarpsAcross * T::kWarpRows, wc = warp % kWarpsAcross * T::kWarpCols;
  float* smem = smem_all + (size_t)group * kStages * T::kStageFloats;
  const int all = (int)(zeros ? Bf.tiles : ne);

  for (bool first = true;; first = false) {
    // dynamic: from the table's counter (it hands out non-empty tiles only); else a group's
    // first tile is its own, so that few tiles fall on warps of different schedulers
    if (tid == 0)
      s_next[group] = dynamic ? atomicAdd(&Bf.bdev->mul_ticket, 1)
                              : (first ? group : T::kGroups + atomicAdd(s_taken, 1));
    tile_sync<T>(group);   // also: the previous tile's readers are done with the ring
    const int64_t w = dynamic ? s_next[group] : blockIdx.x + (int64_t)s_next[group] * gridDim.x;
    if (w >= (dynamic ? ne : all)) break;
    const int g = Bf.order[w];
    const Inst& in = R.at(inst_of(R, Bf, g));
    if (w >= ne) {
      zero_tile<LEAF, T::kThreads>(in, g - in.tile0, tid);
      tile_sync<T>(group);   // s_next is rewritten next
      continue;
    }
    const int beg = Bf.tile_beg[g], cnt = Bf.cnt[g];
    const int bn = in.bn;
    const int64_t m = in.m, kd = in.kd, n = in.n;
    const int64_t lda = in.lda, ldb = in.ldb, ldc = in.ldc;
    const float* __restrict__ A = in.A;
    const float* __restrict__ B = in.B;
    float* __restrict__ C = in.C;
    const bool vec_a = (lda % 4) == 0, vec_b = (ldb % 4) == 0, vec_c = (ldc % 4) == 0;
    const uint16_t* __restrict__ k_idx = Bf.k_idx + beg;
    const int64_t t = g - in.tile0;
    const int i = (int)(t / bn), j = (int)(t % bn);
    const int64_t r0 = (int64_t)i * LEAF, c0 = (int64_t)j * LEAF;

    uint64_t acc[TM][TN / 2];
#pragma unroll
    for (int u = 0; u < TM; ++u)
#pragma unroll
      for (int v = 0; v < TN / 2; ++v) acc[u][v] = 0ull;

    constexpr int kPerK = LEAF / kSlice;
    const int nslices = cnt * kPerK;
    int k_ahead = __ldg(k_idx) & 0x3ff;   // the inner block of the next slice to stage
    // a tile inside the matrix: this thread's pieces (or entries) of a slice start at
    // fixed distances from two pointers
    const bool inside = r0 + LEAF <= m && c0 + LEAF <= n;
    constexpr int kThr = T::kThreads, kPc = kSlice / 4, kPl = LEAF / 4;
    const int pa = vec_a ? tid / kPc : tid / kSlice, ca = vec_a ? tid % kPc * 4 : tid % kSlice;
    const int pb = vec_b ? tid / kPl : tid / LEAF, cb = vec_b ? tid % kPl * 4 : tid % LEAF;
    const float* base_a = A + (r0 + pa) * lda + ca;
    const float* base_b = B + (int64_t)pb * ldb + c0 + cb;
    auto fetch = [&](int q) {
      if (q < nslices) {
        const int64_t k0 = (int64_t)k_ahead * LEAF + (q % kPerK) * kSlice;
        float* s = smem + (q % kStages) * T::kStageFloats;
        float* sb = s + LEAF * kLdA;
        if (inside && k0 + kSlice <= kd) {
          const float* src = base_a + k0;
          if (vec_a) {
            constexpr int kStep = kThr / kPc;
#pragma unroll
            for (int l = 0; l < LEAF / kStep; ++l, src += kStep * lda)
              tc::copy16(s + (pa + l * kStep) * kLdA + ca, src, 16);
          } else {
            constexpr int kStep = kThr / kSlice;
#pragma unroll 8
            for (int l = 0; l < LEAF / kStep; ++l, src += kStep * lda)
              tc::copy4(s + (pa + l * kStep) * kLdA + ca, src, 4);
          }
          src = base_b + k0 * ldb;
          if (vec_b) {
            constexpr int kStep = kThr / kPl;
#pragma unroll
            for (int l = 0; l < kSlice / kStep; ++l, src += kStep * ldb)
              tc::copy16(sb + (pb + l * kStep) * LEAF + cb, src, 16);
          } else {
            constexpr int kStep = kThr / LEAF;
#pragma unroll 8
            for (int l = 0; l < kSlice / kStep; ++l, src += kStep * ldb)
              tc::copy4(sb + (pb + l * kStep) * LEAF + cb, src, 4);
          }
        } else {
          stage<LEAF, kSlice, kLdA, kThr>(s, A, m, kd, lda, r0, k0, vec_a);
          stage<kSlice, LEAF, LEAF, kThr>(sb, B, kd, n, ldb, k0, c0, vec_b);
        }
        if (q % kPerK == kPerK - 1 && q + 1 < nslices) k_ahead = __ldg(k_idx + q / kPerK + 1) & 0x3ff;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int q = 0; q < kStages - 1; ++q) fetch(q);
    for (int q = 0; q < nslices; ++q) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
      tile_sync<T>(group);   // slice q is here; slice q - 1 has been read
      fetch(q + kStages - 1);
      const float* sa = smem + (q % kStages) * T::kStageFloats + (wr + ty) * kLdA;
      const float* sb = smem + (q % kStages) * T::kStageFloats + LEAF * kLdA + wc + tx * 4;
#pragma unroll
      for (int s2 = 0; s2 < kSlice; s2 += 2) {
        float2 a[TM];
#pragma unroll
        for (int u = 0; u < TM; ++u) a[u] = *reinterpret_cast<const float2*>(sa + kTy * u * kLdA + s2);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          uint64_t b[TN / 2];
#pragma unroll
          for (int h = 0; h < kHalves; ++h) {
            const ulonglong2 x =
                *reinterpret_cast<const ulonglong2*>(sb + (s2 + e) * LEAF + 4 * kTx * h);
            b[2 * h] = x.x;
            b[2 * h + 1] = x.y;
          }
#pragma unroll
          for (int u = 0; u < TM; ++u) {
            const float f = e == 0 ? a[u].x : a[u].y;
            const uint64_t aa = pair(f, f);
#pragma unroll
            for (int v = 0; v < TN / 2; ++v) acc[u][v] = fma2(b[v], aa, acc[u][v]);
          }
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");

    // epilogue: C = alpha * acc + beta * C (the old C is read only when beta != 0)
    const float alpha = in.alpha, beta = in.beta;
    SumSq ss = sumsq_empty();
#pragma unroll
    for (int u = 0; u < TM; ++u) {
      const int64_t r = r0 + wr + ty + kTy * u;
      const bool row_in = r < m;
      float x[TN];
#pragma unroll
      for (int v = 0; v < TN / 2; ++v) unpair(acc[u][v], x[2 * v], x[2 * v + 1]);
#pragma unroll
      for (int h = 0; h < kHalves; ++h) {
        const int64_t c = c0 + wc + 4 * kTx * h + tx * 4;
        float* p = C + r * ldc + c;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float& y = x[4 * h + q];
          y = __fmul_rn(alpha, y);
          if (beta != 0.0f) y = row_in && c + q < n ? __fmaf_rn(beta, p[q], y) : 0.0f;
        }
        if (!row_in) continue;
        if (vec_c && c + 3 < n) {
          *reinterpret_cast<float4*>(p) = make_float4(x[4 * h], x[4 * h + 1], x[4 * h + 2], x[4 * h + 3]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (c + q < n) p[q] = x[4 * h + q];
        }
      }
      if (in.nC) {   // C's norm map for a chained product: the row's stored values
#pragma unroll
        for (int q = 0; q < TN; ++q)
          if (!(row_in && c0 + wc + 4 * kTx * (q / 4) + tx * 4 + q % 4 < n)) x[q] = 0.0f;
        sumsq_group<TN>(ss, x);
      }
    }
    if (in.nC) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, ss.hi, off);
        const float l = __shfl_xor_sync(0xffffffffu, ss.lo, off);
        const int e = __shfl_xor_sync(0xffffffffu, ss.e, off);
        sumsq_merge_any(ss, h, l, e);
      }
      if (lane == 0) s_norm[group * T::kWarps + warp] = ss;
      tile_sync<T>(group);
      if (tid == 0) {
        SumSq tot = s_norm[group * T::kWarps];
        for (int w2 = 1; w2 < T::kWarps; ++w2) {
          const SumSq o = s_norm[group * T::kWarps + w2];
          sumsq_merge_any(tot, o.hi, o.lo, o.e);
        }
        in.nC[t] = sumsq_sqrt(tot);
      }
    }
  }
  if (!dynamic) return;
  // dynamic order: the empty tiles are dealt with a fixed stride
  for (int64_t w = ne + blockIdx.x * T::kGroups + group; w < all; w += (int64_t)gridDim.x * T::kGroups) {
    const int g = Bf.order[w];
    const Inst& in = R.at(inst_of(R, Bf, g));
    zero_tile<LEAF, T::kThreads>(in, g - in.tile0, tid);
  }
}

// Few tiles.  A function of its own: with both forms in the kernel's body the other one
// fetches its first instructions from further on, 1 to 3 us.  The empty tiles are taken by
// single warps (by the groups of four 1 to 2 us more with a dozen of them per SM).
template <int LEAF>
__device__ __noinline__ void multiply_wide(const InstRef& R, const PlanBuffers& Bf, int dynamic,
                                           int zeros) {
  using T = SimtTile<LEAF, true>;
  static_assert(T::kCtaThreads == SimtTile<LEAF, false>::kCtaThreads &&
                    T::kCtaSmem == SimtTile<LEAF, false>::kCtaSmem,
                "one launch serves both forms");
  __shared__ int s_taken, s_zeroed, s_next[T::kGroups];
  __shared__ SumSq s_norm[T::kGroups * T::kWarps];
  if (threadIdx.x == 0) s_taken = s_zeroed = 0;
  __syncthreads();
  const int ne = Bf.bdev->nonempty, lane = threadIdx.x & 31;
  multiply_tiles<T>(R, Bf, ne, dynamic, 0, &s_taken, s_next, s_norm, threadIdx.x);
  if (!zeros) return;
  for (;;) {
    int z = 0;
    if (lane == 0) z = atomicAdd(&s_zeroed, 1);
    z = __shfl_sync(0xffffffffu, z, 0);
    const int64_t w = ne + blockIdx.x + (int64_t)z * gridDim.x;
    if (w >= Bf.tiles) return;
    const int g = Bf.order[w];
    const Inst& in = R.at(inst_of(R, Bf, g));
    zero_tile<LEAF, 32>(in, g - in.tile0, lane);
  }
}

template <int LEAF>
__global__ void __launch_bounds__(SimtTile<LEAF, false>::kCtaThreads, 1)
    simt_kernel(InstRef R, PlanBuffers Bf, int dynamic, int zeros) {
  using T = SimtTile<LEAF, false>;
  __shared__ int s_taken;               // tiles of this SM handed out after its groups' first
  __shared__ int s_next[T::kGroups];
  __shared__ SumSq s_norm[T::kGroups * T::kWarps];
  const int thread = threadIdx.x;
  if (thread == 0) s_taken = 0;
  __syncthreads();
  pdl_wait();
  const int ne = Bf.bdev->nonempty;
  if constexpr (LEAF < 128) {
    const int64_t sms = gridDim.x, empty = zeros ? Bf.tiles - ne : 0;
    if (ne <= sms || (ne <= kWideTiles * sms && empty <= kWideTiles * sms)) {
      multiply_wide<LEAF>(R, Bf, dynamic, zeros);
      return;
    }
  }
  multiply_tiles<T>(R, Bf, ne, dynamic, zeros, &s_taken, s_next, s_norm, thread);
}

template <int LEAF>
cudaError_t launch(const InstRef& ref, const PlanBuffers& b, int schedule, bool zeros,
                   cudaStream_t s) {
  using T = SimtTile<LEAF, false>;
  static int sms[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (sms[dev] == 0) {
    int count = 0;
    e = cudaFuncSetAttribute(simt_kernel<LEAF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)T::kCtaSmem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    sms[dev] = std::max(1, count);
  }
  const int grid = (int)std::min<int64_t>(b.tiles, (int64_t)sms[dev]);
  return launch_pdl(simt_kernel<LEAF>, dim3(grid), dim3(T::kCtaThreads), T::kCtaSmem, s, ref, b,
                    (int)(schedule == kScheduleDynamic), zeros ? 1 : 0);
}

}  // namespace

bool simt_writes_zeros(const InstRef& ref, const PlanBuffers& b, int leaf, bool beside) {
  return !ref.any_scaled && b.tiles * leaf * leaf * (int64_t)sizeof(float) <= own_zero_bytes(leaf, beside);
}

cudaError_t launch_multiply_simt(const InstRef& ref, const PlanBuffers& b, int leaf,
                                 int schedule, bool zeros, cudaStream_t s) {
  switch (leaf) {
    case 32: return launch<32>(ref, b, schedule, zeros, s);
    case 64: return launch<64>(ref, b, schedule, zeros, s);
    case 128: return launch<128>(ref, b, schedule, zeros, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace spamm
