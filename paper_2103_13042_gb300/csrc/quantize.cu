// Operand rounding for the tensor-core multiply (mixed precision on top of the
// paper's FP16 tensor-core kernel, Section 3.3 / Algorithm 3).
//
// For every leaf block that some surviving triple uses (the plan's list of
// needed blocks) a CTA finds e = frexp exponent of its largest magnitude,
// scales by 2^-e (exact), rounds to nearest-even in the operand format (hi)
// and, in split modes, rounds the exact residual scaled by 2^s_lo (lo).  The
// result is written directly as the K-major, 128-byte swizzled image the MMA
// reads: chunk c of a block holds K elements [c*kc, (c+1)*kc) (kc = 128 bytes /
// element size) for every row, 128 bytes per row, 16-byte pieces XOR-swizzled by
// (row mod 8).  A blocks keep their rows; B blocks are transposed (image row n =
// column n of the block).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "tc.cuh"
#include "tc_common.cuh"

namespace spamm {
namespace {

// Round to nearest even, keeping 10 explicit significand bits (TF32), on the
// IEEE bit pattern; NaN/Inf pass through unchanged.
__device__ __forceinline__ float round_tf32(float x) {
  uint32_t u = __float_as_uint(x);
  if ((u & 0x7f800000u) == 0x7f800000u) return x;
  u += 0xfffu + ((u >> 13) & 1u);
  return __uint_as_float(u & 0xffffe000u);
}

// A block's exponent from its largest magnitude.  BF16 and TF32 have FP32's exponent
// range: the scaling only has to keep products and sums inside it, so e is rounded up to a
// multiple of 32 (scaled maximum in [2^-33, 1)).  The roundings are those of the exact
// exponent for every entry above 2^-94 of the block's maximum (hi parts) and above 2^-80
// (lo parts of the split modes), and the blocks of a tile mostly share one exponent sum:
// the multiply's runs (one accumulator pass per change of the sum) stay long.  FP16 keeps
// the exact exponent: its range is the constraint.
template <uint32_t FMT>
__device__ __forceinline__ int block_exponent(float mx) {
  int ex = 0;
  if (mx > 0.0f && mx <= 3.402823466e38f) frexpf(mx, &ex);
  return FMT == tc::kFmtF16 ? ex : ((ex + 31) >> 5) << 5;
}

// Two entries rounded to nearest even and packed (the first in the low half).
template <uint32_t FMT>
__device__ __forceinline__ uint32_t pack_pair(float a, float b) {
  if constexpr (FMT == tc::kFmtBF16) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return (uint32_t)__bfloat16_as_ushort(p.x) | ((uint32_t)__bfloat16_as_ushort(p.y) << 16);
  } else {
    const __half2 p = __floats2half2_rn(a, b);
    return (uint32_t)__half_as_ushort(__low2half(p)) | ((uint32_t)__half_as_ushort(__high2half(p)) << 16);
  }
}

// The two values back (exact).
template <uint32_t FMT>
__device__ __forceinline__ void unpack_pair(uint32_t w, float& a, float& b) {
  if constexpr (FMT == tc::kFmtBF16) {
    a = __uint_as_float(w << 16);
    b = __uint_as_float(w & 0xffff0000u);
  } else {
    a = __half2float(__ushort_as_half((unsigned short)(w & 0xffffu)));
    b = __half2float(__ushort_as_half((unsigned short)(w >> 16)));
  }
}

// One 16-byte piece of an image: v scaled by 2^-ex, rounded (hi), and in split modes
// the exact residual scaled by 2^lo shift, rounded (lo).
template <uint32_t FMT, bool SPLIT>
__device__ __forceinline__ void q_round(float* v, bool pow2_ok, float scale, int ex,
                                        float lo_scale, uint4* ph, uint4* pl) {
  constexpr int N = FMT == tc::kFmtTF32 ? 4 : 8;
#pragma unroll
  for (int z = 0; z < N; ++z) v[z] = pow2_ok ? __fmul_rn(v[z], scale) : ldexpf(v[z], -ex);
  uint32_t w[4];
#pragma unroll
  for (int z = 0; z < 4; ++z) {
    if constexpr (FMT == tc::kFmtTF32) w[z] = __float_as_uint(round_tf32(v[z]));
    else w[z] = pack_pair<FMT>(v[2 * z], v[2 * z + 1]);
  }
  *ph = make_uint4(w[0], w[1], w[2], w[3]);
  if constexpr (SPLIT) {
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      if constexpr (FMT == tc::kFmtTF32) {
        w[z] = __float_as_uint(
            round_tf32(__fmul_rn(__fsub_rn(v[z], __uint_as_float(w[z])), lo_scale)));
      } else {
        float h0, h1;
        unpack_pair<FMT>(w[z], h0, h1);
        w[z] = pack_pair<FMT>(__fmul_rn(__fsub_rn(v[2 * z], h0), lo_scale),
                          __fmul_rn(__fsub_rn(v[2 * z + 1], h1), lo_scale));
      }
    }
    *pl = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Loads X[r][c] of a rows x cols matrix with leading dimension ld, 0 outside it.
__device__ __forceinline__ float ld_or_zero(const float* X, int64_t rows, int64_t cols,
                                            int64_t ld, int64_t r, int64_t c) {
  return (r < rows && c < cols) ? __ldg(X + r * ld + c) : 0.0f;
}

// Leaf 64.  One CTA per used leaf block (the plan's needed-block list), one pass:
// each thread owns UNITS / kThreads 16-byte pieces of the image (unit u = image row
// u / PPR, piece u % PPR; consecutive threads take consecutive pieces, so a warp's
// stores cover whole 128-byte rows), loads their source values into registers (all
// loads of a thread issued before any use), the CTA reduces the block's largest
// magnitude, then every thread scales, rounds and stores.  A B block's image is its
// transpose: when the block is whole and its rows are 16-byte aligned, the CTA first
// copies it row by row (float4, coalesced) into shared memory with one float of
// padding per row and the threads gather their image pieces from there; other B
// blocks are read by columns (for them the staging was slower).  Eight CTAs per SM
// (six: batch rounding 0.85 -> 0.96 ms; TF32 images hold twice the pieces: six);
// the many small blocks hide each other's phases better than the ring of the
// leaf-128 form (256 uneven instances: 0.56 ms against 0.67).
constexpr int kQ64Threads = 256;
template <uint32_t FMT>
constexpr int q64_ctas() { return FMT == tc::kFmtTF32 ? 6 : 8; }

template <uint32_t FMT, int LEAF, bool SPLIT>
__global__ void __launch_bounds__(kQ64Threads, (q64_ctas<FMT>()))
    quantize_kernel(InstRef R, PlanBuffers Bf, OperandImages img) {
  constexpr int kThreads = kQ64Threads;
  using L = TcLayout<FMT, LEAF>;
  constexpr int KC = L::kKc;                 // K elements per 128-byte chunk row
  constexpr int PER16 = 16 / L::kElt;        // elements per 16-byte piece
  constexpr int PPR = LEAF / PER16;          // pieces per image row
  constexpr int UNITS = LEAF * PPR;          // pieces per block image
  constexpr int U = UNITS / kThreads;        // pieces per thread
  static_assert(UNITS % kThreads == 0, "whole pieces per thread");
  __shared__ float s_max[kThreads / 32];
  extern __shared__ float s_blk[];   // [LEAF][LEAF + 1]: one B block, row-major
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int count = Bf.bdev->need_count;
  const float lo_scale = (float)(1 << L::kLoShift);

  for (int idx = blockIdx.x; idx < count; idx += gridDim.x) {
    const uint32_t ent = Bf.need_list[idx];
    const bool isB = (ent >> 31) != 0;
    const int64_t blk = (int64_t)(ent & 0x7fffffffu);   // global block number of A or of B
    const Inst& in = R.at(isB ? inst_of_bblk(R, blk) : inst_of_ablk(R, blk));
    // A block (I, K): rows of A, K along its columns; B block (K, J): K along its rows
    const int64_t lb = blk - (isB ? in.bblk0 : in.ablk0);
    const int64_t gcols = isB ? in.bn : in.bk;                 // blocks per row of the grid
    const int64_t rows = isB ? in.kd : in.m, cols = isB ? in.n : in.kd;
    const int64_t ld = isB ? in.ldb : in.lda;                  // leading dimension
    const float* __restrict__ X = isB ? in.B : in.A;
    const int64_t r0 = (lb / gcols) * LEAF, c0 = (lb % gcols) * LEAF;
    const bool full = r0 + LEAF <= rows && c0 + LEAF <= cols;
    const bool vec = full && (ld & 3) == 0;

    if (isB && vec) {   // stage the block row-major (float4, coalesced), then read it
                        // transposed; the previous block's pieces were read before the
                        // loop's closing barrier
      constexpr int F4 = LEAF / 4;   // float4 per block row
      for (int t = tid; t < LEAF * F4; t += kThreads) {
        const int rr = t / F4, c4 = t - rr * F4;
        const float4 v = __ldg(reinterpret_cast<const float4*>(X + (r0 + rr) * ld + c0) + c4);
        float* d = s_blk + rr * (LEAF + 1) + 4 * c4;
        d[0] = v.x;
        d[1] = v.y;
        d[2] = v.z;
        d[3] = v.w;
      }
      __syncthreads();
    }
    float x[U][PER16];
#pragma unroll
    for (int r = 0; r < U; ++r) {
      const int u = tid + r * kThreads;
      const int row = u / PPR, k0 = (u % PPR) * PER16;
      if (!isB) {   // image row = block row, K along the block's columns
        const float* src = X + (r0 + row) * ld + c0 + k0;
        if (vec) {
#pragma unroll
          for (int q = 0; q < PER16; q += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(src + q));
            x[r][q] = v.x; x[r][q + 1] = v.y; x[r][q + 2] = v.z; x[r][q + 3] = v.w;
          }
        } else if (full) {
#pragma unroll
          for (int q = 0; q < PER16; ++q) x[r][q] = __ldg(src + q);
        } else {
#pragma unroll
          for (int q = 0; q < PER16; ++q) x[r][q] = ld_or_zero(X, rows, cols, ld, r0 + row, c0 + k0 + q);
        }
      } else if (vec) {   // image row = block column, K along the block's rows (staged)
#pragma unroll
        for (int q = 0; q < PER16; ++q) x[r][q] = s_blk[(k0 + q) * (LEAF + 1) + row];
      } else if (full) {
#pragma unroll
        for (int q = 0; q < PER16; ++q) x[r][q] = __ldg(X + (r0 + k0 + q) * ld + c0 + row);
      } else {
#pragma unroll
        for (int q = 0; q < PER16; ++q) x[r][q] = ld_or_zero(X, rows, cols, ld, r0 + k0 + q, c0 + row);
      }
    }
    // largest magnitude of the block (NaN ignored, as fmaxf does)
    float mx = 0.0f;
#pragma unroll
    for (int r = 0; r < U; ++r)
#pragma unroll
      for (int q = 0; q < PER16; ++q) mx = fmaxf(mx, fabsf(x[r][q]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (lane == 0) s_max[warp] = mx;
    __syncthreads();
    mx = 0.0f;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) mx = fmaxf(mx, s_max[w]);
    const int ex = block_exponent<FMT>(mx);
    if (tid == 0) (isB ? img.eb : img.ea)[blk] = ex;
    // 2^-ex as a float when it is a normal number (the usual case), else ldexpf
    const bool pow2_ok = ex >= -126 && ex <= 126;
    const float scale = pow2_ok ? __int_as_float((127 - ex) << 23) : 1.0f;

    uint8_t* hi_img = (isB ? img.b_hi : img.a_hi) + blk * (int64_t)L::kBlockBytes;
    uint8_t* lo_img = SPLIT ? (isB ? img.b_lo : img.a_lo) + blk * (int64_t)L::kBlockBytes : nullptr;
#pragma unroll
    for (int r = 0; r < U; ++r) {
      const int u = tid + r * kThreads;
      const int row = u / PPR, k0 = (u % PPR) * PER16;
      uint4 ph, pl;
      q_round<FMT, SPLIT>(x[r], pow2_ok, scale, ex, lo_scale, &ph, &pl);
      const uint32_t off = (uint32_t)(k0 / KC) * (LEAF * 128) + tc::sw128_offset(row, (k0 % KC) / PER16);
      *reinterpret_cast<uint4*>(hi_img + off) = ph;
      if constexpr (SPLIT) *reinterpret_cast<uint4*>(lo_img + off) = pl;
    }
    __syncthreads();   // s_max and s_blk are rewritten for the next block
  }
}

// Leaf 128.  A CTA streams the used leaf blocks (the plan's needed-block list) with a fixed
// stride through a ring of kStages shared-memory buffers, filled by asynchronous
// copies of 16 bytes kStages - 1 blocks ahead (rows that are not 16-byte aligned
// from the boundary at or below their first entry).  Of the block at hand each thread reads
// its image pieces into registers, the CTA reduces the largest magnitude, and every
// thread scales, rounds and stores.  An A piece is a run of a row; a B piece
// (transposed image) is a run of a column, two neighbouring pieces of 16
// neighbouring columns per warp, so that both the reads and the 32-byte sectors
// stored are whole.  Bound by HBM: the block is read once and the image written
// once.
template <uint32_t FMT, int LEAF, bool SPLIT>
struct QCfg {
  using L = TcLayout<FMT, LEAF>;
  static constexpr int kThreads = 512;
  static constexpr int kWarps = kThreads / 32;
  static constexpr int kLd = LEAF + 4;                      // floats per staged row (16-byte rows)
  static constexpr int kStages = 3;
  static constexpr int kCtas = 1;                           // per SM
  static constexpr int kInFloats = LEAF * kLd;
  static constexpr int kDescs = kStages + 1;
  static constexpr size_t kDescOffset = (size_t)kStages * kInFloats * sizeof(float);
  static constexpr size_t kSmem = kDescOffset + kDescs * 64;
  static_assert(kSmem * kCtas <= 226 * 1024, "shared memory");
};

// Where a needed-block entry lies.
struct QBlock {
  const float* src;      // the block's first entry
  const float* end;      // the end of its matrix
  int64_t ld;
  int64_t blk;           // global block number
  int rows, cols;        // of the block inside the matrix (rows 0: no block)
  int vec;               // rows 16-byte aligned
  int isB;               // a block of B
};
static_assert(sizeof(QBlock) <= 64, "one slot per block in flight");

template <int LEAF>
__device__ __forceinline__ QBlock q_block(const InstRef& R, uint32_t ent) {
  QBlock q;
  q.isB = (int)(ent >> 31);
  q.blk = (int64_t)(ent & 0x7fffffffu);
  const Inst& in = R.at(q.isB ? inst_of_bblk(R, q.blk) : inst_of_ablk(R, q.blk));
  // A block (I, K): rows of A, K along its columns; B block (K, J): K along its rows
  const int lb = (int)(q.blk - (q.isB ? in.bblk0 : in.ablk0));
  const int gcols = q.isB ? in.bn : in.bk;                   // blocks per row of the grid
  const int bi = lb / gcols, bj = lb - bi * gcols;
  const int64_t rows = q.isB ? in.kd : in.m, cols = q.isB ? in.n : in.kd;
  const int64_t r0 = (int64_t)bi * LEAF, c0 = (int64_t)bj * LEAF;
  q.ld = q.isB ? in.ldb : in.lda;
  q.src = (q.isB ? in.B : in.A) + r0 * q.ld + c0;
  q.end = (q.isB ? in.B : in.A) + (rows - 1) * q.ld + cols;
  q.rows = (int)min((int64_t)LEAF, rows - r0);
  q.cols = (int)min((int64_t)LEAF, cols - c0);
  q.vec = (q.ld & 3) == 0;   // the operands are 16-byte aligned
  return q;
}

// Distance of row r of a block from the 16-byte boundary its staged row starts at.
__device__ __forceinline__ int q_shift(const QBlock& q, int r) {
  return (int)(((uint32_t)(reinterpret_cast<uintptr_t>(q.src) >> 2) + (uint32_t)r * (uint32_t)q.ld) & 3u);
}

// Starts the copies of a block into a stage.  Aligned rows: zeros outside the
// matrix; others: whatever the matrix holds beside the block.
template <int LEAF, int LD, int THREADS>
__device__ __forceinline__ void q_fetch(float* dst, const QBlock& q) {
  constexpr int kPer = LEAF / 4, kStep = THREADS / kPer;
  const int tid = threadIdx.x;
  const int c = tid % kPer * 4, r0 = tid / kPer;
  const float* src = q.src + (int64_t)r0 * q.ld + c;
  if (q.vec) {
    const int left = q.cols - c, bytes = left >= 4 ? 16 : (left > 0 ? left * 4 : 0);
#pragma unroll
    for (int l = 0; l < LEAF / kStep; ++l, src += kStep * q.ld) {
      const int b = r0 + l * kStep < q.rows ? bytes : 0;
      tc::copy16(dst + (r0 + l * kStep) * LD + c, b ? src : q.src, b);
    }
  } else {
    // piece c / 4 of a row, and one more per row for the entries the shift moves out
    auto piece = [&](int r, const float* at, float* to) {
      const float* p = reinterpret_cast<const float*>(reinterpret_cast<uintptr_t>(at) & ~(uintptr_t)15);
      const int64_t left = q.end - p;
      if (r < q.rows && left > 0) tc::copy16(to, p, left >= 4 ? 16 : (int)left * 4);
    };
#pragma unroll
    for (int l = 0; l < LEAF / kStep; ++l, src += kStep * q.ld)
      piece(r0 + l * kStep, src, dst + (r0 + l * kStep) * LD + c);
    if (tid < LEAF) piece(tid, q.src + (int64_t)tid * q.ld + LEAF, dst + tid * LD + LEAF);
  }
}

template <uint32_t FMT, int LEAF, bool SPLIT>
__global__ void __launch_bounds__(QCfg<FMT, LEAF, SPLIT>::kThreads, (QCfg<FMT, LEAF, SPLIT>::kCtas))
    quantize_ring_kernel(InstRef R, PlanBuffers Bf, OperandImages img) {
  using C = QCfg<FMT, LEAF, SPLIT>;
  using L = typename C::L;
  constexpr int KC = L::kKc;                 // K elements per 128-byte chunk row
  constexpr int PER16 = 16 / L::kElt;        // elements per 16-byte piece
  constexpr int PPR = LEAF / PER16;          // pieces per image row
  constexpr int U = LEAF * PPR / C::kThreads;   // pieces per thread
  extern __shared__ __align__(128) uint8_t smem[];
  float* ring = reinterpret_cast<float*>(smem);
  QBlock* descs = reinterpret_cast<QBlock*>(smem + C::kDescOffset);
  __shared__ float s_max[2][C::kWarps];
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int count = Bf.bdev->need_count;
  const float lo_scale = (float)(1 << L::kLoShift);
  // block number b of this CTA is entry blockIdx.x + b * gridDim.x of the list; the
  // last warp decodes it kStages blocks ahead (its list entry read one further ahead)
  const int step = gridDim.x;
  auto entry = [&](int64_t b) -> uint32_t {
    const int64_t i = blockIdx.x + b * step;
    return i < count ? __ldg(Bf.need_list + i) : 0xffffffffu;
  };
  auto decode = [&](int b, uint32_t ent) {
    QBlock q{};
    if (blockIdx.x + (int64_t)b * step < count) q = q_block<LEAF>(R, ent);
    descs[b % C::kDescs] = q;
  };
  uint32_t ahead = 0u;
  if (warp == C::kWarps - 1) {
    if (lane < C::kStages) decode(lane, entry(lane));
    ahead = entry(C::kStages);
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < C::kStages - 1; ++b) {
    const QBlock q = descs[b];
    if (q.rows > 0) q_fetch<LEAF, C::kLd, C::kThreads>(ring + b * C::kInFloats, q);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  uint32_t par = 0;
  for (int b = 0;; ++b) {
    asm volatile("cp.async.wait_group %0;" ::"n"(C::kStages - 2) : "memory");
    __syncthreads();   // block b is here, block b - 1 has been read, descriptor b + kStages - 1 too
    const QBlock q = descs[b % C::kDescs];
    if (q.rows == 0) break;
    {
      const QBlock f = descs[(b + C::kStages - 1) % C::kDescs];
      if (f.rows > 0)
        q_fetch<LEAF, C::kLd, C::kThreads>(ring + (b + C::kStages - 1) % C::kStages * C::kInFloats, f);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (warp == C::kWarps - 1) {
      if (lane == 0) decode(b + C::kStages, ahead);
      ahead = entry((int64_t)b + C::kStages + 1);
    }
    const float* in = ring + b % C::kStages * C::kInFloats;
    float x[U][PER16];
    const bool whole = q.rows == LEAF && q.cols == LEAF;
    if (!q.isB) {   // image row = block row: consecutive threads take consecutive pieces
#pragma unroll
      for (int l = 0; l < U; ++l) {
        const int u = tid + l * C::kThreads, row = u / PPR, k0 = u % PPR * PER16;
        const float* p = in + row * C::kLd + k0;
        if (q.vec) {
#pragma unroll
          for (int z = 0; z < PER16; z += 4) {
            const float4 v = *reinterpret_cast<const float4*>(p + z);
            x[l][z] = v.x; x[l][z + 1] = v.y; x[l][z + 2] = v.z; x[l][z + 3] = v.w;
          }
        } else {   // four reads at a time, rotated among the lanes that share their banks
          p += q_shift(q, row);
          const int rot = lane >> 3;
#pragma unroll
          for (int z = 0; z < PER16; z += 4) {
            float t[4];
#pragma unroll
            for (int y = 0; y < 4; ++y) t[y] = p[z + ((y + rot) & 3)];
#pragma unroll
            for (int y = 0; y < 4; ++y) {   // entry y was read in turn (y - rot) & 3
              const int w = (y - rot) & 3;
              const float e = w == 0 ? t[0] : (w == 1 ? t[1] : (w == 2 ? t[2] : t[3]));
              x[l][z + y] = whole || (row < q.rows && k0 + z + y < q.cols) ? e : 0.0f;
            }
          }
        }
      }
    } else {        // image row = block column: a warp takes 16 columns x 2 pieces
#pragma unroll
      for (int l = 0; l < U; ++l) {
        const int v = warp + l * C::kWarps;
        const int row = v % (LEAF / 16) * 16 + (lane >> 1);
        const int k0 = (v / (LEAF / 16) * 2 + (lane & 1)) * PER16;
#pragma unroll
        for (int z = 0; z < PER16; ++z) {
          if (q.vec) {
            x[l][z] = in[(k0 + z) * C::kLd + row];
          } else {
            const float e = in[(k0 + z) * C::kLd + q_shift(q, k0 + z) + row];
            x[l][z] = whole || (k0 + z < q.rows && row < q.cols) ? e : 0.0f;
          }
        }
      }
    }
    // largest magnitude of the block (NaN ignored, as fmaxf does)
    float mx = 0.0f;
#pragma unroll
    for (int l = 0; l < U; ++l)
#pragma unroll
      for (int z = 0; z < PER16; ++z) mx = fmaxf(mx, fabsf(x[l][z]));
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));   // mx >= 0
    if (lane == 0) s_max[par][warp] = mx;
    __syncthreads();
    mx = s_max[par][lane < C::kWarps ? lane : 0];
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
    par ^= 1u;
    const int ex = block_exponent<FMT>(mx);
    if (tid == 0) (q.isB ? img.eb : img.ea)[q.blk] = ex;
    // 2^-ex as a float when it is a normal number (the usual case), else ldexpf
    const bool pow2_ok = ex >= -126 && ex <= 126;
    const float scale = pow2_ok ? __int_as_float((127 - ex) << 23) : 1.0f;
    uint8_t* hi_img = (q.isB ? img.b_hi : img.a_hi) + q.blk * (int64_t)L::kBlockBytes;
    uint8_t* lo_img = SPLIT ? (q.isB ? img.b_lo : img.a_lo) + q.blk * (int64_t)L::kBlockBytes : nullptr;
#pragma unroll
    for (int l = 0; l < U; ++l) {
      int row, k0;
      if (!q.isB) {
        const int u = tid + l * C::kThreads;
        row = u / PPR;
        k0 = u % PPR * PER16;
      } else {
        const int v = warp + l * C::kWarps;
        row = v % (LEAF / 16) * 16 + (lane >> 1);
        k0 = (v / (LEAF / 16) * 2 + (lane & 1)) * PER16;
      }
      const uint32_t off = (uint32_t)(k0 / KC) * (LEAF * 128) + tc::sw128_offset(row, (k0 % KC) / PER16);
      uint4 ph, pl;
      q_round<FMT, SPLIT>(x[l], pow2_ok, scale, ex, lo_scale, &ph, &pl);
      *reinterpret_cast<uint4*>(hi_img + off) = ph;
      if constexpr (SPLIT) *reinterpret_cast<uint4*>(lo_img + off) = pl;
    }
  }
}

template <uint32_t FMT, int LEAF, bool SPLIT>
cudaError_t launch_q(const InstRef& ref, const PlanBuffers& b, const OperandImages& img,
                     cudaStream_t s) {
  using C = QCfg<FMT, 128, SPLIT>;
  void (*kern)(InstRef, PlanBuffers, OperandImages);
  if constexpr (LEAF == 64) kern = quantize_kernel<FMT, 64, SPLIT>;
  else kern = quantize_ring_kernel<FMT, 128, SPLIT>;
  constexpr int kThreads = LEAF == 64 ? kQ64Threads : C::kThreads;
  constexpr size_t kSmem = LEAF == 64 ? (size_t)64 * 65 * sizeof(float) : C::kSmem;
  static int wave[64] = {};   // resident CTAs per device (occupancy x SMs)
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (wave[dev] == 0) {
    int sms = 0, per_sm = 0;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, kSmem);
    if (e != cudaSuccess) return e;
    wave[dev] = sms * std::max(1, per_sm);
  }
  // the list length is known on the device only: one full wave of CTAs
  const int64_t cap = b.ablks + b.bblks;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(cap, (int64_t)wave[dev]));
  return launch_pdl(kern, dim3(grid), dim3(kThreads), kSmem, s, ref, b, img);
}

}  // namespace

cudaError_t launch_quantize(spamm_precision_t prec, int leaf, const InstRef& ref,
                            const PlanBuffers& b, const OperandImages& img, cudaStream_t s) {
  const bool l64 = leaf == 64;
  switch (prec) {
    case SPAMM_BF16:
      return l64 ? launch_q<tc::kFmtBF16, 64, false>(ref, b, img, s)
                 : launch_q<tc::kFmtBF16, 128, false>(ref, b, img, s);
    case SPAMM_FP16:
      return l64 ? launch_q<tc::kFmtF16, 64, false>(ref, b, img, s)
                 : launch_q<tc::kFmtF16, 128, false>(ref, b, img, s);
    case SPAMM_BF16_SPLIT:
      return l64 ? launch_q<tc::kFmtBF16, 64, true>(ref, b, img, s)
                 : launch_q<tc::kFmtBF16, 128, true>(ref, b, img, s);
    case SPAMM_FP16_SPLIT:
      return l64 ? launch_q<tc::kFmtF16, 64, true>(ref, b, img, s)
                 : launch_q<tc::kFmtF16, 128, true>(ref, b, img, s);
    case SPAMM_TF32X3:
      return l64 ? launch_q<tc::kFmtTF32, 64, true>(ref, b, img, s)
                 : launch_q<tc::kFmtTF32, 128, true>(ref, b, img, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace spamm
