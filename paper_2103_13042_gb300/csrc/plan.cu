// Pair test and work-queue build (Algorithm 1 skip rule, Algorithm 2 bitmap and
// map_offset, Section 3.5.1 valid multiplications), for all output tiles of
// all instances of a table at once.
//
// Output tiles are enumerated in bands of 8 block rows, column by column inside
// a band; a unit is up to 32 consecutive tiles of one band (8 rows x 4 columns
// in a full band).  Stream order:
//   prep   (only when some instance needs ||A||_F ||B||_F before its products
//          are counted, or the table has more than kScanUnits units) per-CTA
//          sums of squared norms; clears the accumulators.
//   count  one CTA per unit: the unit's block rows of A and block columns of B
//          are turned into FP32 mantissa/exponent "screen" forms in shared
//          memory; a lane owns a tile, the warps share its k in 32-wide words
//          (the tile's survivor bitmask, built in a register: no ballots, no
//          cross-lane reductions per tile); skipped products are summed for
//          the bounds; split modes bin the surviving products by binade;
//          per-unit totals and longest-first bucket counts
//          (floor(log2 survivors) + 1).
//   fill   every CTA derives the first slots of its units itself, from the
//          totals of all units before them (no separate scan kernel); the
//          bitmask words are expanded into k lists (increasing, at
//          tile_beg[t] + rank); each non-empty tile takes its slot in the
//          longest-first order (bucket start + earlier units + rank, in
//          enumeration order inside a bucket), each empty tile its slot after
//          all non-empty ones; the blocks some surviving triple uses are
//          listed once each, 32 of them per atomic.
// Per-instance statistics come from a fill CTA of their own; in split modes every
// fill CTA forms the flag binade of its units' instances.
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "plan.cuh"

namespace spamm {

TauScreen make_tau_screen(double tau) {
  TauScreen t{};
  t.tau = tau;
  t.all = tau == 0.0;
  t.none = std::isinf(tau);
  if (!t.all && !t.none) {
    int e;
    double m = std::frexp(tau, &e);
    t.e = e;
    // the FP32 screen is decisive outside [1 - 2^-20, 1 + 2^-20] * m
    t.m_hi = (float)(m * (1.0 + std::ldexp(1.0, -20)));
    t.m_lo = (float)(m * (1.0 - std::ldexp(1.0, -20)));
  }
  return t;
}

namespace {

constexpr int kPrepThreads = 256;
constexpr int kCountWarps = 4;
constexpr int kCountThreads = kCountWarps * 32;
constexpr int kFillWarps = 8;
constexpr int kFillThreads = kFillWarps * 32;
constexpr int kUnitWarps = 4;        // fill: warps sharing one unit's tiles
constexpr int kStatWarps = 4;        // parts of an instance's sums over its units
constexpr int kHistWarps = 8;
constexpr int kHistTiles = 32;       // histogram: tiles per CTA
constexpr int kBandRows = 8;         // block rows per band of the tile enumeration
// Tables of at most kScanUnits units: a fill CTA reads every unit's totals (64
// bytes each).  Larger ones: groups of units, whose totals the count kernel
// adds up with atomics, so a fill CTA reads the groups and its own group's units.
constexpr int kScanUnits = 1024;
static_assert(kOrderKeys <= 12, "order buckets fit a unit's totals");

// Slots of a unit's (or a group's) totals, kPartInts per unit.
enum : int { kPartS = 0 /* survivors */, kPartNe = 12, kPartMax = 13 };   // 1 .. 11: buckets

// Columns of a unit: 32 tiles, and at most 16 staged rows and columns.
__host__ __device__ __forceinline__ int unit_cols(int bm) {
  if (bm >= kBandRows) return 32 / kBandRows;
  const int c = 32 / bm;
  return c < 16 - bm ? c : 16 - bm;
}

struct Unit {
  int r0, rows, j0, cols;   // block rows r0 .. r0 + rows - 1, columns j0 .. j0 + cols - 1
};

__device__ __forceinline__ Unit unit_at(const Inst& in, int lu) {
  const int uc = unit_cols(in.bm);
  const int per_band = (in.bn + uc - 1) / uc;
  const int band = lu / per_band;
  Unit u;
  u.r0 = band * kBandRows;
  u.rows = min(kBandRows, in.bm - u.r0);
  u.j0 = (lu - band * per_band) * uc;
  u.cols = min(uc, in.bn - u.j0);
  return u;
}

__host__ __device__ __forceinline__ int units_of(const Inst& in) {
  const int uc = unit_cols(in.bm);
  return ((in.bm + kBandRows - 1) / kBandRows) * ((in.bn + uc - 1) / uc);
}

// Longest-first bucket of a survivor count c >= 1: floor(log2 c) + 1.  Near-
// equal counts share a bucket, so the order keeps the enumeration's locality.
__device__ __forceinline__ int order_key(int c) { return 32 - __clz(c); }

// Screens of the pair test.  Zero norms take the mantissa 0.5 and an exponent
// below every sum that can survive, non-finite ones an exponent above every
// sum that can be skipped (also against a zero: NaN products survive).
constexpr int kTestZero = -100000, kTestNonFinite = 300000;

// make_screen's mantissa (rounded to nearest even) and exponent from the bit
// pattern: integer operations only, the FP64 pipe is narrow on this part.
__device__ __forceinline__ Screen test_screen(double x) {
  const int hi = __double2hiint(x);
  const uint32_t lo = (uint32_t)__double2loint(x);
  Screen s;
  if (hi >= 0x00100000 && hi < 0x7ff00000) {   // positive and normal
    const uint32_t m = (uint32_t)(hi & 0xfffff) << 3 | lo >> 29;
    const uint32_t up = ((lo & 0x1fffffffu) + (m & 1u)) > 0x10000000u ? 1u : 0u;
    s.m = __uint_as_float((126u << 23) + m + up);   // a carry gives 1.0
    s.e = (hi >> 20) - 1022;
    return s;
  }
  s = make_screen(x);
  if (s.e == kZeroExp) {
    s.m = 0.5f;
    s.e = kTestZero;
  } else if (s.e == kNonFiniteExp) {
    s.e = kTestNonFinite;
  }
  return s;
}

// tau in the form the test uses: mantissa window and exponent.  tau = 0 puts the
// exponent below every sum, tau = +Inf between the finite and the non-finite ones.
struct TestTau {
  float lo, hi;
  int e;
};

__device__ __forceinline__ TestTau test_tau(const TauScreen& T) {
  if (T.all) return TestTau{1.0f, 1.0f, -1000000};
  if (T.none) return TestTau{1.0f, 1.0f, 150000};
  return TestTau{T.m_lo, T.m_hi, T.e};
}

// q 2^D, D clamped to [-3, 4], for q = mA mB in [0.25, 1] and D = eA + eB - eT:
// !(na * nb < tau) holds if it is >= T.hi and fails if it is < T.lo; between the
// two (1 +- 2^-20) the FP64 product decides.
__device__ __forceinline__ float screen_value(float q, int D) {
  return __int_as_float(__float_as_int(q) + (min(max(D, -3), 4) * (1 << 23)));
}

// Extended-range FP32 sums (ExtSum, value m * 2^e): sums of relative products
// far below the FP32 range (decay matrices reach 1e-80 and less) keep ~24
// bits.  Terms below 2^-40 of the running sum are dropped.

// Binade of a positive normal FP32 value.
__device__ __forceinline__ int fexp(float x) {
  return (int)((__float_as_uint(x) >> 23) & 0xffu) - 127;
}

// s += q * 2^E (q > 0 normal), the rounding error of the addition collected in `low`
// (the scale of s.m).  The magnitudes are compared by their true binades; a term below
// 2^-40 of the other side is dropped.  Mantissas stay below 2^41, so the aligned product
// never leaves the FP32 range.
__device__ __forceinline__ void ext_add_two(ExtSum& s, float& low, float q, int E) {
  if (!(q > 0.0f)) return;
  const int ea = s.e + fexp(s.m), eb = E + fexp(q);
  if (s.m == 0.0f || eb > ea + 40) {
    s = ExtSum{q, E};
    low = 0.0f;
    return;
  }
  if (eb < ea - 40) return;
  float err;
  two_sum(s.m, __fmul_rn(q, pow2f(E - s.e)), s.m, err);   // |E - s.e| <= 84
  low = __fadd_rn(low, err);
  while (s.m >= 1099511627776.0f) {         // 2^40: renormalise
    s.m *= pow2f(-40);
    low *= pow2f(-40);
    s.e += 40;
  }
}

// Per-lane sum of a tile's skipped products q 2^D (q = mA mB in [0.25, 1]), held
// as (S + C) 2^Emax with Emax the largest exponent seen so far; terms more than 126
// binades below Emax are dropped.  A product that is not skipped comes with
// D = kSkipNone, far below every reference.  Eight products share one rescaling
// of the sum, without branches: along a decay matrix's rows every other
// product raises the reference.  They are summed in pairs, and C takes the rounding
// error of adding them to S, so that the error does not grow with the length of a
// lane's share of k (relative RMS error of a sum of 64 and of 1024 uniform terms:
// 4.1e-8 and 4.0e-8; one chain: 7.1e-8 and 1.3e-7).
struct SkipSum {
  float S, C;
  int Emax;
};
constexpr int kSkipNone = -(1 << 29);
constexpr int kSkipStart = kSkipNone + 1000;   // the empty sum's reference

// 2^k for -126 <= k <= 0, and 0 for k < -126.
__device__ __forceinline__ float pow2f_or_zero(int k) {
  return __int_as_float(max(k + 127, 0) << 23);
}

template <int N>
__device__ __forceinline__ void skip_add(SkipSum& s, const float (&q)[N], const int (&D)[N]) {
  int e = s.Emax;
#pragma unroll
  for (int z = 0; z < N; ++z) e = max(e, D[z]);
  float x[N];
#pragma unroll
  for (int z = 0; z < N; z += 2) {
    x[z / 2] = __fmul_rn(q[z], pow2f_or_zero(D[z] - e));
    if (z + 1 < N) x[z / 2] = __fmaf_rn(q[z + 1], pow2f_or_zero(D[z + 1] - e), x[z / 2]);
  }
#pragma unroll
  for (int w = N / 4; w > 0; w /= 2)
#pragma unroll
    for (int z = 0; z < w; ++z) x[z] = __fadd_rn(x[2 * z], x[2 * z + 1]);
  const float scale = pow2f_or_zero(max(s.Emax - e, -127));
  float err;
  two_sum(__fmul_rn(s.S, scale), x[0], s.S, err);
  s.C = __fmaf_rn(s.C, scale, err);
  s.Emax = e;
}

// The tile's sum from the lanes' (or warps') four shares, in pairs.
template <int LANES>
__device__ __forceinline__ float skip_total(const float (&S)[kCountWarps][LANES],
                                            const int (&E)[kCountWarps][LANES], int lane, int emax) {
  static_assert(kCountWarps == 4, "two pairs");
  float x[4];
#pragma unroll
  for (int w = 0; w < 4; ++w)
    x[w] = __fmul_rn(S[w][lane], pow2f_or_zero(max(E[w][lane] - emax, -127)));
  return __fadd_rn(__fadd_rn(x[0], x[1]), __fadd_rn(x[2], x[3]));
}

// Warp total of ExtSums in one pass: every lane rescales its sum to 2^-40 of
// the warp's largest binade (smaller terms dropped) and the
// FP32 values are added with xor shuffles (a fixed order).
__device__ __forceinline__ ExtSum ext_warp_sum_fast(ExtSum s) {
  constexpr int kNone = -(1 << 29);
  const int eb = s.m > 0.0f ? s.e + fexp(s.m) : kNone;   // true binade of the lane's sum
  int emax = eb;
  for (int off = 16; off > 0; off >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, off));
  if (emax == kNone) return ExtSum{0.0f, 0};
  float v = 0.0f;
  if (eb >= emax - 40) v = s.m * pow2f(s.e - (emax - 40));   // exponent in [-80, 40]
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  ExtSum r{v, emax - 40};
  while (r.m >= 1099511627776.0f) {   // keep the mantissa below 2^40 (v < 2^89)
    r.m *= pow2f(-40);
    r.e += 40;
  }
  return r;
}

// s += q * 2^E without branches and without the error term: for short sums on a critical
// path, whose lanes would take every side of them.
__device__ __forceinline__ void ext_add_flat(ExtSum& s, float q, int E) {
  const int ea = s.e + fexp(s.m), eb = E + fexp(q);
  const bool any = q > 0.0f, none = s.m == 0.0f;
  const bool take = any && (none || eb > ea + 40);
  const bool both = any && !none && eb <= ea + 40 && eb >= ea - 40;
  float m = __fmaf_rn(q, pow2f(min(max(E - s.e, -84), 84)), s.m);
  int e = s.e;
#pragma unroll
  for (int t = 0; t < 3; ++t) {   // renormalise (m < 2^83)
    const bool big = m >= 1099511627776.0f;
    m = big ? m * pow2f(-40) : m;
    e += big ? 40 : 0;
  }
  s.m = take ? q : (both ? m : s.m);
  s.e = take ? E : (both ? e : s.e);
}

__device__ __forceinline__ ExtSum ext_warp_sum(ExtSum s) {
#pragma unroll 1
  for (int off = 16; off > 0; off >>= 1) {
    const float m = __shfl_xor_sync(0xffffffffu, s.m, off);
    const int e = __shfl_xor_sync(0xffffffffu, s.e, off);
    ext_add_flat(s, m, e);
  }
  return s;
}

__device__ __forceinline__ double ext_value(ExtSum s) {
  if (s.m == 0.0f) return 0.0;
  const int e = fexp(s.m) + s.e;   // the value's binade: built from the bits when normal
  if (e > -1022 && e < 1023) {
    const uint32_t f = __float_as_uint(s.m) & 0x7fffffu;
    return __hiloint2double((e + 1023) << 20 | (int)(f >> 3), (int)(f << 29));
  }
  return ldexp((double)s.m, s.e);
}

// floor(log2(fl(fl(na nb) * inv))) clamped to the flag bins: the binade of a relative norm
// product, taken from one FP64 multiply so that every implementation bins it alike.
__device__ __forceinline__ int rel_bin(double p, double inv) {
  const double r = __dmul_rn(p, inv);
  if (!(r > 0.0)) return kFlagBinMin;
  if (isinf(r)) return 1;
  const int b = ilogb(r);
  return b < kFlagBinMin ? kFlagBinMin : (b > 1 ? 1 : b);
}

__host__ __device__ __forceinline__ int prep_parts(const Inst& in) {
  const int64_t na = (int64_t)in.bm * in.bk, nb = (int64_t)in.bk * in.bn;
  return (int)(((na > nb ? na : nb) + kPrepThreads - 1) / kPrepThreads);
}

__device__ __forceinline__ int inst_of_prep_cta(const InstRef& r, int cta) {
  return find_inst(r, cta, [](const Inst& x) { return (int64_t)x.prep0; });
}
__device__ __forceinline__ int inst_of_unit(const InstRef& r, int unit) {
  return find_inst(r, unit, [](const Inst& x) { return (int64_t)x.count0; });
}

// Partial sums of squared norms (kPrepThreads of A's and of B's per CTA) and, for
// the histogram, the screen forms; clears the accumulators of the later kernels.
__global__ void __launch_bounds__(kPrepThreads)
    prep_kernel(InstRef R, PlanBuffers Bf, int screens) {
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x;
  const Inst& in = R.at(inst_of_prep_cta(R, blockIdx.x));
  const int64_t na = (int64_t)in.bm * in.bk, nb = (int64_t)in.bk * in.bn;
  const int lc = blockIdx.x - in.prep0;
  const int64_t idx = (int64_t)lc * kPrepThreads + tid;
  if (lc == 0) {   // one CTA per instance clears its bins; the rest is dealt over the grid
    PlanDevice* pd = in.pd;
    for (int q = tid; q < kFlagBins; q += kPrepThreads) {
      pd->bin_sum[q] = 0.0;
      pd->bin_cnt[q] = 0;
    }
    if (tid < kHistBins) pd->hist[tid] = 0u;
    if (tid == 0) pd->ticket = 0u;
  }
  {
    const int64_t g0 = (int64_t)blockIdx.x * kPrepThreads + tid;
    const int64_t gs = (int64_t)gridDim.x * kPrepThreads;
    for (int64_t g = g0; g < Bf.need_words_a + Bf.need_words_b; g += gs) Bf.need_bits[g] = 0u;
    if (Bf.group_shift) {
      const int64_t words =
          (int64_t)((Bf.count_ctas + (1 << Bf.group_shift) - 1) >> Bf.group_shift) * kPartInts;
      for (int64_t g = g0; g < words; g += gs) Bf.group[g] = 0;
    }
    if (g0 == 0) Bf.bdev->need_count = 0;
  }
  double qa = 0.0, qb = 0.0;
  if (idx < na) {
    const double a = in.nA[idx];
    if (screens) Bf.sA[in.ablk0 + idx] = make_screen(a);
    qa = a * a;
  }
  if (idx < nb) {
    const double b = in.nB[idx];
    if (screens) {
      const int64_t k = idx / in.bn, j = idx % in.bn;
      Bf.sBT[in.bblk0 + j * in.bk + k] = make_screen(b);
    }
    qb = b * b;
  }
  for (int off = 16; off > 0; off >>= 1) {
    qa += __shfl_xor_sync(0xffffffffu, qa, off);
    qb += __shfl_xor_sync(0xffffffffu, qb, off);
  }
  __shared__ double s_w[2][kPrepThreads / 32];
  if ((tid & 31) == 0) {
    s_w[0][tid / 32] = qa;
    s_w[1][tid / 32] = qb;
  }
  __syncthreads();
  if (tid < 2) {
    double x = 0.0;
    for (int w = 0; w < kPrepThreads / 32; ++w) x += s_w[tid][w];
    (tid ? Bf.part_b : Bf.part_a)[blockIdx.x] = x;
  }
}

// ||A||_F^2 (lane 0) and ||B||_F^2 (lane 1) from `count` partial sums at `first`, by one
// warp in a fixed order (every caller gets the same bits): the even lanes add up
// A's, the odd ones B's, so that one square root serves both (FP64 is scarce here).
// live = false: no load (instance_stats).
__device__ __forceinline__ double sum_norms2(const PlanBuffers& Bf, int first, int count,
                                             bool live = true) {
  const int lane = threadIdx.x & 31;
  const double* p = ((lane & 1) ? Bf.part_b : Bf.part_a) + first;
  double x = 0.0;
#pragma unroll 4
  for (int i = lane >> 1; i < count; i += 16) x += live ? __ldcg(p + i) : 0.0;
  for (int off = 16; off > 1; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// After prep: 1 / (||A|| ||B||) for a CTA of the instance (one warp calls it);
// `publish`: also write the norms to the instance's statistics.
__device__ __forceinline__ double instance_norms(const Inst& in, const PlanBuffers& Bf,
                                                 bool publish) {
  const double x = sqrt(sum_norms2(Bf, in.prep0, prep_parts(in)));
  const double na = __shfl_sync(0xffffffffu, x, 0), nb = __shfl_sync(0xffffffffu, x, 1);
  const double ab = na * nb, inv = ab > 0.0 ? 1.0 / ab : 0.0;
  if (publish && (threadIdx.x & 31) == 0) {
    in.pd->norm_a = na;
    in.pd->norm_b = nb;
    in.pd->inv_ab = inv;
  }
  return inv;
}

// The flag binade m = the largest mm in [kFlagBinMin - 1, 1] with
// c1 * sum_{bins < mm} p <= budget, in two halves of one warp each.  flag_prefix: the
// sums below every bin, in a fixed order (7 consecutive bins per lane, then a warp
// scan of the lane totals).  flag_pick: they grow with the bin, so every lane tests its
// first bin, and seven lanes the bins of the last lane that passed (a test of all seven
// by every lane is ten times the FP64 instructions, at 64 cycles each).
constexpr int kBinsPerLane = (kFlagBins + 31) / 32;   // 7

__device__ __forceinline__ void flag_prefix(const Inst& in, double* below) {
  const int lane = threadIdx.x & 31;
  double v[kBinsPerLane];
  double run = 0.0;
#pragma unroll
  for (int q = 0; q < kBinsPerLane; ++q) {
    const int b = lane * kBinsPerLane + q;
    v[q] = b < kFlagBins ? __ldcg(&in.pd->bin_sum[b]) : 0.0;
  }
#pragma unroll
  for (int q = 0; q < kBinsPerLane; ++q) run += v[q];
  double incl = run;
#pragma unroll 1
  for (int off = 1; off < 32; off <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  double x = incl - run;     // sum of the bins before this lane's first
#pragma unroll
  for (int q = 0; q < kBinsPerLane; ++q) {
    below[lane * kBinsPerLane + q] = x;
    x += v[q];
  }
  __syncwarp();
}

__device__ __forceinline__ int flag_pick(const Inst& in, double ab, double bound2,
                                         const double* below) {
  const int lane = threadIdx.x & 31;
  const double budget = 0.5 * (in.target_rel * ab - bound2);
  const bool first = budget >= 0.0 && in.c1 * below[lane * kBinsPerLane] <= budget &&
                     lane * kBinsPerLane < kFlagBins;
  const unsigned pass = __ballot_sync(0xffffffffu, first);
  if (pass == 0u) return kFlagBinMin - 1;
  const int b = (31 - __clz(pass)) * kBinsPerLane + min(lane, kBinsPerLane - 1);
  const bool ok = b < kFlagBins && in.c1 * below[b] <= budget;
  return kFlagBinMin + __reduce_max_sync(0xffffffffu, ok ? b : 0);
}

// One instance's sums over its units.
struct UnitSums {
  int S, ne, km;
  ExtSum b1, b2;
};

// One warp's part v of an instance's sums: its lane l takes the units 32 v + l,
// 32 v + l + 32 kStatWarps, ... (four units' loads at a time).  The kStatWarps parts
// are merged in order (merge_sums), whoever forms them, so that a single call and
// a batch give the same bits.  WHAT: 1 the counts and b1, 2 b2, 3 all.  live = false: no
// load (instance_stats).
template <int WHAT>
__device__ __forceinline__ UnitSums unit_sums(const Inst& in, const PlanBuffers& Bf, int v,
                                              bool live = true) {
  const int units = units_of(in);
  constexpr int nt = 32 * kStatWarps;
  UnitSums r{0, 0, 0, {0.0f, 0}, {0.0f, 0}};
  if (32 * v >= units) return r;   // uniform over the warp
  for (int q0 = 32 * v + (threadIdx.x & 31); q0 < units; q0 += 4 * nt) {
    int s4[4];
    int4 hi[4], bb[4];
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const int64_t q = in.count0 + q0 + z * nt;
      s4[z] = 0;
      hi[z] = bb[z] = make_int4(0, 0, 0, 0);
      if (live && q0 + z * nt < units) {
        if (WHAT & 1) {
          s4[z] = __ldcg(Bf.part + q * kPartInts + kPartS);
          hi[z] = __ldcg(reinterpret_cast<const int4*>(Bf.part + q * kPartInts + kPartNe));
        }
        bb[z] = __ldcg(reinterpret_cast<const int4*>(Bf.part_bound + 2 * q));
      }
    }
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      r.S += s4[z];
      r.ne += hi[z].x;
      r.km = max(r.km, hi[z].y);
      if (WHAT & 1) ext_add_flat(r.b1, __int_as_float(bb[z].x), bb[z].y);
      if (WHAT & 2) ext_add_flat(r.b2, __int_as_float(bb[z].z), bb[z].w);
    }
  }
  if (WHAT & 1) {
    r.S = __reduce_add_sync(0xffffffffu, r.S);
    r.ne = __reduce_add_sync(0xffffffffu, r.ne);
    r.km = __reduce_max_sync(0xffffffffu, r.km);
    r.b1 = ext_warp_sum(r.b1);
  }
  if (WHAT & 2) r.b2 = ext_warp_sum(r.b2);
  return r;
}

__device__ __forceinline__ void merge_sums(UnitSums& u, const UnitSums& v) {
  u.S += v.S;
  u.ne += v.ne;
  u.km = max(u.km, v.km);
  ext_add_flat(u.b1, v.b1.m, v.b1.e);
  ext_add_flat(u.b2, v.b2.m, v.b2.e);
}

// The statistics of one instance from the parts of its sums, by one warp: lane 2 merges
// the parts of b2, the others those of b1; one square root and one division for all of
// them.  norm2: the operands' squared norms, which are then written too; null: the count
// kernel left the norms in the statistics.  Returns the split-flag binade (below:
// flag_prefix's sums); publish = false: only that.
__device__ __forceinline__ int write_stats(const Inst& in, const UnitSums* parts, int nparts,
                                           const double* norm2, bool full, bool publish,
                                           const double* below) {
  const int lane = threadIdx.x & 31;
  const bool prepped = norm2 == nullptr;
  PlanDevice* pd = in.pd;
  double x = 0.0;
  if (lane < 2 && publish) x = prepped ? __ldcg(lane ? &pd->norm_b : &pd->norm_a) : norm2[lane];
  UnitSums u = parts[0];
  // (parts formed for the binade only hold no b1)
  const ExtSum none{0.0f, 0};
  ExtSum bound = lane == 2 ? u.b2 : (full ? u.b1 : none);
#pragma unroll 1
  for (int v = 1; v < nparts; ++v) {
    const ExtSum y = lane == 2 ? parts[v].b2 : (full ? parts[v].b1 : none);
    ext_add_flat(bound, y.m, y.e);
    u.S += parts[v].S;
    u.ne += parts[v].ne;
    u.km = max(u.km, parts[v].km);
  }
  const double root = sqrt(lane == 2 ? ext_value(bound) : x);
  if (lane == 2 || !prepped) x = root;
  const double na = __shfl_sync(0xffffffffu, x, 0), nb = __shfl_sync(0xffffffffu, x, 1);
  const double bound2 = __shfl_sync(0xffffffffu, x, 2);
  const double ab = na * nb;
  const int m = in.split ? flag_pick(in, ab, bound2, below) : kFlagBinMin - 1;
  if (!full) return m;
  const double cube = (double)in.bm * (double)in.bk * (double)in.bn;
  const double quot = (lane == 0 ? 1.0 : (double)u.S) / (lane == 0 ? ab : cube);
  const double ratio = __shfl_sync(0xffffffffu, quot, 1);
  long long f = 0;
  if (in.split) {
    for (int b = lane; b < kFlagBins; b += 32)
      if (kFlagBinMin + b >= m) f += (long long)__ldcg(&pd->bin_cnt[b]);
    for (int off = 16; off > 0; off >>= 1) f += __shfl_xor_sync(0xffffffffu, f, off);
  }
  if (lane == 0 && publish) {
    pd->survivors = u.S;
    pd->max_tile = u.km;
    pd->nonempty = u.ne;
    if (!prepped) {
      pd->norm_a = na;
      pd->norm_b = nb;
      pd->inv_ab = ab > 0.0 ? quot : 0.0;
    }
    pd->bound1 = ext_value(bound);
    pd->bound2 = bound2;
    pd->valid_ratio = ratio;
    pd->flag_exp = m;
    pd->flagged = f;
  }
  return m;
}

// Part v of one instance's sums into shared memory, by one warp.
template <int WHAT>
__device__ __forceinline__ void stat_part(const Inst& in, const PlanBuffers& Bf, UnitSums* parts,
                                          int v, bool live = true) {
  const UnitSums u = unit_sums<WHAT>(in, Bf, v, live);
  if ((threadIdx.x & 31) != 0) return;
  if (WHAT & 1) {
    parts[v].S = u.S;
    parts[v].ne = u.ne;
    parts[v].km = u.km;
    parts[v].b1 = u.b1;
  }
  if (WHAT & 2) parts[v].b2 = u.b2;
}

// The statistics of one instance by a CTA of kStatWarps warps, or twice as many: then
// the second half forms b2.  The norms (not prepped) are added up beside.  publish = false:
// the same instructions without a load from the plan's buffers or a store to them.
__device__ __noinline__ void instance_stats(const Inst& in, const PlanBuffers& Bf, bool prepped,
                                            bool publish) {
  __shared__ UnitSums s_u[kStatWarps];
  __shared__ double s_below[32 * kBinsPerLane], s_norm2[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (!prepped && warp == kStatWarps - 1) {
    const double x = sum_norms2(Bf, in.count0, units_of(in), publish);
    if (lane < 2) s_norm2[lane] = x;
  }
  if (blockDim.x < 2 * 32 * kStatWarps)
    stat_part<3>(in, Bf, s_u, warp, publish);
  else if (warp < kStatWarps)
    stat_part<1>(in, Bf, s_u, warp, publish);
  else if (warp < 2 * kStatWarps)
    stat_part<2>(in, Bf, s_u, warp - kStatWarps, publish);
  if (warp == 0 && in.split) flag_prefix(in, s_below);
  __syncthreads();
  if (warp == 0) (void)write_stats(in, s_u, kStatWarps, prepped ? nullptr : s_norm2, true, publish, s_below);
}


// Screens of one staged row or column: whole words of 32 k (the tail holds
// zero norms) and two more, so that the rows start 16 bytes apart modulo the
// 128 bytes of a shared-memory wavefront.
__host__ __device__ __forceinline__ int staged_len(int bk) { return ((bk + 31) & ~31) + 2; }

// A unit's screens into shared memory (rows of A, then columns of B, their
// exponents relative to eT), by kCountThreads threads.  Units of four columns: a warp
// takes two rows of A and a quarter of B's (k, column) pairs of 32 k (whole 32-byte
// sectors), four times 32 k at a time: twelve loads in flight, one round trip up to 128
// blocks (rows and columns in turn took three).
__device__ __forceinline__ void stage_unit(const Inst& in, const Unit& u, Screen* sa, Screen* sb,
                                           int eT) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bk = in.bk, bn = in.bn, len = staged_len(bk), kpad = len - 2;
  const double* __restrict__ nA = in.nA;
  const double* __restrict__ nB = in.nB;
  if (u.cols == 4) {
    static_assert(kBandRows <= 2 * kCountWarps && kCountThreads == 128, "two rows, one pair");
    const int x1 = warp + kCountWarps, kb = tid >> 2, c = tid & 3;
    const bool has0 = warp < u.rows, has1 = x1 < u.rows;
    const double* a0 = nA + (int64_t)(u.r0 + warp) * bk;
    const double* a1 = a0 + (int64_t)kCountWarps * bk;
    const double* b0 = nB + u.j0 + c;
    for (int w0 = 0; w0 < kpad; w0 += 128) {
      double v[3][4];
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int k = w0 + 32 * z + lane, k2 = w0 + 32 * z + kb;
        v[0][z] = has0 && k < bk ? a0[k] : 0.0;
        v[1][z] = has1 && k < bk ? a1[k] : 0.0;
        v[2][z] = k2 < bk ? b0[(int64_t)k2 * bn] : 0.0;
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int k = w0 + 32 * z + lane, k2 = w0 + 32 * z + kb;
        if (w0 + 32 * z >= kpad) break;
        if (has0) sa[warp * len + k] = test_screen(v[0][z]);
        if (has1) sa[x1 * len + k] = test_screen(v[1][z]);
        Screen b = test_screen(v[2][z]);
        b.e -= eT;
        sb[c * len + k2] = b;
      }
    }
  } else {
    for (int x = warp; x < u.rows; x += kCountWarps) {
      const double* src = nA + (int64_t)(u.r0 + x) * bk;
#pragma unroll 8
      for (int k = lane; k < kpad; k += 32) sa[x * len + k] = test_screen(k < bk ? src[k] : 0.0);
    }
    for (int k = tid; k < kpad; k += kCountThreads)
#pragma unroll 4
      for (int c = 0; c < u.cols; ++c) {
        Screen b = test_screen(k < bk ? nB[(int64_t)k * bn + u.j0 + c] : 0.0);
        b.e -= eT;
        sb[c * len + k] = b;
      }
  }
}

// One CTA per unit.  A lane owns a tile, so nothing is reduced across lanes per
// tile and a word of the survivor mask is built in a register; about 25
// instructions per triple and lane, bound by issue and by the latency of staging
// (twelve loads in flight per thread).  The previous form (a warp per tile, lanes
// over k: ballots and some 150 instructions of reductions per tile) took 69 us at
// bk = 256 (1.7e7 triples), this one 40; for 256 uneven split instances 148 -> 55.
template <bool SPLIT, bool BAND>
__global__ void __launch_bounds__(kCountThreads)
    count_kernel(InstRef R, PlanBuffers Bf, int prepped, int stats) {
  extern __shared__ __align__(16) Screen s_scr[];   // [rows][len] of A, then [cols][len] of B
  __shared__ double s_bin_sum[SPLIT ? kFlagBins : 1];
  __shared__ int s_bin_cnt[SPLIT ? kFlagBins : 1];
  __shared__ float s_S[kCountWarps][32];
  __shared__ int s_E[kCountWarps][32], s_cnt[kCountWarps][32];
  __shared__ double s_inv;
  __shared__ bool s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ii = inst_of_unit(R, blockIdx.x);
  const Inst& in = R.at(ii);
  const int lu = blockIdx.x - in.count0;
  const Unit u = unit_at(in, lu);
  const int bm = in.bm, bk = in.bk, bn = in.bn;
  const bool split = SPLIT && in.split, band = BAND && in.band;
  const double* __restrict__ nA = in.nA;
  const double* __restrict__ nB = in.nB;
  const TestTau T = test_tau(in.T);
  asm volatile("" ::"r"(u.r0), "r"(u.rows), "r"(u.j0), "r"(u.cols), "r"(bk), "l"(nA), "l"(nB),
               "f"(T.lo), "l"(Bf.part), "l"(Bf.cnt), "l"(Bf.surv_mask), "l"(Bf.need_bits));
  pdl_wait();   // the above needs only the arguments and the instance table
  pdl_trigger();
  if (!prepped) {   // the accumulators of the fill kernel
    const int64_t gs = (int64_t)gridDim.x * kCountThreads;
    if (in.quant)
      for (int64_t g = (int64_t)blockIdx.x * kCountThreads + tid;
           g < Bf.need_words_a + Bf.need_words_b; g += gs)
        Bf.need_bits[g] = 0u;
    if (blockIdx.x == 0 && tid == 0) Bf.bdev->need_count = 0;
  }
  // the unit's screens (B's exponents relative to tau's)
  const int len = staged_len(bk), kpad = len - 2;
  Screen* sa = s_scr;
  Screen* sb = s_scr + u.rows * len;
  stage_unit(in, u, sa, sb, T.e);
  if (split) {
    for (int i = tid; i < kFlagBins; i += kCountThreads) {
      s_bin_sum[i] = 0.0;
      s_bin_cnt[i] = 0;
    }
  }
  __syncthreads();

  // lane -> tile (column by column inside the unit)
  const int c = lane / u.rows, r = lane - c * u.rows;
  const bool act = c < u.cols;
  const int i = u.r0 + r, j = u.j0 + c;
  const int64_t t = (int64_t)i * bn + j;
  const int nch = kpad >> 5;
  SkipSum sk{0.0f, 0.0f, kSkipStart};
  int count = 0;
  const double* pa = nA + (int64_t)i * bk;
  const double* pb = nB + j;
  if (act) {
    const TestTau Th = BAND ? test_tau(in.T_hi) : T;
    const int dhi = BAND ? T.e - Th.e : 0;
    const float4* ra = reinterpret_cast<const float4*>(sa + r * len);
    const float4* rb = reinterpret_cast<const float4*>(sb + c * len);
    for (int w = warp; w < nch; w += kCountWarps) {
      uint32_t mask = 0u, near = 0u;   // near: the FP64 product decides
#pragma unroll
      for (int o = 0; o < 4; ++o) {    // eight k: four 16-byte reads of each operand
        float q[8];
        int D[8];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const float4 a2 = ra[w * 16 + o * 4 + h], b2 = rb[w * 16 + o * 4 + h];
          q[2 * h] = __fmul_rn(a2.x, b2.x);
          q[2 * h + 1] = __fmul_rn(a2.z, b2.z);
          D[2 * h] = __float_as_int(a2.y) + __float_as_int(b2.y);
          D[2 * h + 1] = __float_as_int(a2.w) + __float_as_int(b2.w);
        }
#pragma unroll
        for (int z = 0; z < 8; ++z) {
          const uint32_t bit = 1u << (8 * o + z);
          const float v = screen_value(q[z], D[z]);
          bool s = v >= T.lo;                        // a near product: settled below
          if (s && v < T.hi) near |= bit;
          if (BAND && band) {
            const float v2 = screen_value(q[z], D[z] + dhi);
            if (v2 >= Th.hi) s = false;
            else if (v2 >= Th.lo) near |= s ? bit : 0u;
          }
          if (s) mask |= bit;
          if (s) D[z] = kSkipNone;
        }
        skip_add<8>(sk, q, D);
      }
      const int left = bk - w * 32;
      if (left < 32) mask &= (1u << left) - 1u;
      for (near &= mask; near; near &= near - 1u) {
        const int bit = __ffs(near) - 1, k = w * 32 + bit;
        const double p = __dmul_rn(pa[k], pb[(int64_t)k * bn]);
        bool s = !(p < in.T.tau);
        if (BAND && band && s) s = p < in.T_hi.tau;
        if (s) continue;
        mask &= ~(1u << bit);
        const Screen a = sa[r * len + k], b = sb[c * len + k];
        const float q1[1] = {__fmul_rn(a.m, b.m)};
        const int D1[1] = {a.e + b.e};
        skip_add<1>(sk, q1, D1);
      }
      count += __popc(mask);
      Bf.surv_mask[in.mask0 + t * nch + w] = mask;
    }
  }
  s_S[warp][lane] = __fadd_rn(sk.S, sk.C);
  s_E[warp][lane] = sk.Emax;
  s_cnt[warp][lane] = count;
  const int any = __syncthreads_or(count);
  if (prepped && ((split && any) || lu == 0)) {
    if (warp == kCountWarps - 1) {
      const double v = instance_norms(in, Bf, lu == 0);
      if (lane == 0) s_inv = v;
    }
    __syncthreads();
  }
  if (split && act) {   // surviving products by binade (a lane reads back its own words)
    const double inv = s_inv;
    for (int w = warp; w < nch && count > 0; w += kCountWarps)
      for (uint32_t bits = Bf.surv_mask[in.mask0 + t * nch + w]; bits; bits &= bits - 1u) {
        const int k = w * 32 + __ffs(bits) - 1;
        const double p = __dmul_rn(pa[k], pb[(int64_t)k * bn]);
        const int bin = rel_bin(p, inv);
        atomicAdd(&s_bin_sum[bin - kFlagBinMin], p);
        atomicAdd(&s_bin_cnt[bin - kFlagBinMin], 1);
      }
  }
  if (split && any) __syncthreads();
  if (warp == 0) {
    // the tile's totals over the warps (fixed order), then the unit's
    count = 0;
    int emax = kSkipNone;
#pragma unroll
    for (int w = 0; w < kCountWarps; ++w) {
      count += s_cnt[w][lane];
      emax = max(emax, s_E[w][lane]);
    }
    const float S = skip_total(s_S, s_E, lane, emax);
    const ExtSum tot = S > 0.0f ? ExtSum{S, emax + T.e} : ExtSum{0.0f, 0};
    const ExtSum b1 = ext_warp_sum_fast(tot);
    const ExtSum b2 = ext_warp_sum_fast(ExtSum{__fmul_rn(tot.m, tot.m), 2 * tot.e});
    const int64_t g = in.tile0 + t;
    if (act) {
      Bf.cnt[g] = count;
      if (R.count > 1) Bf.tile_inst[g] = ii;
    }
    const int key = count > 0 ? order_key(count) : 0;
    int val = __reduce_add_sync(0xffffffffu, count);        // lane kPartS
#pragma unroll
    for (int q = 1; q < kOrderKeys; ++q) {
      const int n = __popc(__ballot_sync(0xffffffffu, key == q));
      if (lane == q) val = n;
    }
    const int ne = __popc(__ballot_sync(0xffffffffu, count > 0));
    const int km = __reduce_max_sync(0xffffffffu, count);
    if (lane == kPartNe) val = ne;
    if (lane == kPartMax) val = km;
    if (lane < kPartInts) {
      Bf.part[(int64_t)blockIdx.x * kPartInts + lane] = lane <= kPartMax ? val : 0;
      if (Bf.group_shift && lane < kPartNe)
        atomicAdd(&Bf.group[(int64_t)(blockIdx.x >> Bf.group_shift) * kPartInts + lane], val);
    }
    if (lane == 0)
      *reinterpret_cast<int4*>(Bf.part_bound + 2 * (int64_t)blockIdx.x) =
          make_int4(__float_as_int(b1.m), b1.e, __float_as_int(b2.m), b2.e);
  } else if (warp == 1 && !prepped) {
    // this unit's share of the squared norms of A and B
    const int units = units_of(in);
    const int64_t na = (int64_t)bm * bk, nb = (int64_t)bk * bn;
    const int64_t la = (na + units - 1) / units, lb = (nb + units - 1) / units;
    double qa = 0.0, qb = 0.0;
    for (int64_t x = lu * la + lane; x < min(na, (lu + 1) * la); x += 32) qa = __fma_rn(nA[x], nA[x], qa);
    for (int64_t x = lu * lb + lane; x < min(nb, (lu + 1) * lb); x += 32) qb = __fma_rn(nB[x], nB[x], qb);
    for (int off = 16; off > 0; off >>= 1) {
      qa += __shfl_xor_sync(0xffffffffu, qa, off);
      qb += __shfl_xor_sync(0xffffffffu, qb, off);
    }
    if (lane == 0) {
      Bf.part_a[blockIdx.x] = qa;
      Bf.part_b[blockIdx.x] = qb;
    }
  }
  if (split && any) {
    for (int q = tid; q < kFlagBins; q += kCountThreads) {
      if (s_bin_cnt[q]) {
        atomicAdd(&in.pd->bin_sum[q], s_bin_sum[q]);
        atomicAdd(&in.pd->bin_cnt[q], (unsigned long long)s_bin_cnt[q]);
      }
    }
  }
  if (!stats) return;
  // the last unit of the instance forms its statistics
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&in.pd->ticket, 1u) == (unsigned)units_of(in) - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  instance_stats(in, Bf, true, true);
}

// ---------------------------------------------------------------------------
// Certified reference tau: the largest grid point -60 + 60 x / 2^36 (log10 of tau
// relative to ||A|| ||B||) whose skipped-product bound bound2 is at most ref_rel
// ||A|| ||B||, by the 36 decisions of a bisection, four of them per pass: a pass
// forms bound2 at the 15 inner points of the current interval at once (a triple's
// product falls between two of them and is added to that gap's sum of its tile;
// a tile's bound at a point is the sum of the gaps below it), and its last CTA
// takes the four decisions and lays out the next points.  No host round trip in
// between: 36 counting half-plans with a synchronisation each took 1.0 ms at 64
// blocks per side, this takes 0.11 (nine passes of about 12 us each).
// ---------------------------------------------------------------------------

// Grid point x as a threshold.
__device__ __forceinline__ double cert_tau(double ab, long long x) {
  return ab * exp10(ldexp((double)(15 * (x - (1ll << 36))), -34));
}

// Norms (after prep), the first points and cleared sums: one warp.
__global__ void cert_init_kernel(InstRef R, PlanBuffers Bf, double ref_rel) {
  pdl_wait();
  pdl_trigger();
  const Inst& in = R.at(0);
  CertState* cs = Bf.cert;
  const int lane = threadIdx.x;
  (void)instance_norms(in, Bf, true);
  __syncwarp();
  const double ab = in.pd->norm_a * in.pd->norm_b;
  if (lane < kCertPoints) {
    cs->tau[lane] = cert_tau(ab, (long long)(lane + 1) << 32);
    cs->sum[lane] = 0.0;
  }
  if (lane == 0) {
    cs->lo = 0;
    cs->step = 1ll << 32;
    cs->ab = ab;
    cs->limit = ref_rel * ab;
    cs->ticket = 0u;
  }
}

// One pass: one CTA per unit.
__global__ void __launch_bounds__(kCountThreads) cert_pass_kernel(InstRef R, PlanBuffers Bf) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) Screen s_scr[];
  __shared__ double s_tau[kCertPoints];
  __shared__ int s_exp[kCertPoints];
  __shared__ Screen s_pt[kCertPoints];
  __shared__ float2 s_cum[kCertPoints][40];   // a tile's sum up to each point: value, exponent
  // sums of the gaps, relative to 2^s_exp, with the rounding errors of their additions
  __shared__ float2 s_gap[kCountWarps][kCertPoints][32];
  __shared__ float s_S[kCountWarps][32];
  __shared__ int s_E[kCountWarps][32];
  __shared__ bool s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Inst& in = R.at(0);
  CertState* cs = Bf.cert;
  const Unit u = unit_at(in, blockIdx.x);
  const int bk = in.bk, bn = in.bn, len = staged_len(bk);
  Screen* sa = s_scr;
  Screen* sb = s_scr + u.rows * len;
  stage_unit(in, u, sa, sb, 0);
  if (tid < kCertPoints) {
    s_tau[tid] = cs->tau[tid];
    s_pt[tid] = test_screen(cs->tau[tid]);
    s_exp[tid] = s_pt[tid].e;
  }
  for (int x = tid; x < kCountWarps * kCertPoints * 32; x += kCountThreads)
    (&s_gap[0][0][0])[x] = make_float2(0.0f, 0.0f);
  __syncthreads();
  // FP32 windows around the lowest and the highest point (1 -+ 2^-20): products
  // outside them need no FP64
  const Screen t0 = test_screen(s_tau[0]), t1 = test_screen(s_tau[kCertPoints - 1]);
  constexpr float kBelow = 1.0f - 9.5367431640625e-7f, kAbove = 1.0f + 9.5367431640625e-7f;
  const float lo0 = t0.m * kBelow, hi1 = t1.m * kAbove;
  const int c = lane / u.rows, r = lane - c * u.rows;
  const bool act = c < u.cols;
  const int i = u.r0 + r, j = u.j0 + c;
  SkipSum sk{0.0f, 0.0f, kSkipStart};
  if (act) {
    const double* pa = in.nA + (int64_t)i * bk;
    const double* pb = in.nB + j;
    for (int k0 = warp * 8; k0 < bk; k0 += 8 * kCountWarps) {
      float q[8];
      int D[8];
#pragma unroll
      for (int z = 0; z < 8; ++z) {
        const int k = k0 + z;
        const Screen a = sa[r * len + k], b = sb[c * len + k];
        const float q0 = __fmul_rn(a.m, b.m);
        const int E = a.e + b.e;
        q[z] = q0;
        D[z] = E;                                                 // below every point
        if (screen_value(q0, E - t0.e) < lo0) continue;
        D[z] = kSkipNone;                                         // survives the lowest point
        if (k >= bk || screen_value(q0, E - t1.e) >= hi1) continue;
        // between the points: how many are at or below the product; FP64 (and the
        // norms from memory) only next to a point
        int gap = 0;
        bool near = false;
#pragma unroll
        for (int b2 = 8; b2 > 0; b2 >>= 1) {
          if (gap + b2 > kCertPoints) continue;
          const Screen t = s_pt[gap + b2 - 1];
          const float v = screen_value(q0, E - t.e);
          if (v >= t.m * kAbove) gap += b2;
          else if (v >= t.m * kBelow) near = true;
        }
        if (near) {
          const double p = __dmul_rn(pa[k], pb[(int64_t)k * bn]);
          gap = 0;
#pragma unroll
          for (int b2 = 8; b2 > 0; b2 >>= 1)
            if (gap + b2 <= kCertPoints && !(p < s_tau[gap + b2 - 1])) gap += b2;
        }
        if (gap == 0) D[z] = E;
        else if (gap < kCertPoints) {
          float2& g = s_gap[warp][gap - 1][lane];
          float2 t;
          two_sum(g.x, __fmul_rn(q0, pow2f_or_zero(min(0, E - s_exp[gap] - 2))), t.x, t.y);
          g = make_float2(t.x, __fadd_rn(g.y, t.y));
        }
      }
      skip_add<8>(sk, q, D);
    }
  }
  s_S[warp][lane] = __fadd_rn(sk.S, sk.C);
  s_E[warp][lane] = sk.Emax;
  __syncthreads();
  for (int p = warp; p < kCertPoints - 1; p += kCountWarps) {   // every gap over the warps
    float g[kCountWarps];
#pragma unroll
    for (int w = 0; w < kCountWarps; ++w) g[w] = __fadd_rn(s_gap[w][p][lane].x, s_gap[w][p][lane].y);
    s_gap[0][p][lane].x = __fadd_rn(__fadd_rn(g[0], g[1]), __fadd_rn(g[2], g[3]));
  }
  __syncthreads();
  // the tiles' sums up to every point (a lane per tile), then the points' sums of
  // squares, eight threads each, in the order of a warp's butterfly (both by one warp,
  // a point after the other, took 11 of the 24 us that a pass then lasted)
  if (warp == 0) {
    int emax = kSkipNone;
#pragma unroll
    for (int w = 0; w < kCountWarps; ++w) emax = max(emax, s_E[w][lane]);
    const float S = skip_total(s_S, s_E, lane, emax);
    ExtSum cum = S > 0.0f ? ExtSum{S, emax} : ExtSum{0.0f, 0};
    float low = 0.0f;   // what the additions to cum.m have rounded off
    for (int p = 0; p < kCertPoints; ++p) {
      if (p > 0) ext_add_two(cum, low, s_gap[0][p - 1][lane].x, s_exp[p] + 2);
      s_cum[p][lane] = make_float2(__fadd_rn(cum.m, low), __int_as_float(cum.e));
    }
  }
  __syncthreads();
  static_assert(kCountThreads >= 8 * (kCertPoints + 1), "eight threads per point");
  const int pt = tid >> 3, sub = tid & 7;
  if (warp < (kCertPoints + 1) / 4) {   // whole warps: point kCertPoints is empty
    constexpr int kNone = -(1 << 29);
    float sq[4];
    int e[4], eb[4], emax = kNone;
#pragma unroll
    for (int z = 0; z < 4; ++z) {   // tiles sub, sub + 16, sub + 8, sub + 24
      const float2 x = pt < kCertPoints ? s_cum[pt][sub + (z & 1) * 16 + (z >> 1) * 8] : make_float2(0.0f, 0.0f);
      // a sum's own binade keeps its square inside the FP32 range
      const int own = x.x > 0.0f ? fexp(x.x) : 0;
      const float m = x.x > 0.0f ? ldexpf(x.x, -own) : 0.0f;
      sq[z] = __fmul_rn(m, m);
      e[z] = 2 * (__float_as_int(x.y) + own);
      eb[z] = sq[z] > 0.0f ? e[z] + fexp(sq[z]) : kNone;
      emax = max(emax, eb[z]);
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, off));
    float v[4];
#pragma unroll
    for (int z = 0; z < 4; ++z)
      v[z] = eb[z] != kNone && eb[z] >= emax - 40 ? sq[z] * pow2f(e[z] - (emax - 40)) : 0.0f;
    float sum = (v[0] + v[1]) + (v[2] + v[3]);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    ExtSum r{sum, emax - 40};
    while (r.m >= 1099511627776.0f) {   // keep the mantissa below 2^40
      r.m *= pow2f(-40);
      r.e += 40;
    }
    if (sub == 0 && sum > 0.0f) atomicAdd(&cs->sum[pt], ext_value(r));
  }
  // the last CTA takes the pass's four decisions
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&cs->ticket, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!s_last || warp != 0) return;
  __threadfence();
  const double x = sqrt(lane < kCertPoints ? __ldcg(&cs->sum[lane]) : 0.0);
  const unsigned ok = __ballot_sync(0xffffffffu, lane < kCertPoints && x <= cs->limit);
  int at = 0;                        // point 0 is the interval's lower end
#pragma unroll
  for (int b2 = 8; b2 > 0; b2 >>= 1)
    if ((ok >> (at + b2 - 1)) & 1u) at += b2;
  const long long step = cs->step, lo = cs->lo + at * step, next = step >> 4;
  __syncwarp();
  if (lane < kCertPoints) {
    if (next > 0) cs->tau[lane] = cert_tau(cs->ab, lo + (lane + 1) * next);
    cs->sum[lane] = 0.0;
  }
  if (lane == 0) {
    cs->lo = lo;
    cs->step = next;
    cs->ticket = 0u;
  }
}

// Sum of squared tile norms over the tiles with survivors (one CTA).
__global__ void __launch_bounds__(1024) tile_norms_kernel(InstRef R, PlanBuffers Bf) {
  pdl_wait();
  __shared__ double s_w[32];
  const Inst& in = R.at(0);
  const int64_t tiles = (int64_t)in.bm * in.bn;
  double x = 0.0;
#pragma unroll 4
  for (int64_t t = threadIdx.x; t < tiles; t += 1024)
    if (Bf.cnt[t] > 0) x = __fma_rn(in.nC[t], in.nC[t], x);
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x < 32) {
    x = s_w[threadIdx.x];
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    if (threadIdx.x == 0) Bf.cert->norm = sqrt(x);
  }
}

// Histogram bin of r = fl(fl(na nb) * inv) (one FP64 multiply, no other rounding):
// floor(-log2 r) clamped to [0, 63]; r = 0 or NaN goes to bin 63, +Inf to 0.
__device__ __forceinline__ int hist_bin_exact(double p, double inv) {
  const double r = __dmul_rn(p, inv);
  if (!(r > 0.0)) return kHistBins - 1;
  if (isinf(r)) return 0;
  int e;
  const double m = frexp(r, &e);          // r = m 2^e, m in [0.5, 1)
  const int t = -e + (m == 0.5 ? 1 : 0);
  return t < 0 ? 0 : (t > kHistBins - 1 ? kHistBins - 1 : t);
}

// The same bin from the screen forms in FP32; the FP64 form decides whenever
// the FP32 product lies within 2^-20 of a power of two.
__device__ __forceinline__ int hist_bin_screened(Screen a, Screen b, float inv_m, int inv_e,
                                                 const double* pa, const double* pb, double inv) {
  if ((a.e == kZeroExp || b.e == kZeroExp) && inv > 0.0 && !isinf(inv)) return kHistBins - 1;
  if (a.e == kNonFiniteExp || b.e == kNonFiniteExp || a.e == kZeroExp || b.e == kZeroExp ||
      !(inv > 0.0) || isinf(inv))
    return hist_bin_exact(__dmul_rn(*pa, *pb), inv);
  const float q = __fmul_rn(__fmul_rn(a.m, b.m), inv_m);   // in [0.125, 1]
  const uint32_t frac = __float_as_uint(q) & 0x7fffffu;
  if (frac < 8u || frac > 0x7fffffu - 8u) return hist_bin_exact(__dmul_rn(*pa, *pb), inv);
  // r = q' 2^(b0) with q' in (1, 2) not a power of two: floor(-log2 r) = -b0 - 1
  const int b0 = a.e + b.e + inv_e + ((int)((__float_as_uint(q) >> 23) & 0xffu) - 127);
  const int t = -b0 - 1;
  return t < 0 ? 0 : (t > kHistBins - 1 ? kHistBins - 1 : t);
}

// Histogram of every triple of every instance: one warp per output tile,
// lanes over k; equal bins of a warp are merged with match_any before the
// shared-memory atomics, CTA totals go to the instance's global bins.
__global__ void __launch_bounds__(kHistWarps * 32)
    hist_kernel(InstRef R, PlanBuffers Bf) {
  __shared__ unsigned int s_hist[kHistBins];
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
  const int ii = inst_of_unit(R, blockIdx.x);
  const Inst& in = R.at(ii);
  const int bk = in.bk, bn = in.bn;
  const double* nA = in.nA;
  const double* nB = in.nB;
  for (int q = threadIdx.x; q < kHistBins; q += blockDim.x) s_hist[q] = 0u;
  __syncthreads();
  __shared__ double s_inv;
  if (warp == 0) {
    const double v = instance_norms(in, Bf, blockIdx.x == in.count0);
    if (lane == 0) s_inv = v;
  }
  __syncthreads();
  const double inv = s_inv;
  int inv_e;
  const float inv_m = (float)frexp(inv, &inv_e);
  const int64_t tiles = (int64_t)in.bm * bn;
  const int64_t lt0 = (int64_t)(blockIdx.x - in.count0) * kHistTiles;
  for (int r = 0; r < kHistTiles / kHistWarps; ++r) {
    const int64_t t = lt0 + warp + (int64_t)r * kHistWarps;
    if (t >= tiles) break;
    const int i = (int)(t / bn), j = (int)(t % bn);
    const Screen* ra = Bf.sA + in.ablk0 + (int64_t)i * bk;
    const Screen* rb = Bf.sBT + in.bblk0 + (int64_t)j * bk;
    for (int k0 = 0; k0 < bk; k0 += 32) {
      const int k = k0 + lane;
      const bool act = k < bk;
      int bin = kHistBins;   // inactive lanes: a bin of their own
      if (act)
        bin = hist_bin_screened(ra[k], rb[k], inv_m, inv_e, nA + (int64_t)i * bk + k,
                                nB + (int64_t)k * bn + j, inv);
      const unsigned same = __match_any_sync(0xffffffffu, bin);
      if (act && lane == __ffs(same) - 1) atomicAdd(&s_hist[bin], (unsigned)__popc(same));
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < kHistBins; q += blockDim.x)
    if (s_hist[q]) atomicAdd(&in.pd->hist[q], s_hist[q]);
}

__device__ __forceinline__ void add4(int4& a, const int4& b) {
  a.x += b.x;
  a.y += b.y;
  a.z += b.z;
  a.w += b.w;
}
__device__ __forceinline__ int4 shfl_xor4(const int4& v, int off) {
  return make_int4(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off),
                   __shfl_xor_sync(0xffffffffu, v.z, off), __shfl_xor_sync(0xffffffffu, v.w, off));
}

// A lane's tile of a unit: lane c * rows + r has row r, column c.
struct FillLane {
  Unit u;
  int ii, nch, c, r, i, j;
  bool act;
  int64_t g, mask;   // tile; its first mask word
};

__device__ __forceinline__ FillLane fill_lane(const InstRef& R, int un) {
  FillLane f;
  f.ii = inst_of_unit(R, un);
  const Inst& in = R.at(f.ii);
  f.u = unit_at(in, un - in.count0);
  f.nch = (in.bk + 31) >> 5;
  const int lane = threadIdx.x & 31;
  f.c = lane / f.u.rows;
  f.r = lane - f.c * f.u.rows;
  f.act = f.c < f.u.cols;
  f.i = f.u.r0 + f.r;
  f.j = f.u.j0 + f.c;
  const int64_t t = (int64_t)f.i * in.bn + f.j;
  f.g = in.tile0 + t;
  f.mask = in.mask0 + t * f.nch;
  return f;
}

// Puts the blocks of A and B that a unit's triples use on the list of needed blocks, by
// one warp.
__device__ __forceinline__ void need_blocks(const InstRef& R, const PlanBuffers& Bf, const FillLane& f) {
  const Inst& in = R.at(f.ii);
  if (!in.quant) return;
  const int lane = threadIdx.x & 31, bk = in.bk, nch = f.nch;
  for (int w0 = 0; w0 < nch; w0 += 4) {
    uint32_t word[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      word[q] = f.act && w0 + q < nch ? __ldcg(Bf.surv_mask + f.mask + w0 + q) : 0u;
    // the blocks of A and B that the unit's triples use: lane x < rows holds row x
    // of A, the next cols lanes the columns of B, 32 k per word; the four words'
    // round trips go out together
    uint32_t mine[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      mine[q] = 0u;
      if (!__any_sync(0xffffffffu, word[q] != 0u)) continue;
      for (int x = 0; x < f.u.rows + f.u.cols; ++x) {
        const bool in_set = x < f.u.rows ? f.r == x : f.c == x - f.u.rows;
        const uint32_t o = __reduce_or_sync(0xffffffffu, in_set ? word[q] : 0u);
        if (lane == x) mine[q] = o;
      }
    }
    const bool isB = lane >= f.u.rows;
    const int bi = isB ? f.u.j0 + lane - f.u.rows : f.u.r0 + lane;   // column of B / row of A
    uint32_t* w = Bf.need_bits + (isB ? Bf.need_words_a + in.needb0 : in.needa0) +
                  (int64_t)bi * nch + w0;
    uint32_t fresh[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)   // a plain read first: a bit once set stays set
      fresh[q] = mine[q] ? mine[q] & ~__ldcg(w + q) : 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (fresh[q]) fresh[q] = mine[q] & ~atomicOr(w + q, mine[q]);
    int n = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) n += __popc(fresh[q]);
    int end = n;
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, end, off);
      if (lane >= off) end += y;
    }
    const int total = __shfl_sync(0xffffffffu, end, 31);
    if (total > 0) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&Bf.bdev->need_count, total);
      at = __shfl_sync(0xffffffffu, at, 0) + end - n;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        for (; fresh[q]; fresh[q] &= fresh[q] - 1u) {
          const int64_t k = (w0 + q) * 32 + __ffs(fresh[q]) - 1;
          Bf.need_list[at++] = isB ? (uint32_t)(in.bblk0 + k * in.bn + bi) | 0x80000000u
                                   : (uint32_t)(in.ablk0 + (int64_t)bi * bk + k);
        }
    }
  }
}

// Work queues of `per_cta` consecutive units per CTA (kUnitWarps warps per
// unit).  The first slots come from the totals of all units (or of the groups
// of units): a few KB from L2 per CTA, instead of a scan kernel of its own
// between count and fill.  Count and fill together, without the memset, prep and
// finalize launches they replace: 30 -> 11 us at 32 blocks per side, 48 -> 17 at
// 64 (10% of the triples survive), 169 -> 26 at 128 (half of them survive: one
// atomic per word of needed blocks instead of two per triple).  Then bound by
// instruction fetches and round trips: what needs only the arguments is done while the
// count kernel runs, the list of needed blocks is made beside the scan, short lists
// are written by a lane per tile.  Inside the product's chain the kernel takes 4.7 us at
// 32 blocks per side (7.1 before), 5.5 for 4 x 18 x 100 blocks (11.4), 12 at 128 with
// split flags (21).
__global__ void __launch_bounds__(kFillThreads)
    fill_kernel(InstRef R, PlanBuffers Bf, int per_cta, int prepped) {
  constexpr int kMaxPer = 32;
  __shared__ __align__(16) int s_red[kFillWarps][2 * kPartInts];
  __shared__ int s_base[kPartInts];          // buckets 1 .. 11: first slots of the CTA's units
  __shared__ int s_nonempty;                 // non-empty tiles of all units
  __shared__ int s_part[kMaxPer][kPartInts];
  __shared__ UnitSums s_u[kStatWarps], s_w[kFillWarps];
  __shared__ double s_below[kFillWarps][32 * kBinsPerLane];
  __shared__ int s_m[kMaxPer];               // split flag binade of instance ii0 + z
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int U = Bf.count_ctas;
  const int u0 = blockIdx.x * per_cta, u1 = min(U, u0 + per_cta);
  const int sub = warp / kUnitWarps, wu = warp % kUnitWarps;
  // what needs only the arguments and the instance table, while the count kernel runs
  const int ii0 = u0 < U ? inst_of_unit(R, u0) : 0;
  const int first = R.at(ii0).count0;   // of u0's instance
  FillLane f = fill_lane(R, min(u0 + sub, U - 1));
  asm volatile("" ::"r"(f.ii), "r"(f.nch), "r"(f.i), "r"(f.j), "l"(f.g), "l"(f.mask), "r"(first),
               "l"(Bf.cnt), "l"(Bf.surv_mask), "l"(Bf.part), "l"(Bf.group), "l"(Bf.order),
               "l"(Bf.tile_beg), "l"(Bf.k_idx), "l"(Bf.need_bits), "l"(Bf.need_list), "l"(Bf.bdev));
  if (u0 >= U) {   // no split modes: one more CTA per instance forms its statistics
    // twice: the first pass, while the count kernel still runs, only fetches the
    // instructions (it loads nothing that kernel writes)
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      if (pass == 1) {
        pdl_wait();
        pdl_trigger();
      }
      instance_stats(R.at(blockIdx.x - (U + per_cta - 1) / per_cta), Bf, prepped != 0, pass == 1);
      __syncthreads();
    }
    return;
  }
  pdl_wait();
  pdl_trigger();
  // the first unit of this warp: its counts and first words, on their way while
  // the totals are added up
  int count_next = 0;
  uint32_t word_next[4] = {0u, 0u, 0u, 0u};
  if (u0 + sub < u1 && f.act) {
    count_next = __ldcg(Bf.cnt + f.g);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < f.nch) word_next[q] = __ldcg(Bf.surv_mask + f.mask + q);
  }
  const int ii1 = R.any_split ? inst_of_unit(R, u1 - 1) : ii0;
  // split modes: the flag binade of every instance with units here, one warp per
  // instance; the sums of a lone one are formed by the upper warps while the lower
  // ones add up the totals, and finished below
  const bool lone = R.any_split && ii0 == ii1;
  if (R.any_split && !lone) {
    for (int z = warp; z <= ii1 - ii0; z += kFillWarps) {
      const Inst& in = R.at(ii0 + z);
      UnitSums u = unit_sums<3>(in, Bf, 0);
      for (int v = 1; v < kStatWarps && 32 * v < units_of(in); ++v)
        merge_sums(u, unit_sums<3>(in, Bf, v));
      if (in.split) flag_prefix(in, s_below[warp]);
      if (lane == 0) s_w[warp] = u;
      __syncwarp();
      const int m = write_stats(in, s_w + warp, 1, nullptr, in.count0 >= u0, true, s_below[warp]);
      if (lane == 0) s_m[z] = m;
    }
  }
  // the roles up to the scan's result: the first warps add up the totals (warp 0
  // finishes them), the last kStatWarps form a lone instance's statistics, and the
  // kNeedWarps before the last list the blocks that the CTA's units need, which
  // depends on neither: they only arrive at the barrier before the scan, and wait for
  // its result on a barrier of their own
  constexpr int kNeedWarps = kFillWarps / kUnitWarps, kNeed0 = kFillWarps - 1 - kNeedWarps;
  const bool needs = warp >= kNeed0 && warp < kNeed0 + kNeedWarps;
  const int scan_warps = lone ? kFillWarps - kStatWarps : kNeed0;
  const int scan_threads = scan_warps * 32;
  if (lone && warp >= scan_warps) {   // the counts and b1: for the CTA that writes them
    const Inst& in = R.at(ii0);
    if (in.count0 >= u0) stat_part<3>(in, Bf, s_u, warp - scan_warps);
    else stat_part<2>(in, Bf, s_u, warp - scan_warps);
  }
  if (warp < scan_warps) {
    // four threads per unit, a quarter of its slots each, eight units' loads at a time:
    // the buckets' totals over all units and over those before u0; survivors of u0's
    // instance before u0.  (A thread per unit with all slots in registers is
    // straight-line code of 24 warp reductions: its instruction fetches alone took 1 us.)
    static_assert(kPartInts == 16 && kPartS == 0, "slots by quarters");
    const int quarter = tid & 3, step = scan_threads / 4, gs = Bf.group_shift;
    const int n = (U + (1 << gs) - 1) >> gs, ub = u0 >> gs, lb = first >> gs;
    const int4* units = reinterpret_cast<const int4*>(Bf.part) + quarter;
    const int4* src = gs ? reinterpret_cast<const int4*>(Bf.group) + quarter : units;
    int4 tot = make_int4(0, 0, 0, 0), bef = tot;
    for (int q0 = tid >> 2; q0 < n; q0 += 8 * step) {
      int4 x[8];
#pragma unroll
      for (int z = 0; z < 8; ++z)
        x[z] = q0 + z * step < n ? __ldcg(src + (int64_t)(q0 + z * step) * 4) : make_int4(0, 0, 0, 0);
#pragma unroll
      for (int z = 0; z < 8; ++z) {
        const int q = q0 + z * step;
        add4(tot, x[z]);
        if (quarter == 0 && q < lb) x[z].x = 0;
        if (q < ub) add4(bef, x[z]);
      }
    }
    if (gs) {
      for (int q = (ub << gs) + (tid >> 2); q < u0; q += step) add4(bef, __ldcg(units + (int64_t)q * 4));
      if (quarter == 0)
        for (int q = (lb << gs) + (tid >> 2); q < first; q += step) bef.x -= __ldcg(units + (int64_t)q * 4).x;
    }
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
      add4(tot, shfl_xor4(tot, off));
      add4(bef, shfl_xor4(bef, off));
    }
    if (lane < 4) {
      reinterpret_cast<int4*>(s_red[warp])[lane] = tot;
      reinterpret_cast<int4*>(s_red[warp])[4 + lane] = bef;
    }
    for (int x = tid; x < (u1 - u0) * kPartInts; x += scan_threads)
      s_part[x / kPartInts][x % kPartInts] = __ldcg(Bf.part + (int64_t)u0 * kPartInts + x);
  }
  if (needs) {
    asm volatile("bar.arrive 1, %0;" ::"n"(kFillThreads) : "memory");
    for (int un = u0 + warp - kNeed0; un < u1; un += kNeedWarps) need_blocks(R, Bf, fill_lane(R, un));
  } else if (lone && warp == scan_warps) {   // beside the last warp, which waits for it
    asm volatile("bar.arrive 1, %0;" ::"n"(kFillThreads) : "memory");
    flag_prefix(R.at(ii0), s_below[0]);
    asm volatile("bar.arrive 4, 64;" ::: "memory");
  } else {
    asm volatile("bar.sync 1, %0;" ::"n"(kFillThreads) : "memory");
  }
  if (warp == kFillWarps - 1 && lone) {
    const Inst& in = R.at(ii0);   // the CTA of its first unit also writes its statistics
    asm volatile("bar.sync 4, 64;" ::: "memory");
    const int m = write_stats(in, s_u, kStatWarps, nullptr, in.count0 >= u0, true, s_below[0]);
    if (lane == 0) s_m[0] = m;
  }
  if (warp == 0) {
    // lane q: bucket q's total and the part before u0; largest bucket first
    int a = 0, b = 0;
    if (lane < kOrderKeys)
      for (int w = 0; w < scan_warps; ++w) {
        if (lane != kPartS) a += s_red[w][lane];
        b += s_red[w][kPartInts + lane];
      }
    int upto = a;   // non-empty tiles in the buckets up to this lane's
#pragma unroll
    for (int off = 1; off < 16; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, upto, off);
      if (lane >= off) upto += y;
    }
    const int all = __shfl_sync(0xffffffffu, upto, 15);
    const int below = all - upto;   // in those above it
    const int ne_before = __reduce_add_sync(0xffffffffu, lane >= 1 ? b : 0);
    if (lane < kOrderKeys) s_base[lane] = lane == kPartS ? b : below + b;
    if (lane == kPartNe) s_base[lane] = ne_before;
    if (lane == 0) {
      s_nonempty = all;
      if (blockIdx.x == 0) Bf.bdev->nonempty = all;
    }
  }
  constexpr int kOthers = kFillThreads - 32 * kNeedWarps, kLate = 64 + 32 * kNeedWarps;
  if (needs) {
    asm volatile("bar.sync 3, %0;" ::"n"(kLate) : "memory");
  } else {
    if (warp == 0 || warp == kFillWarps - 1) asm volatile("bar.arrive 3, %0;" ::"n"(kLate) : "memory");
    asm volatile("bar.sync 2, %0;" ::"n"(kOthers) : "memory");
  }
  const int nonempty = s_nonempty;
  for (int un = u0 + sub; un < u1; un += kFillWarps / kUnitWarps) {
    const bool first_round = un == u0 + sub;
    if (!first_round) f = fill_lane(R, un);
    const int ii = f.ii, nch = f.nch, r = f.r, i = f.i, j = f.j;
    const Inst& in = R.at(ii);
    const int bk = in.bk, bn = in.bn;
    const Unit u = f.u;
    const bool act = f.act;
    const int64_t g = f.g;
    const int count = first_round ? count_next : (act ? Bf.cnt[g] : 0);
    // lane q: the unit's first slot in bucket q, lane 0: survivors before it in
    // its instance, lane kPartNe: non-empty tiles before it
    int base = 0;
    if (lane < kPartInts) {
      base = s_base[lane];
      const int q0 = max(u0, in.count0);   // the CTA's first unit of this instance
      if (lane == kPartS && in.count0 > u0) base = 0;
      for (int q = lane == kPartS ? q0 : u0; q < un; ++q) base += s_part[q - u0][lane];
    }
    int incl = count;
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += y;
    }
    const int beg = (int)in.kidx0 + __shfl_sync(0xffffffffu, base, kPartS) + incl - count;
    const int key = count > 0 ? order_key(count) : 0;
    const unsigned same = __match_any_sync(0xffffffffu, key);
    const int slot0 = __shfl_sync(0xffffffffu, base, key);
    const unsigned ne_mask = __ballot_sync(0xffffffffu, count > 0);
    const int ne0 = __shfl_sync(0xffffffffu, base, kPartNe);
    const unsigned lower = (1u << lane) - 1u;
    if (wu == 0 && act) {
      Bf.tile_beg[g] = beg;
      if (count > 0) {
        Bf.order[slot0 + __popc(same & lower)] = (int)g;
      } else {
        const int64_t pos = in.tile0 + (int64_t)u.r0 * bn + (int64_t)j * u.rows + r;
        Bf.order[nonempty + (pos - (ne0 + __popc(ne_mask & lower)))] = (int)g;
      }
    }
    // expand the bitmask words.  Up to 16 entries per tile on average: a lane per tile
    // (a warp per tile spends 900 cycles on each, however few its entries are); more: a
    // warp per tile, whose stores are coalesced
    const bool few = __shfl_sync(0xffffffffu, incl, 31) <= 16 * 32;
    const uint32_t* mrow = Bf.surv_mask + f.mask;
    const int split = in.split;
    const int m = split ? s_m[ii - ii0] : 0;
    const double inv = split && ne_mask ? in.pd->inv_ab : 0.0;
    int cursor = beg;
    for (int w0 = 0; w0 < nch; w0 += 4) {
      uint32_t word[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        word[q] = first_round && w0 == 0 ? word_next[q]
                                         : (count > 0 && w0 + q < nch ? __ldg(mrow + w0 + q) : 0u);
      if (few) {   // a lane per tile, a warp per word, four entries at a time
        uint32_t bits = 0u;
        int at = cursor;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (q == wu) bits = word[q];
          if (q < wu) at += __popc(word[q]);
        }
        const int k0 = (w0 + wu) * 32;
        while (bits) {
          int k[4], v[4];
#pragma unroll
          for (int z = 0; z < 4; ++z) {
            v[z] = k[z] = bits ? k0 + __ffs(bits) - 1 : -1;
            bits &= bits - 1u;
          }
          if (split) {
            double pa[4], pb[4];
#pragma unroll
            for (int z = 0; z < 4; ++z) {
              pa[z] = k[z] >= 0 ? in.nA[(int64_t)i * bk + k[z]] : 0.0;
              pb[z] = k[z] >= 0 ? in.nB[(int64_t)k[z] * bn + j] : 0.0;
            }
#pragma unroll
            for (int z = 0; z < 4; ++z)
              if (k[z] >= 0 && rel_bin(__dmul_rn(pa[z], pb[z]), inv) >= m) v[z] |= kSplitFlag;
          }
#pragma unroll
          for (int z = 0; z < 4; ++z)
            if (k[z] >= 0) Bf.k_idx[at++] = (uint16_t)v[z];
        }
      } else {
        unsigned todo = ne_mask;
        int turn = 0;
        while (todo) {
          const int src = __ffs(todo) - 1;
          todo &= todo - 1u;
          if ((turn++ & (kUnitWarps - 1)) != wu) continue;
          int at = __shfl_sync(0xffffffffu, cursor, src);
          const int si = __shfl_sync(0xffffffffu, i, src), sj = __shfl_sync(0xffffffffu, j, src);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t bits = __shfl_sync(0xffffffffu, word[q], src);
            if (bits == 0u) continue;   // uniform over the warp
            if ((bits >> lane) & 1u) {
              const int k = (w0 + q) * 32 + lane;
              uint16_t v = (uint16_t)k;
              if (split && rel_bin(__dmul_rn(in.nA[(int64_t)si * bk + k], in.nB[(int64_t)k * bn + sj]),
                                   inv) >= m)
                v |= kSplitFlag;
              Bf.k_idx[at + __popc(bits & lower)] = v;
            }
            at += __popc(bits);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) cursor += __popc(word[q]);
    }
  }
}

}  // namespace

int count_ctas_of(const Inst& in) { return units_of(in); }

void set_general(Inst& in, int64_t m, int64_t kd, int64_t n, int64_t lda, int64_t ldb,
                 int64_t ldc, float alpha, float beta, int leaf) {
  in.m = m;
  in.kd = kd;
  in.n = n;
  in.lda = lda;
  in.ldb = ldb;
  in.ldc = ldc;
  in.bm = (int)num_blocks(m, leaf);
  in.bk = (int)num_blocks(kd, leaf);
  in.bn = (int)num_blocks(n, leaf);
  in.alpha = alpha;
  in.beta = beta;
}

void set_square(Inst& in, int64_t n, int leaf) { set_general(in, n, n, n, n, n, n, 1.0f, 0.0f, leaf); }

size_t plan_layout(Inst* insts, int count, PlanBuffers* b, char* base, bool norm_parts) {
  int64_t tiles = 0, ablks = 0, bblks = 0, kslots = 0, mwords = 0, groups = 0;
  int64_t need_a = 0, need_b = 0;
  int prep = 0, cnt = 0;
  size_t staged = 0;
  for (int i = 0; i < count; ++i) {
    Inst& in = insts[i];
    const int64_t bm = in.bm, bk = in.bk, bn = in.bn;
    const int rows = in.bm < kBandRows ? in.bm : kBandRows;
    const size_t st = (size_t)(rows + unit_cols(in.bm)) * staged_len(in.bk) * sizeof(Screen);
    staged = staged > st ? staged : st;
    in.tile0 = tiles;
    in.ablk0 = ablks;
    in.bblk0 = bblks;
    in.kidx0 = kslots;
    in.mask0 = mwords;
    in.grp0 = groups;
    in.needa0 = need_a;
    in.needb0 = need_b;
    in.prep0 = prep;
    in.count0 = cnt;
    tiles += bm * bn;
    ablks += bm * bk;
    bblks += bk * bn;
    kslots += bm * bk * bn;
    mwords += bm * bn * ((bk + 31) / 32);
    need_a += bm * ((bk + 31) / 32);
    need_b += bn * ((bk + 31) / 32);
    groups += bm * ((bn + kGroupTiles - 1) / kGroupTiles);
    prep += prep_parts(in);
    cnt += count_ctas_of(in);
  }
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = (off + 255) / 256 * 256;
    char* p = base ? base + off : nullptr;
    off += bytes;
    return p;
  };
  PlanBuffers t{};
  t.tiles = tiles;
  t.groups = groups;
  t.ablks = ablks;
  t.bblks = bblks;
  t.kslots = kslots;
  t.prep_ctas = prep;
  t.count_ctas = cnt;
  t.staged_bytes = staged;
  t.need_words_a = need_a;
  t.need_words_b = need_b;
  int shift = 0;
  if (cnt > kScanUnits) {
    shift = 6;
    while (((int64_t)1 << (2 * shift)) < cnt) ++shift;
  }
  t.group_shift = shift;
  const int nparts = prep > cnt ? prep : cnt;
  const int ugroups = shift ? (cnt + (1 << shift) - 1) >> shift : 0;
  t.pd = reinterpret_cast<PlanDevice*>(take((size_t)count * sizeof(PlanDevice)));
  t.bdev = reinterpret_cast<BatchDevice*>(take(sizeof(BatchDevice)));
  t.need_bits = reinterpret_cast<uint32_t*>(
      take((size_t)(t.need_words_a + t.need_words_b) * sizeof(uint32_t)));
  t.sA = reinterpret_cast<Screen*>(take((size_t)ablks * sizeof(Screen)));
  t.sBT = reinterpret_cast<Screen*>(take((size_t)bblks * sizeof(Screen)));
  t.part_a = reinterpret_cast<double*>(take((size_t)nparts * sizeof(double)));
  t.part_b = reinterpret_cast<double*>(take((size_t)nparts * sizeof(double)));
  t.part = reinterpret_cast<int*>(take((size_t)cnt * kPartInts * sizeof(int)));
  t.part_bound = reinterpret_cast<ExtSum*>(take((size_t)cnt * 2 * sizeof(ExtSum)));
  t.group = reinterpret_cast<int*>(take((size_t)ugroups * kPartInts * sizeof(int)));
  t.cert = reinterpret_cast<CertState*>(take(sizeof(CertState)));
  t.cnt = reinterpret_cast<int*>(take((size_t)tiles * sizeof(int)));
  t.tile_beg = reinterpret_cast<int*>(take((size_t)tiles * sizeof(int)));
  t.order = reinterpret_cast<int*>(take((size_t)tiles * sizeof(int)));
  t.k_idx = reinterpret_cast<uint16_t*>(take((size_t)kslots * sizeof(uint16_t)));
  t.tile_inst = reinterpret_cast<int*>(take((size_t)tiles * sizeof(int)));
  t.surv_mask = reinterpret_cast<uint32_t*>(take((size_t)mwords * sizeof(uint32_t)));
  t.need_list = reinterpret_cast<uint32_t*>(take((size_t)(ablks + bblks) * sizeof(uint32_t)));
  t.norm_part = norm_parts ? take((size_t)tiles * kMaxEpiWarps * sizeof(NormPart)) : nullptr;
  for (int i = 0; i < count; ++i) insts[i].pd = t.pd ? t.pd + i : nullptr;
  if (b) *b = t;
  return (off + 255) / 256 * 256;
}

InstRef make_ref(const Inst* host_insts, const Inst* dev_table, int count) {
  InstRef r{};
  r.count = count;
  r.table = dev_table;
  if (!dev_table) r.one = host_insts[0];
  for (int i = 0; i < count; ++i) {
    r.any_split |= host_insts[i].split != 0;
    r.any_band |= host_insts[i].band != 0;
    r.any_norm_out |= host_insts[i].nC != nullptr;
    r.any_scaled |= host_insts[i].alpha != 1.0f || host_insts[i].beta != 0.0f;
  }
  return r;
}

namespace {

// Some instance needs ||A|| ||B|| while its products are counted, or the units
// are totalled in groups: the prep kernel runs first.
bool needs_prep(const InstRef& ref, const PlanBuffers& b) {
  return ref.any_split || b.group_shift != 0;
}

cudaError_t launch_prep(const InstRef& ref, const PlanBuffers& b, int screens, cudaStream_t s) {
  return launch_pdl(prep_kernel, dim3(b.prep_ctas), dim3(kPrepThreads), 0, s, ref, b, screens);
}

cudaError_t launch_count(const InstRef& ref, const PlanBuffers& b, int prepped, int stats,
                         cudaStream_t s) {
  auto* kern = ref.any_band ? (ref.any_split ? count_kernel<true, true> : count_kernel<false, true>)
                            : (ref.any_split ? count_kernel<true, false> : count_kernel<false, false>);
  {   // opt in to the largest size once per device and variant
    static bool opted[64][4] = {};
    const int v = (ref.any_band ? 2 : 0) + (ref.any_split ? 1 : 0);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !opted[dev][v]) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(16 * staged_len(kMaxBd) * sizeof(Screen)));
      if (e != cudaSuccess) return e;
      if (dev >= 0 && dev < 64) opted[dev][v] = true;
    }
  }
  return launch_pdl(kern, dim3(b.count_ctas), dim3(kCountThreads), b.staged_bytes, s, ref, b, prepped,
                    stats);
}

}  // namespace

cudaError_t run_plan_count_half(const InstRef& ref, const PlanBuffers& b, cudaStream_t s) {
  const int prepped = needs_prep(ref, b) ? 1 : 0;
  cudaError_t e = prepped ? launch_prep(ref, b, 0, s) : cudaSuccess;
  return e == cudaSuccess ? launch_count(ref, b, prepped, 0, s) : e;
}

cudaError_t run_plan_queue_half(const InstRef& ref, const PlanBuffers& b, cudaStream_t s) {
  // two CTAs per SM (each reads the totals of all units), four when the totals
  // are grouped; at most 32 units each
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int want = std::max(1, sms * (b.group_shift ? 4 : 2));
  const int per = std::min(32, std::max(1, (b.count_ctas + want - 1) / want));
  const int grid = (b.count_ctas + per - 1) / per + (ref.any_split ? 0 : ref.count);
  return launch_pdl(fill_kernel, dim3(grid), dim3(kFillThreads), 0, s, ref, b, per,
                    needs_prep(ref, b) ? 1 : 0);
}

cudaError_t run_plan(const InstRef& ref, const PlanBuffers& b, cudaStream_t s) {
  cudaError_t e = run_plan_count_half(ref, b, s);
  if (e == cudaSuccess) e = run_plan_queue_half(ref, b, s);
  return e;
}

cudaError_t run_plan_count(const InstRef& ref, const PlanBuffers& b, cudaStream_t s) {
  // the statistics come from the last count CTA: its ticket needs the prep kernel
  cudaError_t e = launch_prep(ref, b, 0, s);
  return e == cudaSuccess ? launch_count(ref, b, 1, 1, s) : e;
}

cudaError_t run_certify(const InstRef& ref, const PlanBuffers& b, double ref_rel, cudaStream_t s) {
  static bool opted[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!opted[dev]) {
    e = cudaFuncSetAttribute(cert_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(16 * staged_len(kMaxBd) * sizeof(Screen)));
    if (e != cudaSuccess) return e;
    opted[dev] = true;
  }
  e = launch_prep(ref, b, 0, s);
  if (e == cudaSuccess) e = launch_pdl(cert_init_kernel, dim3(1), dim3(32), 0, s, ref, b, ref_rel);
  for (int pass = 0; pass < kCertBits / 4 && e == cudaSuccess; ++pass)
    e = launch_pdl(cert_pass_kernel, dim3(b.count_ctas), dim3(kCountThreads), b.staged_bytes, s, ref, b);
  return e;
}

cudaError_t run_tile_norms(const InstRef& ref, const PlanBuffers& b, cudaStream_t s) {
  return launch_pdl(tile_norms_kernel, dim3(1), dim3(1024), 0, s, ref, b);
}

cudaError_t run_histogram(const InstRef& ref, const PlanBuffers& b, cudaStream_t s) {
  cudaError_t e = launch_prep(ref, b, 1, s);
  if (e != cudaSuccess) return e;
  hist_kernel<<<b.count_ctas, kHistWarps * 32, 0, s>>>(ref, b);
  return cudaPeekAtLastError();
}

}  // namespace spamm
