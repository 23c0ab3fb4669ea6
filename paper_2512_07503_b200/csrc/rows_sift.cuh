// Row kernels that sift a row by a sampled threshold: the sampling head (guidance merge, temperature, top-K,
// softmax, the row's own draw) in one pass over the logits.
//
// A row is cut into segments of consecutive ids, one per warp.  Its phases:
//
//   sample    256 pieces spread evenly over the row (64 bytes each, 16 where the row is short) give a threshold
//             tau0 that a little more than K of the row's entries reach.
//   sift      every warp takes its segment through shared memory in units of 4 KB per logits array: all entries
//             are merged and compared with tau0, which leaves one bit per entry in a register of the lane; the
//             set bits become a dense list of ids by one scan; the listed entries are merged once more from
//             shared memory and kept with their ids.  Comparing costs ~5 instructions per entry whatever comes of it,
//             keeping is paid for the few per cent that are kept, at full lanes.
//   finish    exact K-th largest among the candidates by a histogram and a ranking inside one bin (ties to the
//             lower id), softmax, output, inverse-CDF draw.  Every warp works on its own candidates, which are in
//             ascending id order already; what the warps exchange is a histogram and a few sums.
//
// A row whose largest entries crowd into one block of ids (image tokens in a vocabulary with text) overruns one segment's list
// while the others are empty.  What finds no room is still counted, and the histogram of all candidates gives a threshold that
// hardly more than K entries reach: with that the row is sifted once more, every unit taking a run of one list for the
// whole row.  us a step with the top-K in an eighth of the ids, all of it redone by
// row_generic() before: 1,024 rows of 65,536 bf16, K=2,000: 598 -> 259; 1,000 of 65,536 fp16, K=100: 560 -> 124; 231 of 50,264, K=500:
// 136 -> 71; 1,024 of 65,536, K=8,192: 907 -> 436 (ordinary rows of these shapes: 75.7 -> 76.8, 55.3 -> 55.9, 27.9 -> 27.9, 169 -> 170).  One list for
// all rows from the start costs ordinary rows a tenth (a barrier per row, an atomic per unit, loops over short runs).
//
// A row whose candidates cannot contain its top-K for sure (fewer than K), do not fit the list even so, or have no finite
// maximum is redone by row_generic() from global memory: results are exact for any input.
//
// Two kernels share the phases:
//
//   rows_stream_kernel   many rows: one persistent CTA per SM of up to three teams of eight warps and one sampler warp for
//                        each team.  A team sifts and finishes a row; the teams take the CTA's rows in turn, so that one
//                        sifts while others finish.  The rows' units come through one ring of shared-memory slots per
//                        segment, in row order.  The samplers find the thresholds of rows to come: a team's own sample
//                        phase (its first row's) is 9-14 K cycles of barriers and short searches that would hold up
//                        eight warps (with every row sampled by its team: 94 us where this takes 82).
//   rows_cluster_kernel  few rows: one cluster of up to eight CTAs of sixteen warps per row, the whole row in shared
//                        memory at once.  Every CTA sifts into lists of its own and sends them to the first one (distributed
//                        shared memory), which finishes the row.
//
// What bounds it: at V=65,536 and K=2,000 a row is about 40 K warp instructions at 56 % of the issue slots; a row of the
// memory stream alone would be 12.3 K cycles, and takes 14 K.  us a step (in brackets the kernels that took these shapes before):
// 1,024 rows of 65,536 bf16, K=2,000: 73.5 (88.4 with a kernel of one id range per filter thread); of 16,384: 44.9 (68.2);
// 1,024 ragged rows of 16,384 fp32, K=1,000: 41.7 (59.4); 1,024 rows of 32,768 bf16 without guidance: 44.5 (64.7); 231 rows of
// 50,264, K=500: 27.4 (100.8, four radix passes and a compaction over the row in the L2); 1,024 rows of 65,536, K=8,192:
// 139.0 (524); 16 rows of 4,096 fp32, K=64: 11.2 (16.7, tiles dealt to filter warps).
//
// Every wait on an mbarrier is bounded; a wait that gives up marks the row (and the CTA's unfinished rows) with
// kRowStatusTimeout, and the CTA waits (bounded) for its copies in flight before it exits.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "rows_pipeline.cuh"

namespace sjd {

constexpr int kSiftPieces = 256;          // sample pieces per row
constexpr int kSiftGroups = 1024;         // sample groups per row (at most)
constexpr int kSiftBins = 1024;           // bins of the candidates' histogram
constexpr int kBinsLow = 768;             // candidates' bins 1 .. kBinsLow cover the lowest eighth of their values
constexpr float kBinsCross = (8.0f * (kBinsLow + 1) - (kSiftBins - 2)) / 7.0f;  // where the upper bins' line starts
constexpr int kMemberCap = 512;           // members of the threshold bin ranked by brute force
constexpr int kUnitBytes = 4096;          // bytes of one logits array per unit: 128 for each lane
constexpr int kTeamWarps = 8;             // stream kernel: warps per team
constexpr int kTeamThreads = kTeamWarps * 32;
constexpr int kMaxTeams = 3;
constexpr int kMaxSlots = 4;              // ring slots per warp
constexpr int kAskAhead = 256 << 10;      // bytes of logits (whole rows) a CTA asks into the L2 before it may begin
constexpr int kStreamRows = 64;           // live rows a CTA takes in one launch (the host splits larger problems)
constexpr int kClusterWarps = 16;
constexpr int kMaxCluster = 8;

struct SiftCfg {
  int piece_stride;  // elements between the starts of two sample pieces (a multiple of 8)
  int piece_vecs;    // 16-byte vectors per piece: 4, 2 or 1
  int groups;        // groups per vector, each represented by its largest element: 1, 2 or 4
  int rank;          // rank of tau0 among the groups, from the top
  int packed;        // 1: entries may be screened in packed 16-bit arithmetic (see SiftScreen)
  int seg_len;       // ids per segment, a multiple of 8
  int units;         // units per segment
  int seg_cap;       // candidates a segment's list holds (a multiple of 8)
  int pool;          // entries of all lists of a row (a multiple of 8, below 65,536)
  int scratch;       // cluster kernel, rows that crowd: ids that a warp can list apart from these
  int teams, slots;  // stream kernel: teams per CTA, ring slots per warp
  int once;          // stream kernel: the logits of the call exceed the L2
  int row_begin, row_end;  // stream kernel: this launch covers rows [row_begin, row_end)
};

// Member of the threshold bin: value and id as one number, the larger the earlier it ranks (value descending, id ascending; the two
// zeros are equal values).
__device__ __forceinline__ uint64_t sift_member(float y, int id) {
  return (uint64_t)float_key(__fadd_rn(y, 0.0f)) << 32 | (uint32_t)~id;
}
__device__ __forceinline__ float member_value(uint64_t member) { return key_float((uint32_t)(member >> 32)); }
__device__ __forceinline__ int member_id(uint64_t member) { return (int)~(uint32_t)member; }

// Fine bins and one coarse bin per 32 of them: whoever counts in a fine bin counts in its coarse bin as well, which costs
// next to nothing and makes the search for a rank two scans of 32 words, done while everybody waits.
struct alignas(16) SiftHist {
  union {
    uint32_t fine[kSiftBins];        // zero whenever it is not in use
    uint64_t member[kMemberCap];     // the threshold bin's members, after the histogram's last search
  };
  uint32_t coarse[kSiftBins / 32];
  __device__ __forceinline__ void count(uint32_t bin) {
    atomicAdd(&fine[bin], 1u);
    atomicAdd(&coarse[bin >> 5], 1u);
  }
};

// what the warps that work on one row share
struct alignas(16) SiftShared {
  SiftHist hist;
  uint64_t wtot[kClusterWarps];
  uint32_t wcnt[kClusterWarps];
  uint64_t wz[kClusterWarps];
  uint32_t max_key;   // largest candidate
  uint32_t over;      // a list ran over, or a wait gave up
  uint32_t taken;     // a row that crowds: entries of its list that are given out
  int members;
  uint32_t rank_bin, rank_above, rank_count;  // results of a rank search
  float thr_y;
  int thr_id;
  float ptok;
  uint32_t rnd_lo, rnd_hi;
};

// barrier of the warps that work on one row
template <int NT>
__device__ __forceinline__ void row_sync(int bar) {
  asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NT) : "memory");
}

// ---------------------------------------------------------------------------------------------------
// logits: sixteen bytes of each array at a time
// ---------------------------------------------------------------------------------------------------
template <int DTYPE>
struct SiftTraits {
  static constexpr int kElem = DTYPE == 0 ? 4 : 2;           // bytes
  static constexpr int kVec = 16 / kElem;                    // elements per 16-byte vector
  static constexpr int kUnit = kUnitBytes / kElem;           // elements per unit
  static constexpr int kPiece = 64 / kElem;                  // elements of 64 bytes; a lane has two such pieces of a unit
};

// Merged logits of one vector, packed in pairs: d = c - u; g = fma(s, d, u); y = g * inv_T, one rounding per
// operation (a 16-bit c goes into the subtraction as it is).
template <int DTYPE, bool HAS_U, bool HAS_T>
__device__ __forceinline__ void merge_vec(const uint4& cv, const uint4& uv, uint64_t s2, uint64_t t2,
                                          uint64_t (&y)[SiftTraits<DTYPE>::kVec / 2]) {
  const uint32_t cw[4] = {cv.x, cv.y, cv.z, cv.w}, uw[4] = {uv.x, uv.y, uv.z, uv.w};
#pragma unroll
  for (int k = 0; k < SiftTraits<DTYPE>::kVec / 2; ++k) {
    uint64_t g;
    if (DTYPE == 0) {
      g = (uint64_t)cw[2 * k & 3] | ((uint64_t)cw[(2 * k + 1) & 3] << 32);
      if (HAS_U) {
        const uint64_t u = (uint64_t)uw[2 * k & 3] | ((uint64_t)uw[(2 * k + 1) & 3] << 32);
        g = fma2(s2, sub2(g, u), u);
      }
    } else if (HAS_U) {
      uint64_t u;
      if (DTYPE == 1) {
        u = pack2(bf16_lo(uw[k]), bf16_hi(uw[k]));
      } else {
        const float2 f = f16_pair(uw[k]);
        u = pack2(f.x, f.y);
      }
      g = fma2(s2, sub2_narrow<DTYPE>(cw[k], u), u);
    } else if (DTYPE == 1) {
      g = pack2(bf16_lo(cw[k]), bf16_hi(cw[k]));
    } else {
      const float2 f = f16_pair(cw[k]);
      g = pack2(f.x, f.y);
    }
    if (HAS_T) g = mul2(g, t2);
    y[k] = g;
  }
}

__device__ __forceinline__ uint32_t lds32(uint32_t at) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at));
  return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t at) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(at));
  return v;
}

// y of one staged entry; a NaN ranks with -inf.
template <int DTYPE, bool HAS_U, bool HAS_T>
__device__ __forceinline__ float merge_entry(uint32_t c_at, uint32_t u_at, float s, float inv_T) {
  float c, u = 0.0f;
  if (DTYPE == 0) {
    c = __uint_as_float(lds32(c_at));
    if (HAS_U) u = __uint_as_float(lds32(u_at));
  } else if (DTYPE == 1) {
    c = __uint_as_float(lds16(c_at) << 16);
    if (HAS_U) u = __uint_as_float(lds16(u_at) << 16);
  } else {
    c = f16_pair(lds16(c_at)).x;
    if (HAS_U) u = f16_pair(lds16(u_at)).x;
  }
  float g = HAS_U ? __fmaf_rn(s, __fsub_rn(c, u), u) : c;
  if (HAS_T) g = __fmul_rn(g, inv_T);
  return fmaxf(g, __int_as_float(0xff800000));
}

__device__ __forceinline__ uint32_t scan_incl(uint32_t v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += n;
  }
  return v;
}

// ---------------------------------------------------------------------------------------------------
// rank search: the bin b with (entries above b) < target <= (entries in b and above), by one
// warp, which also leaves the histogram zero.  A bin is 0 when there are fewer than `target` entries in bins 1 and
// above.
// ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ void rank_search(SiftShared* sm, SiftHist* h, uint32_t t) {
  const int lane = threadIdx.x & 31;
  const uint32_t sum = h->coarse[31 - lane];  // lane 0 takes the topmost
  const uint32_t upto = scan_incl(sum, lane);
  const uint32_t votes = __ballot_sync(0xffffffffu, upto - sum < t && t <= upto);
  uint32_t bin = 0, before = 0, count = 0;
  if (votes != 0u) {
    const int l1 = __ffs((int)votes) - 1;
    const uint32_t above1 = __shfl_sync(0xffffffffu, upto - sum, l1);
    const uint32_t f = h->fine[32 * (31 - l1) + 31 - lane];
    const uint32_t a2 = above1 + scan_incl(f, lane) - f;
    const int l2 = __ffs((int)__ballot_sync(0xffffffffu, a2 < t && t <= a2 + f)) - 1;
    bin = (uint32_t)(32 * (31 - l1) + 31 - l2);
    before = __shfl_sync(0xffffffffu, a2, l2);
    count = __shfl_sync(0xffffffffu, f, l2);
  }
  if (lane == 0) {
    sm->rank_bin = bin;
    sm->rank_above = before;
    sm->rank_count = count;
  }
  __syncwarp();
#pragma unroll
  for (int x = 0; x < kSiftBins / 128; ++x) reinterpret_cast<uint4*>(h->fine)[lane + 32 * x] = make_uint4(0u, 0u, 0u, 0u);
  h->coarse[lane] = 0u;
}

// ---------------------------------------------------------------------------------------------------
// sample phase
// ---------------------------------------------------------------------------------------------------
// A row's sample is cut into groups of G neighbouring elements, each represented by its largest.  With exchangeable entries
// a group has its maximum above t with probability 1 - (1 - p(t))^G, which is how the host translates the wanted share p
// of entries into a rank among maxima: a fraction of the work for nearly the same sharpness while few entries lie above the
// threshold (where many do, it takes smaller groups of fewer vectors).  tau0 only steers how many candidates there are;
// the result is exact whatever it is, so the maxima may be rounded to bf16.
//
// The candidates' bins are 1 .. kSiftBins - 1; bin 0 takes what is no candidate.  bin(y) is the smaller of two rising lines
// over y - tau0, the first of which spends kBinsLow bins on the lowest eighth of [tau0, largest sample value], where
// the candidates crowd: the threshold's bin then holds a handful of members.  Any rising function would do: a
// higher bin never holds a smaller value.
struct SiftBinning {
  float tau0, s1, s2;
  __device__ __forceinline__ float at(float y) const {
    const float d = __fsub_rn(y, tau0);
    return fminf(__fmaf_rn(d, s1, 1.0f), __fmaf_rn(d, s2, kBinsCross));
  }
};
__device__ __forceinline__ SiftBinning sift_bins(float tau0, float top) {
  const float range = __fsub_rn(top, tau0);
  const float per = range > 0.0f ? __fdiv_rn(1.0f, range) : 0.0f;
  // (finite slopes however narrow the range: tau0 itself has to fall into bin 1)
  const float most = 3.0e38f;
  return SiftBinning{tau0, fminf(__fmul_rn(8.0f * kBinsLow, per), most), fminf(__fmul_rn((kSiftBins - 2) - kBinsCross, per), most)};
}

// A sample's load, issued where it stands.  It is to stay in the L2 until its row comes through the ring, half a dozen rows
// later: without the hint an eighth of the logits came from memory twice.
__device__ __forceinline__ uint4 ldg_now(const void* p) {
  uint4 v;
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
  return v;
}

// packed 16-bit arithmetic: DTYPE 1 bf16, 2 fp16
template <int DTYPE>
__device__ __forceinline__ uint32_t fma_pair(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  if (DTYPE == 2) asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  else asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
template <int DTYPE>
__device__ __forceinline__ uint32_t sub_pair(uint32_t a, uint32_t b) {
  uint32_t r;
  if (DTYPE == 2) asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  else asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
template <int DTYPE>
__device__ __forceinline__ uint32_t largest2(uint32_t m, uint32_t w) {  // max(m, |w|) of both halves; a NaN is passed over
  uint32_t r;
  if (DTYPE == 2) asm("{\n\t.reg .b32 t;\n\tabs.f16x2 t, %2;\n\tmax.f16x2 %0, %1, t;\n\t}" : "=r"(r) : "r"(m), "r"(w));
  else asm("{\n\t.reg .b32 t;\n\tabs.bf16x2 t, %2;\n\tmax.bf16x2 %0, %1, t;\n\t}" : "=r"(r) : "r"(m), "r"(w));
  return r;
}
template <int DTYPE>
__device__ __forceinline__ float largest_of(uint32_t m) {
  if (DTYPE == 2) {
    const float2 f = f16_pair(m);
    return fmaxf(f.x, f.y);
  }
  return fmaxf(bf16_lo(m), bf16_hi(m));
}
// a float in the 16-bit type, rounded to nearest, twice in a word
template <int DTYPE>
__device__ __forceinline__ uint32_t pair_of(float x) {
  uint32_t r;
  if (DTYPE == 2) asm("cvt.rn.f16x2.f32 %0, %1, %1;" : "=r"(r) : "f"(x));
  else asm("cvt.rn.bf16x2.f32 %0, %1, %1;" : "=r"(r) : "f"(x));
  return r;
}

// the largest number of the type below the one that a word holds twice (zero: the negative number next to it)
__device__ __forceinline__ uint32_t pair_below(uint32_t t) {
  return (t & 0x7fffu) == 0u ? 0x80018001u : (t & 0x8000u) ? t + 0x00010001u : t - 0x00010001u;
}

// 16-bit logits: entries are screened in packed 16-bit arithmetic, two to an instruction, and only what passes is merged
// exactly.  With guidance g = s (c - u) + u reaches g0 (the value before the temperature) only if (t - (1 - s) u) - s c < 0
// for a t that lies below g0 by more than the bracket can be off: the product-sum's own rounding cannot change its sign, the
// bracket is off by its rounding, 2^-8 (bf16) or 2^-11 (fp16) of |1 - s| |u| + |t| at most, and t by as much of |t|.  The exact
// path rounds as well: c - u and the sum, in 32 bits, put g off by 2^-24 of |g| and of |u| each, which matters where s is 1 and
// |u| outweighs the threshold.  So s and 1 - s have to be numbers of the type (the host sees to that), and |u| has to stay
// below a limit that t was chosen for: a unit that holds a larger one is compared exactly, and so is a row for which the 32-bit
// roundings outweigh the 16-bit ones, or whose products with 1/T may be subnormal.  About a tenth more entries pass than reach
// tau0; they end as candidates below tau0, in bin 0.  Without guidance c is compared with the largest number of the type below
// g0.  A NaN (the merge of two tokens masked with -inf) has no sign and does not pass.
// Two instructions per entry instead of four; worth it while few entries pass anyway (the host's rule): 1,000 rows of 65,536
// fp16 entries, K=100: 59.7 -> 57.3 us.
struct SiftScreen {
  uint32_t s2, b2, t2;  // -s, s - 1 and t, pairs
  float u_limit;        // negative: this row is compared exactly
};
template <int DTYPE, bool HAS_U, bool HAS_T>
__device__ __forceinline__ SiftScreen sift_screen(const RowArgs& a, const SiftCfg& cfg, float tau0, float u_max) {
  SiftScreen r{0u, 0u, 0u, -1.0f};
  if (DTYPE == 0 || !cfg.packed) return r;
  if (HAS_T && !(fabsf(tau0) >= 1.0e-30f)) return r;
  constexpr float kRound = DTYPE == 2 ? 0x1p-11f : 0x1p-8f;
  float g0 = HAS_T ? __fdiv_rn(tau0, a.inv_T) : tau0;
  g0 = __fmaf_rd(fabsf(g0), -0x1p-20f, g0);
  if (HAS_U) {
    const float b = 1.0f - a.s, limit = 1.25f * u_max, reach = fabsf(b) * limit + 2.0f * fabsf(g0);
    const float narrow = 0x1p-22f * limit;  // the 32-bit roundings, with room
    if (!(reach < 3.0e4f) || !(narrow <= kRound * reach)) return r;
    r.s2 = pair_of<DTYPE>(-a.s);
    r.b2 = pair_of<DTYPE>(-b);
    r.t2 = pair_below(pair_of<DTYPE>(__fmaf_rn(-1.03f * kRound, reach, g0 - narrow)));
    r.u_limit = limit;
  } else {
    if (!(fabsf(g0) < 3.0e4f)) return r;
    const uint32_t t = pair_of<DTYPE>(g0);
    const float back = DTYPE == 2 ? f16_pair(t).x : bf16_lo(t);
    r.t2 = back >= g0 ? pair_below(t) : t;
    r.u_limit = 0.0f;
  }
  return r;
}

// what a row's threshold is found from
struct alignas(16) SiftSample {
  uint32_t m[kSiftGroups / 2];  // the groups' maxima as bf16 pairs, in no particular order
  uint32_t top_key;             // largest sample value (0 between rows)
  uint32_t u_bits;              // largest |uncond| of the sample, 16-bit types (a float's bits; 0 between rows)
};

// The groups' maxima of a row, by NT threads, four vectors per thread at a time (all there are when 256 threads share the
// work).  The caller sees to the barrier behind it.
template <int DTYPE, bool HAS_U, bool HAS_T, int NT>
__device__ __forceinline__ void sift_sample(const RowArgs& a, const SiftCfg& cfg, SiftSample& out, const char* c_row, const char* u_row,
                                            int tid) {
  constexpr int EV = SiftTraits<DTYPE>::kVec, ES = SiftTraits<DTYPE>::kElem;
  constexpr int NV = NT >= 256 ? kSiftGroups / NT : 4;
  const float neg_inf = __int_as_float(0xff800000);
  const uint64_t s2 = pack2(a.s, a.s), t2 = pack2(a.inv_T, a.inv_T);
  const int vecs = kSiftPieces * cfg.piece_vecs;
  const int shift = cfg.piece_vecs >> 1;  // log2 of 1, 2, 4
  uint16_t* const m = reinterpret_cast<uint16_t*>(out.m);
  auto put = [&](int x, float v) { m[x] = __bfloat16_as_ushort(__float2bfloat16_rn(v)); };
  float top = neg_inf;
  uint32_t u_max = 0u;  // largest |uncond|, a pair
#pragma unroll 1
  for (int v0 = tid; v0 - tid < vecs; v0 += NT * NV) {
    uint4 c[NV], u[HAS_U ? NV : 1];
    uint32_t have = 0;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int v = v0 + j * NT, piece = v >> shift, k = v & (cfg.piece_vecs - 1);
      const int e = piece * cfg.piece_stride + k * EV;
      const bool in = v < vecs && k * EV < cfg.piece_stride && e < a.V;
      have |= in ? 1u << j : 0u;
      const size_t at = in ? (size_t)e * ES : 0;
      c[j] = ldg_now(c_row + at);
      if (HAS_U) u[HAS_U ? j : 0] = ldg_now(u_row + at);
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      uint64_t y2[EV / 2];
      merge_vec<DTYPE, HAS_U, HAS_T>(c[j], u[HAS_U ? j : 0], s2, t2, y2);
      if (HAS_U && DTYPE != 0) {
        const uint4 w = u[HAS_U ? j : 0];
        u_max = largest2<DTYPE>(largest2<DTYPE>(largest2<DTYPE>(largest2<DTYPE>(u_max, w.x), w.y), w.z), w.w);
      }
      float y[EV];
#pragma unroll
      for (int k = 0; k < EV / 2; ++k) unpack2(y2[k], y[2 * k], y[2 * k + 1]);
      const int v = v0 + j * NT;
      const bool in = (have >> j) & 1u;  // (a NaN is passed over by every maximum)
      if (cfg.groups == 1) {
        float all = neg_inf;
#pragma unroll
        for (int k = 0; k < EV / 2; ++k) all = max3(all, y[2 * k], y[2 * k + 1]);
        all = in ? all : neg_inf;
        top = fmaxf(top, all);
        put(min(v, kSiftGroups - 1), all);
      } else {
        float q[4];  // maxima of the vector's quarters
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          q[k] = EV == 8 ? fmaxf(y[(2 * k) % EV], y[(2 * k + 1) % EV]) : y[k];
          q[k] = in ? fmaxf(q[k], neg_inf) : neg_inf;
          top = fmaxf(top, q[k]);
        }
        if (v < vecs) {
          if (cfg.groups == 2) {
            put(2 * v, fmaxf(q[0], q[1]));
            put(2 * v + 1, fmaxf(q[2], q[3]));
          } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) put(4 * v + k, q[k]);
          }
        }
      }
    }
  }
  // groups there are no vectors for
  for (int x = vecs * cfg.groups + tid; x < kSiftGroups; x += NT) m[x] = 0xff80u;
  const uint32_t warp_top = __reduce_max_sync(0xffffffffu, float_key(__fadd_rn(top, 0.0f)));
  if ((tid & 31) == 0) atomicMax(&out.top_key, warp_top);
  if (HAS_U && DTYPE != 0) {
    const uint32_t warp_u = __reduce_max_sync(0xffffffffu, __float_as_uint(largest_of<DTYPE>(u_max)));
    if ((tid & 31) == 0) atomicMax(&out.u_bits, warp_u);
  }
}

// The search for the threshold goes over the bf16 values as 16-bit keys that are ordered like them: the largest key whose
// value at least `rank` of the maxima reach.  How many do is counted by a warp that holds them all, a lane 16 pairs:
// sixteen packed comparisons and additions.
struct SiftMaxima {
  static constexpr int NM = kSiftGroups / 64;
  uint32_t m2[NM];
  __device__ __forceinline__ void load(const SiftSample& in, int lane) {
#pragma unroll
    for (int x = 0; x < NM / 4; ++x) {
      const uint4 v = reinterpret_cast<const uint4*>(in.m)[lane + 32 * x];
      m2[4 * x] = v.x; m2[4 * x + 1] = v.y; m2[4 * x + 2] = v.z; m2[4 * x + 3] = v.w;
    }
  }
  __device__ __forceinline__ uint32_t reaching(uint32_t key) const {
    const uint32_t v = (key & 0x8000u) ? key & 0x7fffu : ~key & 0xffffu;  // bf16 pattern of the key
    const uint32_t t = v | (v << 16);
    uint32_t acc[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int x = 0; x < NM; ++x) {
      uint32_t g;
      asm("set.ge.bf16x2.bf16x2 %0, %1, %2;" : "=r"(g) : "r"(m2[x]), "r"(t));
      asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(acc[x & 3]) : "r"(g));
    }
    asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(acc[0]) : "r"(acc[1]));
    asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(acc[2]) : "r"(acc[3]));
    asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(acc[0]) : "r"(acc[2]));
    return __reduce_add_sync(0xffffffffu, (uint32_t)(bf16_lo(acc[0]) + bf16_hi(acc[0])));
  }
};
// {tau0, largest sample value, largest |uncond| of the sample} for the key found
struct SiftTau {
  float tau0, top, u_max;
};
// Below this value (a bf16 key: -8,192) a token counts as masked.  Where so much of a row is masked that the wanted rank lies among
// the masked groups, the rest of the row is taken whole, so to speak: the threshold goes as far below the least unmasked
// maximum as the largest lies above it, and the row comes again with the threshold that its histogram gives.
constexpr uint32_t kMaskedKey = 0x39ffu;
__device__ __forceinline__ SiftTau sift_tau(uint32_t key, bool whole, const SiftSample& in) {
  const uint32_t top_key = in.top_key;
  const float top = key_float(top_key), lowest = -3.402823466e38f;  // lowest: every finite value is a candidate
  // the maxima were rounded to nearest: the middle between this bf16 value and the one below is what they all reach
  const float at = key_float(key << 16), below = key_float((key - 1u) << 16);
  float tau0 = __fmaf_rd(__fsub_rn(at, below), -0.51f, at);
  if (whole) tau0 = __fsub_rn(tau0, __fsub_rn(top, tau0));
  if (key == 0u || !(tau0 >= lowest) || !(top <= 3.402823466e38f)) tau0 = lowest;
  return SiftTau{tau0, top, __uint_as_float(in.u_bits)};
}
// The lowest of the 256 keys that end at the largest maximum's: two octaves, where an ordinary row's threshold lies (0: fewer are unmasked).
// When `rank` of the maxima reach it, eight bits are left to be found instead of sixteen: a step of the search is some 290 cycles of one warp.
// 1,024 ragged rows of 16,384 fp32: 43.4 -> 42.2 us a step; 1,024 of 32,768 without guidance: 45.2 -> 44.3; 16 of 4,096: 11.6 -> 11.2.
// (Two bits at a time, three counts side by side: slower, 73.5 -> 74.5 at 1,024 rows of 65,536; counts of the keys' bytes in shared memory, by
// the team: 4 to 9 K cycles instead of 4.6 K beside the other teams' loads.)
__device__ __forceinline__ uint32_t window_key(const SiftSample& in) {
  const uint32_t last = (in.top_key >> 16) + 1u;  // (the maxima are rounded to nearest)
  return last >= kMaskedKey + 255u && last <= 0xffffu ? last - 255u : 0u;
}
// by one warp, bit by bit
__device__ __forceinline__ SiftTau sift_threshold(const SiftSample& in, uint32_t rank, int lane) {
  SiftMaxima m;
  m.load(in, lane);
  uint32_t key = window_key(in);
  if (key != 0u && m.reaching(key) >= rank) {
#pragma unroll 1
    for (uint32_t bit = 0x80u; bit != 0u; bit >>= 1)
      if (m.reaching(key + bit) >= rank) key += bit;
    return sift_tau(key, false, in);
  }
  for (bool whole = false;; whole = true) {
    key = 0;
#pragma unroll 1
    for (uint32_t bit = 0x8000u; bit != 0u; bit >>= 1)
      if (m.reaching(key | bit) >= rank) key |= bit;
    if (key >= kMaskedKey || whole) return sift_tau(key, whole, in);
    rank = m.reaching(kMaskedKey);
    if (rank == 0u) return sift_tau(key, false, in);
  }
}

// ---------------------------------------------------------------------------------------------------
// sift phase
// ---------------------------------------------------------------------------------------------------
// Hit bits of 64 bytes per array of a lane: bit k is set when element k reaches tau0, that is when it lies above `below`, the
// number next to tau0.  The sign of below - y is exact (a difference rounds to zero only when it is zero), is not set for a
// NaN (tokens masked with -inf in both arrays merge to one) and is moved in with one funnel shift per element.  Lanes start at different 16-byte pieces (`rot`), so that the eight lanes
// served together touch different banks; the word is rotated back afterwards.
template <int DTYPE, bool HAS_U, bool HAS_T>
__device__ __forceinline__ uint32_t piece_hits(uint32_t c_at, uint32_t u_at, int rot, uint64_t s2, uint64_t t2, uint64_t below2) {
  constexpr int EV = SiftTraits<DTYPE>::kVec;
  uint32_t hits = 0;
#pragma unroll
  for (int j = 3; j >= 0; --j) {
    const uint32_t off = (uint32_t)(((j + rot) & 3) << 4);
    const uint4 c = lds128(c_at + off);
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    if (HAS_U) u = lds128(u_at + off);
    uint64_t y[EV / 2];
    merge_vec<DTYPE, HAS_U, HAS_T>(c, u, s2, t2, y);
#pragma unroll
    for (int k = EV / 2 - 1; k >= 0; --k) {
      const uint64_t t = sub2(below2, y[k]);
      hits = __funnelshift_l((uint32_t)(t >> 32), hits, 1);
      hits = __funnelshift_l((uint32_t)t, hits, 1);
    }
  }
  if (DTYPE != 0) return __funnelshift_l(hits, hits, 8 * rot);
  const uint32_t x = (hits & 0xffffu) * 0x10001u;
  return (x >> (16 - 4 * rot)) & 0xffffu;
}

// The same by packed screening.  The signs of four entries are gathered as bytes of -1 by one permute; a dot product with
// the powers of two makes them four bits.  u_max: largest |uncond| met.
template <int DTYPE, bool HAS_U>
__device__ __forceinline__ uint32_t piece_screened(uint32_t c_at, uint32_t u_at, int rot, const SiftScreen& sc, uint32_t& u_max) {
  int32_t acc = 0;  // minus the hit bits
#pragma unroll
  for (int j = 3; j >= 0; --j) {
    const uint32_t off = (uint32_t)(((j + rot) & 3) << 4);
    const uint4 cv = lds128(c_at + off);
    const uint32_t c[4] = {cv.x, cv.y, cv.z, cv.w};
    uint32_t w[4];
    if (HAS_U) {
      const uint4 uv = lds128(u_at + off);
      const uint32_t u[4] = {uv.x, uv.y, uv.z, uv.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        w[k] = fma_pair<DTYPE>(sc.s2, c[k], fma_pair<DTYPE>(sc.b2, u[k], sc.t2));
        u_max = largest2<DTYPE>(u_max, u[k]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = sub_pair<DTYPE>(sc.t2, c[k]);
    }
    acc <<= 8;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      uint32_t signs;
      asm("prmt.b32 %0, %1, %2, 0xfdb9;" : "=r"(signs) : "r"(w[2 * k]), "r"(w[2 * k + 1]));
      asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(acc) : "r"(signs), "r"(k == 0 ? 0x08040201u : 0x80402010u));
    }
  }
  const uint32_t hits = 0u - (uint32_t)acc;
  return __funnelshift_l(hits, hits, 8 * rot);
}

// ids of the set bits of x (bit 0: id `first`), from the highest down, to the halfwords below `put`
__device__ __forceinline__ uint32_t put_ids(uint32_t x, uint32_t first, uint32_t put) {
  while (x != 0u) {
    uint32_t b;
    asm("bfind.u32 %0, %1;" : "=r"(b) : "r"(x));
    x ^= 1u << b;
    put -= 2u;
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(put), "h"((uint16_t)(first + b)) : "memory");
  }
  return put;
}

// where a warp's candidates go
struct SiftTarget {
  uint32_t y_at, id_at;    // shared-memory addresses of the segment's lists (a cluster's row that crowds: of the row's, in the first CTA)
  uint32_t hist_at;        // of the candidates' histogram (a SiftHist)
  uint32_t scratch_at;     // where ids are listed first: the same as id_at unless that is in another CTA
  uint32_t cap;            // candidates the lists hold
  // a row that crowds: the lists are the row's
  uint32_t taken_at;       // of the number of entries given out
  uint32_t scratch;        // ids the local list holds (0: it is the row's)
};
constexpr uint32_t kNoRoom = 0xffffffffu;

template <bool REMOTE>
__device__ __forceinline__ void put_f32(uint32_t at, float v) {
  if (REMOTE) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory");
  else asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory");
}
template <bool REMOTE>
__device__ __forceinline__ void put_u16(uint32_t at, uint32_t v) {
  if (REMOTE) asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(at), "h"((uint16_t)v) : "memory");
  else asm volatile("st.shared.u16 [%0], %1;" ::"r"(at), "h"((uint16_t)v) : "memory");
}
// whose lists and histogram a sift fills: the CTA's own; the cluster's first CTA's; its own, to the histogram of which other CTAs add
enum { kToOwn = 0, kToFirst = 1, kToShared = 2 };
template <int TO>
__device__ __forceinline__ void count_at(uint32_t at) {
  if (TO == kToFirst) asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], 1;" ::"r"(at) : "memory");
  else if (TO == kToShared) asm volatile("red.relaxed.cluster.shared::cta.add.u32 [%0], 1;" ::"r"(at) : "memory");
  else asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], 1;" ::"r"(at) : "memory");
}

// `n` entries of the row's list, n being lane 31's
template <bool REMOTE>
__device__ __forceinline__ uint32_t take_entries(uint32_t at, uint32_t n, int lane) {
  uint32_t first = 0;
  if (lane == 31) {
    if (REMOTE) asm volatile("atom.relaxed.cluster.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(first) : "r"(at), "r"(n) : "memory");
    else asm volatile("atom.relaxed.cta.shared::cta.add.u32 %0, [%1], %2;" : "=r"(first) : "r"(at), "r"(n) : "memory");
  }
  return __shfl_sync(0xffffffffu, first, 31);
}

// One unit: `valid` elements of it belong to the segment; element 0 has id `rel` in the list's numbering.  n: candidates so far (cap + 1:
// the list has run over).
// CROWDS: the unit takes a run of the row's list, which n becomes: its first entry, and from bit 16 its length (kNoRoom: there was
// none).  Candidates that find no room are counted all the same, so that the row's histogram is complete.
template <int DTYPE, bool HAS_U, bool HAS_T, int TO, bool CROWDS>
__device__ __forceinline__ void sift_unit(const RowArgs& a, uint32_t c_unit, uint32_t u_unit, int valid, uint32_t rel, uint64_t s2,
                                          uint64_t t2, const SiftBinning& bins, const SiftScreen& screen,
                                          const SiftTarget& to, int lane, uint32_t& n, float& vmax) {
  constexpr int ES = SiftTraits<DTYPE>::kElem, EP = SiftTraits<DTYPE>::kPiece, EU = SiftTraits<DTYPE>::kUnit;
  constexpr bool REMOTE = TO == kToFirst;
  uint32_t x0 = 0, x1 = 0;  // hits of the lane's first and second piece
  const bool whole = valid > EU / 2;
  const uint32_t run = whole ? 2 * EP : EP;  // consecutive elements of a lane
  // where this lane's pieces lie and where it starts in them, so that the lanes served together touch different banks
  const uint32_t swap = whole ? ((uint32_t)lane & 4u) << 4 : 0u;
  const uint32_t at0 = whole ? (128u * (uint32_t)lane) ^ swap : 64u * (uint32_t)lane, at1 = at0 ^ 64u;
  const int rot = whole ? lane & 3 : (lane >> 1) & 3;
  // (a unit that is not full is compared exactly: what lies behind its end must not decide how it is compared)
  bool exact = DTYPE == 0 || screen.u_limit < 0.0f || (uint32_t)valid < 32u * run;
  if (DTYPE != 0 && !exact) {
    uint32_t u_max = 0u;
    x0 = piece_screened<DTYPE, HAS_U>(c_unit + at0, u_unit + at0, rot, screen, u_max);
    if (whole) x1 = piece_screened<DTYPE, HAS_U>(c_unit + at1, u_unit + at1, rot, screen, u_max);
    if (HAS_U) exact = __any_sync(0xffffffffu, largest_of<DTYPE>(u_max) > screen.u_limit);
  }
  if (exact) {
    const float below = bins.tau0 == 0.0f ? __int_as_float(0x80000001) : key_float(float_key(bins.tau0) - 1u);
    const uint64_t below2 = pack2(below, below);
    x0 = piece_hits<DTYPE, HAS_U, HAS_T>(c_unit + at0, u_unit + at0, rot, s2, t2, below2);
    if (whole) x1 = piece_hits<DTYPE, HAS_U, HAS_T>(c_unit + at1, u_unit + at1, rot, s2, t2, below2);
  }
  if (swap) {
    const uint32_t x = x0;
    x0 = x1;
    x1 = x;
  }
  if (DTYPE == 0) {
    x0 |= x1 << 16;
    x1 = 0;
  }
  if (valid < EU) {
    const int left = valid - lane * (int)run;
    x0 = left >= 32 ? x0 : left > 0 ? x0 & ((1u << left) - 1u) : 0u;
    x1 = left >= 64 ? x1 : left > 32 ? x1 & ((1u << (left - 32)) - 1u) : 0u;
  }
  const uint32_t inc = scan_incl((uint32_t)(__popc(x0) + __popc(x1)), lane);
  const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
  const uint32_t first = rel + (uint32_t)lane * run;  // id of the lane's first bit
  const uint32_t c_rel = c_unit - rel * (uint32_t)ES, u_rel = u_unit - rel * (uint32_t)ES;
  const bool own_ids = CROWDS && REMOTE && to.scratch != 0u;  // ids are listed apart from the row's list
  uint32_t at = n;  // first entry of the unit's candidates
  if (CROWDS) at = take_entries<REMOTE>(to.taken_at, inc, lane);
  if (__builtin_expect(at + total > to.cap || (own_ids && total > to.scratch), 0)) {
    n = CROWDS ? kNoRoom : to.cap + 1u;
    while ((x0 | x1) != 0u) {  // one of each piece at a time
      float y[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t x = h == 0 ? x0 : x1, id = x != 0u ? first + 32u * h + (uint32_t)__ffs((int)x) - 1u : first;
        y[h] = merge_entry<DTYPE, HAS_U, HAS_T>(c_rel + id * (uint32_t)ES, u_rel + id * (uint32_t)ES, a.s, a.inv_T);
        if (x == 0u) y[h] = __int_as_float(0xff800000);
      }
      x0 &= x0 - 1u;
      x1 &= x1 - 1u;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t bin = min(__float2uint_rz(bins.at(y[h])), (uint32_t)kSiftBins - 1u);
        count_at<TO>(to.hist_at + 4u * bin);
        count_at<TO>(to.hist_at + 4u * (kSiftBins + (bin >> 5)));
        vmax = fmaxf(vmax, y[h]);
      }
    }
    __syncwarp();
    return;
  }
  // ids, from the lane's highest one down
  const uint32_t ids_at = own_ids ? to.scratch_at : to.scratch_at + 2u * at;
  {
    uint32_t put = ids_at + 2u * inc;
    if (DTYPE != 0) put = put_ids(x1, first + 32u, put);
    put_ids(x0, first, put);
  }
  __syncwarp();
  // candidates: merged, binned and kept, two groups of 32 at a time (their loads do not wait for one another)
  auto keep = [&](auto groups, uint32_t i0) {
    constexpr int G = decltype(groups)::value;
    uint32_t id[G];
    float y[G];
#pragma unroll
    for (int j = 0; j < G; ++j) id[j] = lds16(ids_at + 2u * min(i0 + 32u * j + (uint32_t)lane, total - 1u));
#pragma unroll
    for (int j = 0; j < G; ++j)
      y[j] = merge_entry<DTYPE, HAS_U, HAS_T>(c_rel + id[j] * (uint32_t)ES, u_rel + id[j] * (uint32_t)ES, a.s, a.inv_T);
#pragma unroll
    for (int j = 0; j < G; ++j) {
      const uint32_t i = i0 + 32u * j + (uint32_t)lane, k = at + i;
      const bool in = i < total;
      const uint32_t bin = in ? min(__float2uint_rz(bins.at(y[j])), (uint32_t)kSiftBins - 1u) : 0u;
      count_at<TO>(to.hist_at + 4u * bin);
      count_at<TO>(to.hist_at + 4u * (kSiftBins + (bin >> 5)));
      vmax = fmaxf(vmax, y[j]);
      if (in) {
        put_f32<REMOTE>(to.y_at + 4u * k, y[j]);
        if (REMOTE) put_u16<true>(to.id_at + 2u * k, id[j]);
      }
    }
  };
  uint32_t i0 = 0;
  for (; i0 + 32u < total; i0 += 64u) keep(std::integral_constant<int, 2>(), i0);
  if (i0 < total) keep(std::integral_constant<int, 1>(), i0);
  n = CROWDS ? at | (total << 16) : at + total;
}

// exp(y - m) with the rounding of the difference compensated (exp_diff without its case for y = -inf)
__device__ __forceinline__ float exp_diff_finite(float y, float m) {
  const float t = __fsub_rn(y, m);
  const float bb = __fsub_rn(t, y);                                                // ~ -m
  const float err = __fadd_rn(__fsub_rn(y, __fsub_rn(t, bb)), __fsub_rn(-m, bb));  // (y - m) - t, exact
  const float e = expf(t);
  return __fmaf_rn(e, err, e);
}

// An exponential (at most 1) in units of 2^-45.  Sums of these do not depend on the order, so a row's probabilities are the
// same to the last bit whichever warps and lanes its candidates fell to, that is in a call of any number of rows; what is cut
// off is less than 2^-45 of a sum that is at least 1, for each entry.  Against float sums, which differed between the two kernels:
// 1,024 rows of 65,536, K=2,000: 75.4 -> 75.7 us; K=8,192: 166.2 -> 168.5; of 16,384, K=2,000: 46.6 -> 46.9.  (The integers read
// out of the last places of float sums instead of converted: 0.2 to 0.4 us more.)
__device__ __forceinline__ uint64_t fixed_exp(float e) { return __float2ull_rz(__fmul_rn(e, 0x1p45f)); }

// ---------------------------------------------------------------------------------------------------
// finish phase, by the NW warps that work on the row
// ---------------------------------------------------------------------------------------------------
// where the runs of a row that crowds lie in it: run r holds candidates of the ids from (r / units) * seg_len + (r % units) * unit on
struct SiftRuns {
  uint32_t* run;  // first entry in the row's list, and from bit 16 their number
  int n, units, seg_len, unit;
  __device__ __forceinline__ int id0(int r) const { return r / units * seg_len + r % units * unit; }
};
// The first run of warp `part`'s share when NW warps share the candidates about evenly: the number of runs that begin before
// that part of all candidates.
template <int NW>
__device__ __forceinline__ int first_run(const SiftRuns& runs, int part, int lane) {
  uint32_t total = 0;
  for (int r = lane; r < runs.n; r += 32) total += runs.run[r] >> 16;
  total = __reduce_add_sync(0xffffffffu, total);
  const uint32_t bound = (uint32_t)((uint64_t)total * (uint32_t)part / NW);
  uint32_t before = 0;
  int n = 0;
  for (int r0 = 0; r0 < runs.n; r0 += 32) {
    const uint32_t len = r0 + lane < runs.n ? runs.run[r0 + lane] >> 16 : 0u;
    const uint32_t upto = scan_incl(len, lane);
    n += __popc(__ballot_sync(0xffffffffu, r0 + lane < runs.n && before + upto - len < bound));
    before += __shfl_sync(0xffffffffu, upto, 31);
  }
  return part >= NW ? runs.n : n;
}

// Warp w holds the candidates of `per_warp` consecutive segments in lists of seg_cap entries each, seg_n of them in use, ids
// relative to the warp's first one.  CROWDS: the row has one list, `runs` of it in ascending order, of which each warp takes a share;
// their ids are relative to the run's first one.
// Starts with a barrier.  The histogram is zero again and the counters are reset whatever comes of it.
enum { kRowDone = 0, kRowOver = 1, kRowElse = 2 };  // finished; a list had run over; not to be finished here for another reason
template <int NW, bool CROWDS>
__device__ __forceinline__ int finish_row(const RowArgs& a, const SiftCfg& cfg, SiftShared& sm, float* list_y, uint16_t* list_id,
                                          const uint32_t* seg_n, int per_warp, const SiftRuns& runs, const SiftBinning& bins, int row, int pos,
                                          int iter, int draft, int status, int tid, int bar) {
  constexpr int NT = NW * 32;
  const int lane = tid & 31, warp = tid >> 5;
  const uint32_t kcap = (uint32_t)a.kcap;
  const uint32_t below = (1u << lane) - 1u;
  row_sync<NT>(bar);
  if (warp == 0) rank_search(&sm, &sm.hist, kcap);
  if (tid == NT - 1) {
    // the row's own random number, needed at the end
    const Philox4 r = philox4x32_10((uint32_t)pos, (uint32_t)(a.seq_base + row / a.W), (uint32_t)iter, (uint32_t)a.purpose, a.seed_lo,
                                    a.seed_hi);
    sm.rnd_lo = r.x0;
    sm.rnd_hi = r.x1;
    sm.ptok = 0.0f;
  }
  const float vmax = key_float(sm.max_key);
  const bool over = sm.over != 0u;
  row_sync<NT>(bar);
  const uint32_t tbin = sm.rank_bin, need = kcap - sm.rank_above, nbin = sm.rank_count;
  if (tid == 0) {
    sm.max_key = 0u;
    sm.over = 0u;
    if (CROWDS) sm.taken = 0u;
    sm.thr_y = vmax;  // (for raise_threshold)
  }
  // fewer than kcap candidates, a threshold bin too crowded for the ranking, or no finite maximum
  if (over || tbin == 0u || nbin > (uint32_t)kMemberCap || !(vmax <= 3.402823466e38f)) {
    row_sync<NT>(bar);
    return over ? kRowOver : kRowElse;
  }
  // the warp's segments, or its share of the runs: from g0 on, up to g1
  const int g0 = CROWDS ? first_run<NW>(runs, warp, lane) : 0, g1 = CROWDS ? first_run<NW>(runs, warp + 1, lane) : per_warp;
  if (CROWDS) row_sync<NT>(bar);  // (their lengths are changed below)
  const size_t first_seg = CROWDS ? 0 : (size_t)warp * per_warp;
  float* const my_y = list_y + first_seg * cfg.seg_cap;
  uint16_t* const my_id = list_id + first_seg * cfg.seg_cap;
  const int warp_id0 = warp * per_warp * cfg.seg_len;
  // ---- the threshold bin's members
  {
    // (the last bin also holds what lies above its end)
    const bool last = tbin == (uint32_t)kSiftBins - 1u;
    const float lo = (float)tbin, hi = (float)(tbin + 1u);
    for (int g = g0; g < g1; ++g) {
      const uint32_t run = CROWDS ? runs.run[g] : 0u, n = CROWDS ? run >> 16 : seg_n[first_seg + g];
      const uint32_t at_g = CROWDS ? run & 0xffffu : (uint32_t)(g * cfg.seg_cap);
      const int id0 = CROWDS ? runs.id0(g) : warp_id0;
      const float* const y_g = my_y + at_g;
#pragma unroll 4
      for (uint32_t i = (uint32_t)lane; i < n; i += 32u) {
        const float y = y_g[i], x = bins.at(y);
        if (x >= lo && (x < hi || last)) {
          const int at = atomicAdd(&sm.members, 1);  // (as many as the histogram counted: the check keeps the store in bounds)
          if (at < kMemberCap) sm.hist.member[at] = sift_member(y, id0 + (int32_t)my_id[at_g + i]);
        }
      }
    }
  }
  row_sync<NT>(bar);
  // the `need`-th of them by (y descending, id ascending) is the last survivor
  float thr_y;
  int thr_id;
  if (nbin <= 32u) {
    // every warp ranks them for itself, a lane per member
    const uint64_t me = sm.hist.member[min(lane, (int)nbin - 1)];
    uint32_t ahead = 0;
#pragma unroll 4
    for (int x = 0; x < (int)nbin; ++x) ahead += sm.hist.member[x] > me ? 1u : 0u;
    const int who = __ffs((int)__ballot_sync(0xffffffffu, lane < (int)nbin && ahead == need - 1u)) - 1;
    const uint64_t found = shfl_u64(me, who);
    thr_y = member_value(found);
    thr_id = member_id(found);
  } else {
    // A warp per member, a lane per rival; three members at a time, whose chains do not wait for one another.  (bf16 logits leave some
    // forty members with hardly a different value: 1,024 rows of 65,536, K=2,000: 74.4 -> 73.6 us; K=8,192: 142.0 -> 140.0.)  A comparison is
    // one of numbers: with values and ids compared apart it branched, and a row with 327 members, a few entries far above the rest, took 50 K
    // cycles to finish (32 K one member at a time).  64 rows of 524,288 bf16, K=100: 79.1 -> 61.0 us a step (one at a time: 70.2), without guidance
    // 73.3 -> 51.7 (61.8); 64 of 262,144 fp32: 65.7 -> 54.2 (62.1).
    constexpr int M = 3;
    for (uint32_t x = (uint32_t)warp; x < nbin; x += M * NW) {
      uint64_t me[M];
      uint32_t ahead[M];
#pragma unroll
      for (int k = 0; k < M; ++k) {
        me[k] = sm.hist.member[min(x + (uint32_t)(k * NW), nbin - 1u)];
        ahead[k] = 0;
      }
#pragma unroll 2
      for (uint32_t z = (uint32_t)lane; z < nbin; z += 32u) {
        const uint64_t o = sm.hist.member[z];
#pragma unroll
        for (int k = 0; k < M; ++k) ahead[k] += o > me[k] ? 1u : 0u;
      }
#pragma unroll
      for (int k = 0; k < M; ++k) {
        ahead[k] = __reduce_add_sync(0xffffffffu, ahead[k]);
        if (lane == 0 && ahead[k] == need - 1u) {  // (the last member may come twice: the same values)
          sm.thr_y = member_value(me[k]);
          sm.thr_id = member_id(me[k]);
        }
      }
    }
    row_sync<NT>(bar);
    thr_y = sm.thr_y;
    thr_id = sm.thr_id;
  }
  // ---- survivors: exponentials and ids to the front of the warp's lists (of each run), their number and sum.  Four groups of 32
  // at a time: their loads and exponentials do not wait for one another, nor for the stores, which go to places already read.
  int thr_rel = thr_id - warp_id0;
  uint32_t cnt = 0;
  uint64_t z = 0;
  for (int g = g0; g < g1; ++g) {
    const uint32_t run = CROWDS ? runs.run[g] : 0u, n = CROWDS ? run >> 16 : seg_n[first_seg + g];
    const uint32_t at_g = CROWDS ? run & 0xffffu : (uint32_t)(g * cfg.seg_cap);
    const float* const y_g = my_y + at_g;
    const uint16_t* const id_g = my_id + at_g;
    const uint32_t cnt0 = cnt;
    if (CROWDS) thr_rel = thr_id - runs.id0(g);
    constexpr int U = 4;
#pragma unroll 1
    for (uint32_t i0 = 0; i0 < n; i0 += 32u * U) {
      float e[U];
      int id[U];
      uint32_t votes[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const uint32_t i = i0 + 32u * j + (uint32_t)lane;
        e[j] = i < n ? y_g[i] : __int_as_float(0xff800000);
        id[j] = i < n ? (int)id_g[i] : 0x7fffffff;
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const bool alive = e[j] > thr_y || (e[j] == thr_y && id[j] <= thr_rel);
        votes[j] = __ballot_sync(0xffffffffu, alive);  // (every lane has read its entries: they may be overwritten)
        e[j] = exp_diff_finite(e[j], vmax);
      }
      __syncwarp();
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if ((votes[j] >> lane) & 1u) {
          const uint32_t at = (CROWDS ? at_g + cnt - cnt0 : cnt) + (uint32_t)__popc(votes[j] & below);
          my_y[at] = e[j];
          my_id[at] = (uint16_t)id[j];
          z += fixed_exp(e[j]);
        }
        cnt += (uint32_t)__popc(votes[j]);
      }
      __syncwarp();
    }
    if (CROWDS && lane == 0) runs.run[g] = at_g | ((cnt - cnt0) << 16);
  }
  z = warp_sum_u64(z);
  if (lane == 0) {
    sm.wcnt[warp] = cnt;
    sm.wz[warp] = z;
  }
  row_sync<NT>(bar);
  for (uint32_t x = (uint32_t)tid; x < nbin; x += NT) sm.hist.member[x] = 0ull;  // the histogram's words again
  if (tid == 0) sm.members = 0;
  const uint32_t cw = lane < NW ? sm.wcnt[lane] : 0u;
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? cw : 0u);
  if (__reduce_add_sync(0xffffffffu, cw) != kcap) {  // cannot happen; the result stays exact anyway
    row_sync<NT>(bar);  // (the histogram's words are zero before anybody counts in them again)
    return kRowElse;
  }
  const uint64_t Z = warp_sum_u64(lane < NW ? sm.wz[lane] : 0ull);
  const float inv_Z = __fdiv_rn(0x1p45f, __ull2float_rn(Z));  // p = e / Z within 2 ulp
  // ---- output and fixed-point weights
  const int p0 = CROWDS ? g0 : 0, p1 = CROWDS ? g1 : 1;  // where the warp's survivors lie: in the front of its runs, or of its lists
  int32_t* out_ids = a.out_ids + (size_t)row * kcap + before;
  float* out_vals = a.out_vals + (size_t)row * kcap + before;
  uint64_t wsum = 0;
  for (int g = p0; g < p1; ++g) {
    const uint32_t n = CROWDS ? runs.run[g] >> 16 : cnt, at_g = CROWDS ? runs.run[g] & 0xffffu : 0u;
    const int id0 = CROWDS ? runs.id0(g) : warp_id0;
    const float* const y_g = my_y + at_g;
    const uint16_t* const id_g = my_id + at_g;
#pragma unroll 4
    for (uint32_t i = (uint32_t)lane; i < n; i += 32u) {
      const float p = __fmul_rn(y_g[i], inv_Z);
      const int id = id0 + (int)id_g[i];
      out_ids[i] = id;
      out_vals[i] = p;
      wsum += fixed_weight(p);
      if (id == draft) sm.ptok = p;
    }
    if (CROWDS) out_ids += n, out_vals += n;
  }
  wsum = warp_sum_u64(wsum);
  if (lane == 0) sm.wtot[warp] = wsum;
  row_sync<NT>(bar);
  // ---- the row's own draw: fixed-point inverse CDF in ascending id order.  Every warp finds out whether the draw
  // falls to it; the one that holds it gives each lane a run of its survivors.
  const uint64_t x = lane < NW ? sm.wtot[lane] : 0ull;
  uint64_t xi = x;
#pragma unroll
  for (int d = 1; d < NW; d <<= 1) {
    const uint64_t o = shfl_up_u64(xi, d);
    if (lane >= d) xi += o;
  }
  const uint64_t total = shfl_u64(xi, NW - 1);
  const uint64_t t = __umul64hi((uint64_t)sm.rnd_lo | ((uint64_t)sm.rnd_hi << 32), total);
  uint64_t lo = shfl_u64(xi - x, warp);
  const uint64_t hi = shfl_u64(xi, warp);
  if (total == 0ull) {  // all weights rounded to zero: the first survivor
    if (lane == 0 && before == 0u && cnt > 0u) {
      uint32_t at = 0u;
      int id0 = warp_id0;
      if (CROWDS) {
        int g = g0;
        while ((runs.run[g] >> 16) == 0u) ++g;
        at = runs.run[g] & 0xffffu;
        id0 = runs.id0(g);
      }
      a.out_cnt[row] = (int)kcap;
      a.scratch[row] = RowScratch{sm.ptok, id0 + (int32_t)my_id[at], __fmul_rn(my_y[at], inv_Z), status};
    }
  } else if (t >= lo && t < hi) {
    for (int g = p0; g < p1; ++g) {
      const uint32_t n = CROWDS ? runs.run[g] >> 16 : cnt, at_g = CROWDS ? runs.run[g] & 0xffffu : 0u;
      const int id0 = CROWDS ? runs.id0(g) : warp_id0;
      const float* const y_g = my_y + at_g;
      const uint32_t run = (n + 31u) / 32u;
      const uint32_t beg = min((uint32_t)lane * run, n), end = min(beg + run, n);
      uint64_t own = 0;
      for (uint32_t i = beg; i < end; ++i) own += fixed_weight(__fmul_rn(y_g[i], inv_Z));
      uint64_t inc = own;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint64_t o = shfl_up_u64(inc, d);
        if (lane >= d) inc += o;
      }
      uint64_t sum = lo + inc - own;
      if (CROWDS) {
        lo += shfl_u64(inc, 31);
        if (t >= lo) continue;  // the whole warp: the draw lies behind this run
      }
      if (t >= sum && t < sum + own) {
        uint32_t i = beg;
        float p;
        for (;; ++i) {  // ends before `end`: the lane's weights sum to more than t - sum
          p = __fmul_rn(y_g[i], inv_Z);
          sum += fixed_weight(p);
          if (t < sum || i + 1u >= end) break;
        }
        a.out_cnt[row] = (int)kcap;
        a.scratch[row] = RowScratch{sm.ptok, id0 + (int32_t)my_id[at_g + i], p, status};
      }
      break;
    }
  }
  if (CROWDS) row_sync<NT>(bar);  // (the next row's runs may lie anywhere in the list)
  return kRowDone;
}

// By the thread that resets the counters, after a row has run over its lists: from the row's complete histogram a
// threshold that only the entries of the K-th largest one's bin and above reach.  False when even they do not fit, or when
// that would be the threshold there was.
__device__ __forceinline__ bool raise_threshold(const SiftShared& sm, const SiftBinning& bins, int room, SiftTau& tau) {
  const uint32_t bin = sm.rank_bin;
  const float vmax = sm.thr_y;
  if (bin < 2u || (int)(sm.rank_above + sm.rank_count) + 64 > room || !(vmax <= 3.402823466e38f)) return false;
  // the least difference to tau0 that falls into the bin, a little less (some entries of the bin below come along)
  const float d = fmaxf(__fdiv_rn((float)bin - 1.0f, bins.s1), __fdiv_rn((float)bin - kBinsCross, bins.s2));
  const float raised = __fadd_rd(bins.tau0, __fmul_rd(d, 1.0f - 0x1p-14f));
  if (!(raised > bins.tau0)) return false;
  tau.tau0 = raised;
  tau.top = vmax;
  return true;
}

// row_generic as a call of its own: it is rarely needed and its registers and code stay out of the hot loops.
template <int DTYPE, int NT, int BAR>
__device__ __noinline__ void sift_redo(const RowArgs& a, int row, int tid, GenericSmem& sm) {
  row_generic<DTYPE, NT, BAR>(a, row, tid, sm, kRowStatusRedone);
}

__device__ __forceinline__ void init_shared(SiftShared& sm, int tid, int nt) {
  for (int k = tid; k < (int)sizeof(SiftHist) / 16; k += nt) reinterpret_cast<uint4*>(&sm.hist)[k] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    sm.max_key = 0u;
    sm.over = 0u;
    sm.taken = 0u;
    sm.members = 0;
  }
}

// a row and what there is to know about it
struct SiftRow {
  int64_t off;    // of its first logit, in elements
  int32_t row;    // b * W + i
  int32_t pos;    // absolute position: pos_base[b] + i
  int32_t iter;   // iteration counter of its sequence
  int32_t draft;  // its draft token, -1 when every row is drafted
  bool live;      // inside its sequence's window
};
__device__ __forceinline__ SiftRow sift_row(const RowArgs& a, int row) {
  SiftRow r;
  const int b = row / a.W, i = row - b * a.W;
  r.row = row;
  r.off = (int64_t)b * a.stride_b + (int64_t)i * a.stride_w;
  r.live = a.win_len == nullptr || i < a.win_len[b];
  r.pos = (a.pos_base ? a.pos_base[b] : 0) + i;
  r.iter = a.iteration ? a.iteration[b] : a.iteration0;
  r.draft = a.drafts ? a.drafts[row] : -1;
  return r;
}

// ---------------------------------------------------------------------------------------------------
// many rows
// ---------------------------------------------------------------------------------------------------
struct alignas(16) StreamShared {
  SiftRow tab[kStreamRows];                    // the CTA's live rows
  // A unit of one of team t's rows has landed in the slot: [warp][team][slot].  A barrier of its own for every team: a
  // parity wait tells a phase from its neighbours only, so each barrier is waited on by one warp, phase after phase.
  uint64_t full[kTeamWarps * kMaxTeams * kMaxSlots];
  uint32_t used[kTeamWarps * kMaxTeams * kMaxSlots];  // copies issued for that barrier so far
  // for every team: a row's sample is complete, and {tau0, largest sample value} of rows to come, in two places used in turn
  uint64_t sample_full[kMaxTeams], tau_full[2 * kMaxTeams], tau_free[2 * kMaxTeams];
  SiftTau tau[2 * kMaxTeams];
  uint32_t seg_n[kMaxTeams * kTeamWarps];      // candidates per segment
  // Rows that were not finished: those to be redone from the front; from the back places in `tab` of those to be sifted again as
  // rows that crowd (their thresholds wait in their records).
  int32_t redo[kStreamRows];
  int n_live, n_redo, n_again, abort;
};
struct alignas(16) TeamShared {
  SiftShared row;
  SiftSample sample;  // the team's first row's is written by the team, the others' by its sampler
};
// shared memory: StreamShared | TeamShared x teams | list values | list ids | rings.  A team's lists of its segments lie one behind the
// other; a row that crowds has them as one, the last entries of whose values hold its runs.
__host__ __device__ inline size_t sift_stream_rings(const SiftCfg& cfg) {
  const size_t b = sizeof(StreamShared) + cfg.teams * (sizeof(TeamShared) + (size_t)cfg.pool * 6);
  return (b + 127) & ~(size_t)127;
}
__host__ __device__ inline size_t sift_stream_smem(const SiftCfg& cfg, bool has_u) {
  return sift_stream_rings(cfg) + (size_t)kTeamWarps * cfg.slots * kUnitBytes * (has_u ? 2 : 1);
}

// bulk_g2s with an L2 hint
__device__ __forceinline__ void bulk_g2s_hinted(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void ask_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// bounded wait that also ends when another warp of the CTA has given up.  The wait stays suspended in hardware for up to
// a few microseconds at a time: a waiting warp spends next to no issue slots.
__device__ __forceinline__ bool sift_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(4000u)
        : "memory");
    if (ok) return true;
    if (*abort_flag != 0 || clock64() - t0 > kSpinCycles) break;
  }
  return false;
}

// Copies go through the ring of a warp in order: its units of row 0, row 1, ...; team t takes rows t, t + teams, ...  Whoever has worked a
// unit through asks for the copy that goes into its slot next.  The units of a warp begin `step` ids apart, from seg0 on.
template <int DTYPE, bool HAS_U>
__device__ __forceinline__ void issue_unit(const RowArgs& a, StreamShared& st, unsigned char* ring, uint64_t policy, int warp, int teams,
                                           int units, int seg0, int seg_n, int step, int n_live, int k, int unit, int slot) {
  constexpr int ES = SiftTraits<DTYPE>::kElem, EU = SiftTraits<DTYPE>::kUnit;
  while (unit >= units) {
    ++k;
    unit -= units;
  }
  if (k >= n_live) return;
  const uint32_t bytes = (uint32_t)min(seg_n - unit * step, EU) * ES;
  const int64_t off = st.tab[k].off + seg0 + (int64_t)unit * step;
  unsigned char* const dst = ring + (size_t)slot * kUnitBytes * (HAS_U ? 2 : 1);
#ifdef SJD_TEST_DROP_COPY
  if (warp == SJD_TEST_DROP_COPY && k == 1 && unit == 0) return;  // test builds only, see rows_cluster_kernel
#endif
  const int x = (warp * kMaxTeams + k % teams) * kMaxSlots + slot;
  ++st.used[x];
  mbar_arrive_expect_tx(&st.full[x], bytes * (HAS_U ? 2u : 1u));
  bulk_g2s_hinted(dst, row_ptr(a.cond, DTYPE, off), bytes, &st.full[x], policy);
  if (HAS_U) bulk_g2s_hinted(dst + kUnitBytes, row_ptr(a.uncond, DTYPE, off), bytes, &st.full[x], policy);
}
// Logits that exceed the L2 leave it first (they make room for samples and outputs: 1,024 rows of 65,536 74.4 -> 73.4 us);
// smaller ones are left where their writer put them (of 16,384: 45.7, with the hint 46.6).
__device__ __forceinline__ uint64_t ring_policy(const SiftCfg& cfg) {
  uint64_t policy;
  if (cfg.once) asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  else asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy));
  return policy;
}
// A row that is to be sifted again, by one thread: its place in `tab`, and its threshold, which waits in its record.
__device__ __forceinline__ void sift_again(const RowArgs& a, StreamShared& st, int k, const SiftTau& tau) {
  a.scratch[st.tab[k].row] = RowScratch{tau.tau0, (int32_t)__float_as_uint(tau.u_max), tau.top, 0};
  st.redo[kStreamRows - 1 - atomicAdd(&st.n_again, 1)] = k;
}

// A row that crowds, by the team that calls: the part of rows_stream_kernel's loop from the sift on, with one list for the whole
// row and every eighth unit for a warp, so that a block of ids is shared by all.  Returns the ring barriers' parities (`phase` of
// the kernel).
template <int DTYPE, bool HAS_U, bool HAS_T>
__device__ __noinline__ uint32_t stream_crowded_row(const RowArgs& a, const SiftCfg& cfg, unsigned char* smem, int k, uint32_t phase, SiftTau tau) {
  constexpr int EU = SiftTraits<DTYPE>::kUnit, kStep = kTeamWarps * EU;
  constexpr uint32_t kSlot = kUnitBytes * (HAS_U ? 2u : 1u);
  StreamShared& st = *reinterpret_cast<StreamShared*>(smem);
  const int teams = cfg.teams, slots = cfg.slots;
  const int team = (int)threadIdx.x / kTeamThreads, tid = (int)threadIdx.x % kTeamThreads, lane = tid & 31, warp = tid >> 5, bar = 1 + team;
  TeamShared* const team_sm = reinterpret_cast<TeamShared*>(smem + sizeof(StreamShared));
  SiftShared& sm = team_sm[team].row;
  float* const lists = reinterpret_cast<float*>(team_sm + teams);
  float* const list_y = lists + team * cfg.pool;
  uint16_t* const list_id = reinterpret_cast<uint16_t*>(lists + teams * cfg.pool) + team * cfg.pool;
  const int row_units = (a.V + EU - 1) / EU, room = cfg.pool - row_units;
  const SiftRuns runs{reinterpret_cast<uint32_t*>(list_y + room), row_units, row_units, 0, EU};
  unsigned char* const ring = smem + sift_stream_rings(cfg) + (size_t)warp * slots * kSlot;
  const int seg0 = warp * EU, seg_n = max(a.V - seg0, 0), units = (seg_n + kStep - 1) / kStep;
  volatile int* const abort_flag = &st.abort;
  uint64_t* const full = st.full + (warp * kMaxTeams + team) * kMaxSlots;
  const uint64_t s2 = pack2(a.s, a.s), t2 = pack2(a.inv_T, a.inv_T), policy = ring_policy(cfg);
  const SiftBinning bins = sift_bins(tau.tau0, tau.top);
  const SiftScreen screen = sift_screen<DTYPE, HAS_U, HAS_T>(a, cfg, tau.tau0, tau.u_max);
  SiftTarget to;
  to.y_at = smem_u32(list_y);
  to.id_at = to.scratch_at = smem_u32(list_id);
  to.hist_at = smem_u32(&sm.hist);
  to.cap = (uint32_t)room;
  to.taken_at = smem_u32(&sm.taken);
  to.scratch = 0u;
  bool ok = true, over = false;
  float vmax = __int_as_float(0xff800000);
  int slot = (k * units) % slots;
  for (int unit = 0; unit < units; ++unit) {
    ok = sift_wait(&full[slot], (phase >> slot) & 1u, abort_flag);
    if (!ok) break;
    phase ^= 1u << slot;
    const uint32_t c_unit = smem_u32(ring) + (uint32_t)slot * kSlot;
    uint32_t run = 0u;
    sift_unit<DTYPE, HAS_U, HAS_T, kToOwn, true>(a, c_unit, c_unit + kUnitBytes, seg_n - unit * kStep, 0u, s2, t2, bins, screen, to, lane, run,
                                                vmax);
    over = over || run == kNoRoom;
    __syncwarp();
    if (lane == 0) {
      runs.run[unit * kTeamWarps + warp] = run;
      issue_unit<DTYPE, HAS_U>(a, st, ring, policy, warp, teams, units, seg0, seg_n, kStep, st.n_live, k, unit + slots, slot);
    }
    if (++slot == slots) slot = 0;
  }
  const uint32_t wmax = __reduce_max_sync(0xffffffffu, float_key(vmax));
  if (lane == 0) {
    atomicMax(&sm.max_key, wmax);
    if (over || !ok) sm.over = 1u;
    if (!ok) *abort_flag = 1;
  }
  const SiftRow& r = st.tab[k];
  const int result = finish_row<kTeamWarps, true>(a, cfg, sm, list_y, list_id, nullptr, 0, runs, bins, r.row, r.pos, r.iter, r.draft, kRowStatusRedone,
                                                  tid, bar);
  if (result != kRowDone && tid == 0) {
    if (*abort_flag != 0) {
      a.out_cnt[r.row] = 0;
      a.scratch[r.row] = RowScratch{0.0f, -1, 0.0f, kRowStatusTimeout};
    } else {
      st.redo[atomicAdd(&st.n_redo, 1)] = r.row;
    }
  }
  return phase;
}

// After the CTA's last row, by all teams: the rows that are to be sifted again, through the ring as before.
template <int DTYPE, bool HAS_U, bool HAS_T>
__device__ __noinline__ uint32_t stream_again(const RowArgs& a, const SiftCfg& cfg, unsigned char* smem, uint32_t phase) {
  constexpr int EU = SiftTraits<DTYPE>::kUnit, kStep = kTeamWarps * EU;
  StreamShared& st = *reinterpret_cast<StreamShared*>(smem);
  const int teams = cfg.teams, team = (int)threadIdx.x / kTeamThreads, lane = (int)threadIdx.x & 31;
  const int warp = ((int)threadIdx.x % kTeamThreads) >> 5, n = st.n_again;
  const bool lost = st.abort != 0;
  auto sync = [&] { asm volatile("bar.sync %0, %1;" ::"n"(1 + kMaxTeams), "r"(teams * kTeamThreads) : "memory"); };
  sync();  // (everybody has read what is changed now)
  if (threadIdx.x < 32) {
    SiftRow r[kStreamRows / 32];
#pragma unroll
    for (int j = 0; j < kStreamRows / 32; ++j)
      if (lane + 32 * j < n) r[j] = st.tab[st.redo[kStreamRows - 1 - lane - 32 * j]];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kStreamRows / 32; ++j) {
      if (lane + 32 * j >= n) continue;
      st.tab[lane + 32 * j] = r[j];
      if (lost) {
        a.out_cnt[r[j].row] = 0;
        a.scratch[r[j].row] = RowScratch{0.0f, -1, 0.0f, kRowStatusTimeout};
      }
    }
    if (lane == 0) st.n_live = n;
  }
  sync();
  if (lost) return phase;
  const int seg0 = warp * EU, seg_n = max(a.V - seg0, 0), units = (seg_n + kStep - 1) / kStep;
  unsigned char* const ring = smem + sift_stream_rings(cfg) + (size_t)warp * cfg.slots * kUnitBytes * (HAS_U ? 2 : 1);
  if (team == 0 && lane == 0 && units > 0) {
    const uint64_t policy = ring_policy(cfg);
    for (int x = 0; x < cfg.slots; ++x)
      issue_unit<DTYPE, HAS_U>(a, st, ring, policy, warp, teams, units, seg0, seg_n, kStep, n, 0, x, x);
  }
  __syncwarp();
  for (int k = team; k < n; k += teams) {
    const RowScratch what = a.scratch[st.tab[k].row];
    phase = stream_crowded_row<DTYPE, HAS_U, HAS_T>(a, cfg, smem, k, phase,
                                                    SiftTau{what.p_tok, what.samp_prob, __uint_as_float((uint32_t)what.samp_tok)});
  }
  sync();
  return phase;
}

template <int DTYPE, bool HAS_U, bool HAS_T>
__global__ void __launch_bounds__((kTeamThreads + 32) * kMaxTeams, 1)
rows_stream_kernel(const __grid_constant__ RowArgs a, const __grid_constant__ SiftCfg cfg) {
  constexpr int ES = SiftTraits<DTYPE>::kElem, EU = SiftTraits<DTYPE>::kUnit;
  constexpr uint32_t kSlot = kUnitBytes * (HAS_U ? 2u : 1u);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StreamShared& st = *reinterpret_cast<StreamShared*>(smem_raw);
  const int teams = cfg.teams, slots = cfg.slots;
  // warps: those of team 0, of team 1, ..., then a sampler for each team
  const bool sampler = (int)threadIdx.x >= teams * kTeamThreads;
  const int team = sampler ? ((int)threadIdx.x - teams * kTeamThreads) >> 5 : (int)threadIdx.x / kTeamThreads;
  const int tid = sampler ? (int)threadIdx.x & 31 : (int)threadIdx.x % kTeamThreads, lane = tid & 31, warp = tid >> 5, bar = 1 + team;
  TeamShared* const team_sm = reinterpret_cast<TeamShared*>(smem_raw + sizeof(StreamShared));
  SiftShared& sm = team_sm[team].row;
  SiftSample& sample = team_sm[team].sample;
  float* const lists = reinterpret_cast<float*>(team_sm + teams);
  float* const list_y = lists + team * cfg.pool;
  uint16_t* const list_id = reinterpret_cast<uint16_t*>(lists + teams * cfg.pool) + team * cfg.pool;
  unsigned char* const ring = smem_raw + sift_stream_rings(cfg) + (size_t)warp * slots * kSlot;
  if (!sampler) init_shared(sm, tid, kTeamThreads);
  if (threadIdx.x < kTeamWarps * kMaxTeams * kMaxSlots) {
    mbar_init(&st.full[threadIdx.x], 1);
    st.used[threadIdx.x] = 0;
  }
  if (threadIdx.x < 2 * kMaxTeams) {
    mbar_init(&st.tau_full[threadIdx.x], 1);
    mbar_init(&st.tau_free[threadIdx.x], kTeamWarps);
    if (threadIdx.x < kMaxTeams) mbar_init(&st.sample_full[threadIdx.x], kTeamWarps);
  }
  if (tid == 0) sample.top_key = sample.u_bits = 0u;
  if (threadIdx.x == 0) {
    st.n_redo = st.n_again = 0;
    st.abort = 0;
  }
  fence_barrier_init();
  // What a launch that overlaps the previous kernel may do before that kernel's end is shared-memory set-up, and asking the
  // CTA's first rows into the L2 (nothing is read; the L2 is where all writes meet): the memory would lie idle meanwhile.
  if (threadIdx.x < 32) {
    const int64_t bytes = (int64_t)a.V * ES, row = (int64_t)cfg.row_begin + blockIdx.x + (int64_t)lane * gridDim.x;
    if (lane * bytes * (HAS_U ? 2 : 1) < kAskAhead && row < cfg.row_end) {
      const int b = (int)(row / a.W), i = (int)(row - (int64_t)b * a.W);
      const int64_t off = (int64_t)b * a.stride_b + (int64_t)i * a.stride_w;
      ask_l2(row_ptr(a.cond, DTYPE, off), (uint32_t)bytes);
      if (HAS_U) ask_l2(row_ptr(a.uncond, DTYPE, off), (uint32_t)bytes);
    }
    __syncwarp();
  }
  grid_dependency_wait();
  // ---- the CTA's rows: row_begin + blockIdx.x, + gridDim.x, ... (at most kStreamRows).  Rows beyond their sequence's window
  // length get their empty result; the others go into a table, so that no warp reads global memory for them later.
  if (threadIdx.x < 32) {
    int n = 0;
    for (int k0 = 0; k0 < kStreamRows; k0 += 32) {
      const int64_t row = (int64_t)cfg.row_begin + blockIdx.x + (int64_t)(k0 + lane) * gridDim.x;
      SiftRow r;
      r.live = false;
      if (row < cfg.row_end) {
        r = sift_row(a, (int)row);
        if (!r.live) {
          a.out_cnt[row] = 0;
          a.scratch[row] = RowScratch{0.0f, -1, 0.0f, 0};
        }
      }
      const uint32_t votes = __ballot_sync(0xffffffffu, r.live);
      if (r.live) st.tab[n + __popc(votes & ((1u << lane) - 1u))] = r;
      n += __popc(votes);
    }
    if (lane == 0) st.n_live = n;
  }
  __syncthreads();
  const int n_live = st.n_live;
  volatile int* const abort_flag = &st.abort;
  if (sampler) {
    // ======================================= samplers =======================================
    // the thresholds of the team's rows, one or two rows ahead
    for (int k = team, n = 0; k < n_live; k += teams, ++n) {
      if (n == 0) {
        if (!sift_wait(&st.sample_full[team], 0u, abort_flag)) break;
      } else {
        const int64_t off = st.tab[k].off;
        sift_sample<DTYPE, HAS_U, HAS_T, 32>(a, cfg, sample, static_cast<const char*>(row_ptr(a.cond, DTYPE, off)),
                                             HAS_U ? static_cast<const char*>(row_ptr(a.uncond, DTYPE, off)) : nullptr, lane);
      }
      __syncwarp();
      const SiftTau tau = sift_threshold(sample, (uint32_t)cfg.rank, lane);
      const int x = 2 * team + (n & 1);
      if (n >= 2 && !sift_wait(&st.tau_free[x], (uint32_t)((n >> 1) - 1) & 1u, abort_flag)) break;
      __syncwarp();
      if (lane == 0) {
        sample.top_key = 0u;
        sample.u_bits = 0u;
        st.tau[x] = tau;
        mbar_arrive(&st.tau_full[x]);
      }
      __syncwarp();
    }
    __syncthreads();
    return;
  }
  const int seg0 = warp * cfg.seg_len;
  const int seg_n = min(max(a.V - seg0, 0), cfg.seg_len);  // ids of this warp's segment
  const int units = (seg_n + EU - 1) / EU;
  const uint64_t policy = ring_policy(cfg);
  auto issue = [&](int k, int unit, int slot) {
    issue_unit<DTYPE, HAS_U>(a, st, ring, policy, warp, teams, units, seg0, seg_n, EU, n_live, k, unit, slot);
  };
  // The first copies are sent off before anything else (behind the first team's sample: 1,024 rows of 16,384 bf16 46.2 us a step, now 45.3;
  // ragged fp32 ones 42.0 and 41.5; of 65,536 73.2 and 73.7; 444 of 32,768, K=2,500, 41.8 and 40.8), but behind its sample where the CTA has
  // a single row of several units a warp: no other row hides a sample that waits for copies (148 rows of 65,536, K=10: 19.4 before the
  // sample, now 18.6; of fp32 25.0 and 23.7; of 262,144, K=700, 39.7 and 38.8; a unit a warp, 200 rows of 4,096: 12.7 before it, 12.9 behind it).
  if (team == (teams > 1 ? 1 : 0) && lane == 0 && units > 0) {
    if (n_live == 1 && team > 0 && units > 1) mbar_wait(&st.sample_full[0], 0u);
    for (int x = 0; x < slots; ++x) issue(0, x, x);
  }
  __syncwarp();
  // The team's first row: its sample's maxima, for the sampler.  Everybody waits for the CTA's first threshold, so the other
  // teams' samples come behind the first team's.  (Nothing but time depends on it; a CTA whose rows all lie beyond their windows takes no
  // sample.)
  if (team > 0 && n_live > 0) sift_wait(&st.sample_full[0], 0u, abort_flag);
  if (team < n_live) {
    const int64_t off = st.tab[team].off;
    sift_sample<DTYPE, HAS_U, HAS_T, kTeamThreads>(a, cfg, sample, static_cast<const char*>(row_ptr(a.cond, DTYPE, off)),
                                                   HAS_U ? static_cast<const char*>(row_ptr(a.uncond, DTYPE, off)) : nullptr, tid);
    __syncwarp();
    if (lane == 0) mbar_arrive(&st.sample_full[team]);
  }
  const uint64_t s2 = pack2(a.s, a.s), t2 = pack2(a.inv_T, a.inv_T);
  SiftTarget to;
  to.y_at = smem_u32(list_y + warp * cfg.seg_cap);
  to.id_at = to.scratch_at = smem_u32(list_id + warp * cfg.seg_cap);
  to.hist_at = smem_u32(&sm.hist);
  to.cap = (uint32_t)cfg.seg_cap;
  const uint32_t ring_at = smem_u32(ring);
  uint64_t* const full = st.full + (warp * kMaxTeams + team) * kMaxSlots;
  uint32_t phase = 0;      // bit s: parity of the next phase of full[s]
  int tau_at = 0;          // thresholds come through two places in turn
  uint32_t tau_phase = 0;
  for (int k = team; k < n_live; k += teams) {
    // from the CTA's last row on, the verification grid may be scheduled (it waits for this grid's end)
    if (k == n_live - 1) allow_dependent_launch();
    bool ok = *abort_flag == 0;
    const int x = 2 * team + tau_at;
    if (ok) ok = sift_wait(&st.tau_full[x], tau_phase, abort_flag);
    const SiftBinning bins = sift_bins(st.tau[x].tau0, st.tau[x].top);
    const SiftScreen screen = sift_screen<DTYPE, HAS_U, HAS_T>(a, cfg, st.tau[x].tau0, st.tau[x].u_max);
    __syncwarp();
    if (lane == 0) mbar_arrive(&st.tau_free[x]);
    tau_phase ^= (uint32_t)tau_at;
    tau_at ^= 1;
    uint32_t n = 0;
    float vmax = __int_as_float(0xff800000);
    int slot = (k * units) % slots;
    for (int unit = 0; unit < units; ++unit) {
      if (ok) ok = sift_wait(&full[slot], (phase >> slot) & 1u, abort_flag);
      if (!ok) break;
      phase ^= 1u << slot;
      const uint32_t c_unit = ring_at + (uint32_t)slot * kSlot;
      sift_unit<DTYPE, HAS_U, HAS_T, kToOwn, false>(a, c_unit, c_unit + kUnitBytes, seg_n - unit * EU, (uint32_t)(unit * EU), s2, t2, bins,
                                                    screen, to, lane, n, vmax);
      __syncwarp();
      if (lane == 0) issue(k, unit + slots, slot);
      if (++slot == slots) slot = 0;
    }
    const uint32_t wmax = __reduce_max_sync(0xffffffffu, float_key(vmax));
    if (lane == 0) {
      st.seg_n[team * kTeamWarps + warp] = n;
      atomicMax(&sm.max_key, wmax);
      if (n > to.cap || !ok) sm.over = 1u;
      if (!ok) *abort_flag = 1;
    }
    const SiftRow& r = st.tab[k];
    const int result = finish_row<kTeamWarps, false>(a, cfg, sm, list_y, list_id, st.seg_n + team * kTeamWarps, 1, SiftRuns{}, bins, r.row, r.pos,
                                                     r.iter, r.draft, 0, tid, bar);
    if (result != kRowDone && tid == 0) {
      if (*abort_flag != 0) {
        a.out_cnt[r.row] = 0;
        a.scratch[r.row] = RowScratch{0.0f, -1, 0.0f, kRowStatusTimeout};
      } else {
        SiftTau raised{0.0f, 0.0f, __int_as_float(0x7f800000)};  // (|uncond| not known any more: compared exactly)
        if (result == kRowOver && raise_threshold(sm, bins, cfg.pool - (a.V + EU - 1) / EU, raised)) sift_again(a, st, k, raised);
        else st.redo[atomicAdd(&st.n_redo, 1)] = r.row;
      }
    }
  }
  __syncthreads();
  if (st.n_again != 0) phase = stream_again<DTYPE, HAS_U, HAS_T>(a, cfg, smem_raw, phase);
  if (st.abort != 0 && lane == 0) {
    // a wait gave up: the copies in flight have to land (the wait is bounded) before the CTA may go
    for (int s = 0; s < slots; ++s) {
      const uint32_t u = st.used[(warp * kMaxTeams + team) * kMaxSlots + s];
      if (u > 0) mbar_wait(&full[s], (u - 1u) & 1u);
    }
  }
  // ---- rows the single pass could not finish: the exact any-shape path from global memory (rare)
  const int n_redo = st.n_redo;
  for (int x = 0; x < n_redo; ++x) {
    GenericSmem& gs = *reinterpret_cast<GenericSmem*>(team_sm);
    if (teams == 3) sift_redo<DTYPE, 3 * kTeamThreads, 1>(a, st.redo[x], (int)threadIdx.x, gs);
    else if (teams == 2) sift_redo<DTYPE, 2 * kTeamThreads, 1>(a, st.redo[x], (int)threadIdx.x, gs);
    else sift_redo<DTYPE, kTeamThreads, 1>(a, st.redo[x], (int)threadIdx.x, gs);
  }
}

// ---------------------------------------------------------------------------------------------------
// few rows
// ---------------------------------------------------------------------------------------------------
struct alignas(16) ClusterShared {
  SiftShared row;                                // the first CTA's: histogram of the candidates, finish phase
  SiftSample sample;
  uint32_t key[2][kClusterWarps];                // threshold search: what each warp's count says, in two places used in turn
  uint64_t full[kClusterWarps];                  // a warp's segment has landed
  uint32_t seg_n[kClusterWarps * kMaxCluster];   // candidates per segment (the first CTA's)
  uint32_t lost;                                 // a bounded wait of the cluster gave up (the first CTA's)
  uint32_t again;                                // a list of the cluster ran over (in every CTA)
  uint32_t go;                                   // a row that crowds is sifted once more, with `next` (the first CTA's)
  SiftTau next;
};
// shared memory: ClusterShared | list values | list ids | the warps' own ids | cond | uncond.  The lists (one per segment of the row) are
// complete in the cluster's first CTA, the others fill their segments'; of a row that crowds, one for the whole row in the first CTA
// (see rows_stream_kernel).
__host__ __device__ inline size_t sift_cluster_lists(const SiftCfg& cfg, int n_cta) {
  const size_t b = sizeof(ClusterShared) + (size_t)cfg.pool * 6 + (n_cta > 1 ? (size_t)kClusterWarps * cfg.scratch * 2 : 0);
  return (b + 127) & ~(size_t)127;
}
__host__ __device__ inline size_t sift_cluster_stage(const SiftCfg& cfg, int elem_bytes) {  // one array of one segment
  return ((size_t)cfg.seg_len * elem_bytes + kUnitBytes / 2 - 1) & ~(size_t)(kUnitBytes / 2 - 1);
}
__host__ __device__ inline size_t sift_cluster_smem(const SiftCfg& cfg, int n_cta, int elem_bytes, bool has_u) {
  return sift_cluster_lists(cfg, n_cta) + kClusterWarps * sift_cluster_stage(cfg, elem_bytes) * (has_u ? 2 : 1);
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// the shared-memory address of `p` in the cluster's first CTA
__device__ __forceinline__ uint32_t in_first_cta(const void* p) {
  uint32_t at;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"(smem_u32(p)));
  return at;
}

__device__ __forceinline__ void put_16_bytes(uint32_t at, const uint4& v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// what a warp of the cluster has to say about its segment, to the first CTA (by one lane)
__device__ __forceinline__ void tell_first_cta(ClusterShared& sm, uint32_t max_key, bool over, bool lost) {
  asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" ::"r"(in_first_cta(&sm.row.max_key)), "r"(max_key) : "memory");
  if (over) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(in_first_cta(&sm.row.over)), "r"(1u) : "memory");
  if (lost) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(in_first_cta(&sm.lost)), "r"(1u) : "memory");
}

// A row that crowds, by the whole cluster: sifted once more out of shared memory, with the first CTA's `next` threshold and one
// list for the row.  ok: the warp's segment has landed.  Returns the first CTA's result (kRowElse to the others).
template <int DTYPE, bool HAS_U, bool HAS_T>
__device__ __noinline__ int cluster_crowded_row(const RowArgs& a, const SiftCfg& cfg, unsigned char* smem, int row, bool ok) {
  constexpr int ES = SiftTraits<DTYPE>::kElem, EU = SiftTraits<DTYPE>::kUnit;
  ClusterShared& sm = *reinterpret_cast<ClusterShared*>(smem);
  const uint32_t crank = cluster_rank(), csize = cluster_size();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* const list_y = reinterpret_cast<float*>(smem + sizeof(ClusterShared));
  uint16_t* const list_id = reinterpret_cast<uint16_t*>(list_y + cfg.pool);
  const int room = cfg.pool - kClusterWarps * (int)csize * cfg.units;
  const SiftRuns runs{reinterpret_cast<uint32_t*>(list_y + room), kClusterWarps * (int)csize * cfg.units, cfg.units, cfg.seg_len, EU};
  const size_t stage_bytes = sift_cluster_stage(cfg, ES);
  const uint32_t c_at = smem_u32(smem + sift_cluster_lists(cfg, (int)csize) + (size_t)warp * stage_bytes * (HAS_U ? 2 : 1));
  const int seg = (int)crank * kClusterWarps + warp;
  const int seg_n = min(max(a.V - seg * cfg.seg_len, 0), cfg.seg_len), units = (seg_n + EU - 1) / EU;
  const uint64_t s2 = pack2(a.s, a.s), t2 = pack2(a.inv_T, a.inv_T);
  // whether, and with which threshold, from the first CTA, which stays until everybody knows
  uint32_t go, word[3];
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(go) : "r"(in_first_cta(&sm.go)) : "memory");
#pragma unroll
  for (int k = 0; k < 3; ++k)
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(word[k]) : "r"(in_first_cta(&sm.next) + 4u * k) : "memory");
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  if (go == 0u) return kRowElse;
  const SiftTau tau{__uint_as_float(word[0]), __uint_as_float(word[1]), __uint_as_float(word[2])};
  const SiftBinning bins = sift_bins(tau.tau0, tau.top);
  const SiftScreen screen = sift_screen<DTYPE, HAS_U, HAS_T>(a, cfg, tau.tau0, tau.u_max);
  SiftTarget to;
  to.y_at = in_first_cta(list_y);
  to.id_at = in_first_cta(list_id);
  to.hist_at = in_first_cta(&sm.row.hist);
  to.cap = (uint32_t)room;
  to.taken_at = in_first_cta(&sm.row.taken);
  to.scratch = csize > 1 ? (uint32_t)cfg.scratch : 0u;
  to.scratch_at = smem_u32(csize > 1 ? list_id + cfg.pool + warp * cfg.scratch : list_id);
  const uint32_t runs_at = in_first_cta(runs.run + seg * cfg.units);
  float vmax = __int_as_float(0xff800000);
  bool over = false;
  for (int k = 0; k < cfg.units; ++k) {
    uint32_t run = 0u;  // (segments at the row's end have fewer units)
    if (ok && k < units)
      sift_unit<DTYPE, HAS_U, HAS_T, kToFirst, true>(a, c_at + (uint32_t)k * kUnitBytes, c_at + (uint32_t)(stage_bytes + (size_t)k * kUnitBytes),
                                                 seg_n - k * EU, 0u, s2, t2, bins, screen, to, lane, run, vmax);
    over = over || run == kNoRoom;
    if (lane == 0) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(runs_at + 4u * k), "r"(run) : "memory");
    __syncwarp();  // (the warp's own ids are listed again)
  }
  const uint32_t wmax = __reduce_max_sync(0xffffffffu, float_key(vmax));
  if (lane == 0) tell_first_cta(sm, wmax, over, !ok);
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  if (crank != 0 || sm.lost != 0u) return kRowElse;
  const SiftRow r = sift_row(a, row);
  return finish_row<kClusterWarps, true>(a, cfg, sm.row, list_y, list_id, nullptr, 0, runs, bins, row, r.pos, r.iter, r.draft, kRowStatusRedone,
                                         tid, 0);
}

template <int DTYPE, bool HAS_U, bool HAS_T>
__global__ void __launch_bounds__(kClusterWarps * 32, 1)
rows_cluster_kernel(const __grid_constant__ RowArgs a, const __grid_constant__ SiftCfg cfg) {
  constexpr int NT = kClusterWarps * 32;
  constexpr int ES = SiftTraits<DTYPE>::kElem, EU = SiftTraits<DTYPE>::kUnit;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  ClusterShared& sm = *reinterpret_cast<ClusterShared*>(smem_raw);
  const uint32_t crank = cluster_rank(), csize = cluster_size();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* const list_y = reinterpret_cast<float*>(smem_raw + sizeof(ClusterShared));
  uint16_t* const list_id = reinterpret_cast<uint16_t*>(list_y + cfg.pool);
  const size_t stage_bytes = sift_cluster_stage(cfg, ES);
  unsigned char* const stage = smem_raw + sift_cluster_lists(cfg, (int)csize) + (size_t)warp * stage_bytes * (HAS_U ? 2 : 1);
  const int row = (int)(blockIdx.x / csize);
  const uint64_t s2 = pack2(a.s, a.s), t2 = pack2(a.inv_T, a.inv_T);
  init_shared(sm.row, tid, NT);
  if (tid < kClusterWarps) mbar_init(&sm.full[tid], 1);
  if (tid == 0) {
    sm.lost = sm.again = 0u;
    sm.sample.top_key = sm.sample.u_bits = 0u;
  }
  fence_barrier_init();
  __syncthreads();
  cluster_arrive();  // from here on the first CTA's histogram and lists are ready for the others
  if (tid == 0) {    // this CTA's part of the row into the L2 (see rows_stream_kernel)
    const int b = row / a.W, i = row - b * a.W, at = (int)crank * kClusterWarps * cfg.seg_len;
    const int n = min(max(a.V - at, 0), kClusterWarps * cfg.seg_len);
    const int64_t off = (int64_t)b * a.stride_b + (int64_t)i * a.stride_w + at;
    if (n > 0) {
      ask_l2(row_ptr(a.cond, DTYPE, off), (uint32_t)n * ES);
      if (HAS_U) ask_l2(row_ptr(a.uncond, DTYPE, off), (uint32_t)n * ES);
    }
  }
  __syncwarp();
  grid_dependency_wait();
  allow_dependent_launch();
  const SiftRow r = sift_row(a, row);
  if (!r.live) {  // the whole cluster
    if (crank == 0 && tid == 0) {
      a.out_cnt[row] = 0;
      a.scratch[row] = RowScratch{0.0f, -1, 0.0f, 0};
    }
    __syncwarp();
    cluster_wait();
    return;
  }
  const char* const c_row = static_cast<const char*>(row_ptr(a.cond, DTYPE, r.off));
  const char* const u_row = HAS_U ? static_cast<const char*>(row_ptr(a.uncond, DTYPE, r.off)) : nullptr;
  const int seg = (int)crank * kClusterWarps + warp;
  const int seg0 = seg * cfg.seg_len;
  const int seg_n = min(max(a.V - seg0, 0), cfg.seg_len);
  const int units = (seg_n + EU - 1) / EU;
  unsigned char* const u_stage = stage + stage_bytes;
  bool copied = seg_n > 0;
#ifdef SJD_TEST_DROP_COPY
  // test builds only: one warp's copies are never issued, so that the wait for them runs out and the time-out path
  // (status instead of a hang) can be watched
  if (warp == SJD_TEST_DROP_COPY) copied = false;
#endif
  if (copied && lane == 0) {
    const uint32_t bytes = (uint32_t)seg_n * ES;
    mbar_arrive_expect_tx(&sm.full[warp], bytes * (HAS_U ? 2u : 1u));
    bulk_g2s(stage, c_row + (size_t)seg0 * ES, bytes, &sm.full[warp]);
    if (HAS_U) bulk_g2s(u_stage, u_row + (size_t)seg0 * ES, bytes, &sm.full[warp]);
  }
  __syncwarp();
  // every CTA of the cluster finds the threshold for itself: the sample is small, an exchange would cost more
  sift_sample<DTYPE, HAS_U, HAS_T, NT>(a, cfg, sm.sample, c_row, u_row, tid);
  __syncthreads();
  // the search four bits at a time: warp w counts for the digit w, the largest digit that is reached enough is taken
  uint32_t key;
  bool whole = false;
  {
    static_assert(kClusterWarps == 16, "a warp per digit");
    SiftMaxima m;
    m.load(sm.sample, lane);
    const uint32_t window = window_key(sm.sample);
    const bool near = window != 0u && m.reaching(window) >= (uint32_t)cfg.rank;  // (the same in every warp)
    for (uint32_t rank = (uint32_t)cfg.rank;;) {
      key = near ? window : 0u;
#pragma unroll 1
      for (int shift = near ? 4 : 12; shift >= 0; shift -= 4) {
        const uint32_t mine = key + ((uint32_t)warp << shift);
        const bool reached = warp == 0 || m.reaching(mine) >= rank;  // (a key beyond the largest maximum's is reached by none)
        // (Nobody is more than one barrier ahead: a second barrier for every digit is not needed.  What it cost lies within the runs' spread.)
        uint32_t* const said = sm.key[(shift >> 2) & 1];
        if (lane == 0) said[warp] = reached ? mine : 0u;
        __syncthreads();
        key = __reduce_max_sync(0xffffffffu, said[lane & 15]);
      }
      if (key >= kMaskedKey || whole) break;
      rank = m.reaching(kMaskedKey);  // (the same in every warp)
      if (rank == 0u) break;
      whole = true;
    }
  }
  const SiftTau tau = sift_tau(key, whole, sm.sample);
  const SiftBinning bins = sift_bins(tau.tau0, tau.top);
  const SiftScreen screen = sift_screen<DTYPE, HAS_U, HAS_T>(a, cfg, tau.tau0, tau.u_max);
  SiftTarget to;
  // Every CTA sifts into its own lists and histogram (a segment's place in the lists is the same in all CTAs), and the others send
  // theirs to the first one as a whole.  (Entry by entry, stores and counts into the first CTA's memory held the others up by 3.6 K cycles:
  // 32 rows of 65,536 bf16, K=2,000: 18.8 -> 17.3 us a step; 16 rows of 4,096, a CTA each: 11.9 -> 11.7.)
  to.y_at = smem_u32(list_y + (size_t)seg * cfg.seg_cap);
  to.id_at = to.scratch_at = smem_u32(list_id + (size_t)seg * cfg.seg_cap);
  to.hist_at = smem_u32(&sm.row.hist);
  to.cap = (uint32_t)cfg.seg_cap;
  const uint32_t bias = (uint32_t)((seg % (int)csize) * cfg.seg_len);  // ids are kept relative to the finishing warp's first one
  uint32_t n = 0;
  float vmax = __int_as_float(0xff800000);
  const bool ok = seg_n == 0 || mbar_wait(&sm.full[warp], 0u);
  if (ok) {
    const uint32_t c_at = smem_u32(stage), u_at = smem_u32(u_stage);
    for (int k = 0; k < units; ++k)
      sift_unit<DTYPE, HAS_U, HAS_T, kToShared, false>(a, c_at + (uint32_t)k * kUnitBytes, u_at + (uint32_t)k * kUnitBytes, seg_n - k * EU,
                                                       (uint32_t)(k * EU) + bias, s2, t2, bins, screen, to, lane, n, vmax);
  }
  __syncwarp();
  const uint32_t wmax = __reduce_max_sync(0xffffffffu, float_key(vmax));
  cluster_wait();  // every CTA of the cluster has begun
  if (crank != 0) {
    if (n <= to.cap) {  // (lists end on sixteen bytes)
      const uint32_t y_to = in_first_cta(list_y + (size_t)seg * cfg.seg_cap), id_to = in_first_cta(list_id + (size_t)seg * cfg.seg_cap);
      for (uint32_t k = 16u * (uint32_t)lane; k < 4u * n; k += 512u) put_16_bytes(y_to + k, lds128(to.y_at + k));
      for (uint32_t k = 16u * (uint32_t)lane; k < 2u * n; k += 512u) put_16_bytes(id_to + k, lds128(to.id_at + k));
    }
    __syncthreads();  // (this CTA's histogram is complete)
    const uint32_t* const words = reinterpret_cast<const uint32_t*>(&sm.row.hist);  // the fine bins and behind them the coarse ones
    const uint32_t to_words = in_first_cta(words);
    for (int k = tid; k < kSiftBins + kSiftBins / 32; k += NT)
      if (words[k] != 0u) asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(to_words + 4u * k), "r"(words[k]) : "memory");
  }
  if (lane == 0) {
    const bool over = n > to.cap;
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(in_first_cta(&sm.seg_n[seg])), "r"(n) : "memory");
    tell_first_cta(sm, wmax, over, !ok);
    for (uint32_t c = 0; over && c < csize; ++c) {  // every CTA has to know
      uint32_t at;
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(&sm.again)), "r"(c));
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(1u) : "memory");
    }
  }
  if (!ok && copied) mbar_wait(&sm.full[warp], 0u);  // bounded: no copy of this CTA outlives it
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  const bool again = sm.again != 0u;  // (the same in every CTA)
  if (crank != 0 && !again) return;
  int result = kRowElse;
  if (crank == 0 && sm.lost == 0u)
    result = finish_row<kClusterWarps, false>(a, cfg, sm.row, list_y, list_id, sm.seg_n, (int)csize, SiftRuns{}, bins, row, r.pos, r.iter, r.draft,
                                              0, tid, 0);
  if (again) {
    if (crank == 0 && tid == 0) {
      SiftTau next = tau;
      sm.go = result == kRowOver && raise_threshold(sm.row, bins, cfg.pool - kClusterWarps * (int)csize * cfg.units, next) ? 1u : 0u;
      sm.next = next;
    }
    __syncwarp();
    cluster_arrive();  // (the first CTA has reset what the others count in)
    cluster_wait();
    result = cluster_crowded_row<DTYPE, HAS_U, HAS_T>(a, cfg, smem_raw, row, ok);
    if (crank != 0) return;
  }
  if (sm.lost != 0u) {
    if (tid == 0) {
      a.out_cnt[row] = 0;
      a.scratch[row] = RowScratch{0.0f, -1, 0.0f, kRowStatusTimeout};
    }
    return;
  }
  if (result != kRowDone) sift_redo<DTYPE, NT, 0>(a, row, tid, *reinterpret_cast<GenericSmem*>(&sm.sample));
}

}  // namespace sjd
