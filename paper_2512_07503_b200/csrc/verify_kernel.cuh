// Verification stage of the step (paper Section 4.1, Steps 3 and 4): the accept test of Eq. acc-sjdpp
// on every row, the first-rejection prefix, the residual draw of Eq. rej-sjd at the first rejected row,
// and the reuse-or-redraw rule of Eq. reuse (Eq. refine-sjd when reuse is off) for the rows after it.
// One CTA per sequence; it reads what the row stage left in RowScratch and in out_probs.
#pragma once

#include "device_utils.cuh"
#include "row_kernels.cuh"

namespace sjd {

constexpr int kFlagReuse = 1;
constexpr int kFlagDraftAll = 2;
constexpr int kQUniform = -1;

constexpr int kOutInvalid = 0, kOutAccepted = 1, kOutResidual = 2, kOutReused = 3, kOutResampled = 4;
constexpr int kStatusQtok = 1, kStatusEmptyResidual = 2, kStatusDegenerate = 4, kStatusTimeout = 8, kStatusRedone = 16;

// a cache line into the L2
__device__ __forceinline__ void ask_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

struct VerifyArgs {
  int B, W, V, kcap;
  int flags;
  float tau;
  const int32_t* win_len;
  const int32_t* pos_base;
  const int32_t* iteration;
  int iteration0;
  int seq_base;
  uint32_t seed_lo, seed_hi;
  const int32_t* drafts;
  // previous-iteration distributions
  const float* q_tok;
  const int32_t* q_ids;
  const float* q_vals;
  const int32_t* q_cnt;
  // this call's distributions (written by the row stage)
  const int32_t* p_ids;
  const float* p_vals;
  const RowScratch* scratch;
  // outputs
  int32_t* out_accept_len;
  int32_t* out_tokens;
  float* out_tok_prob;
  int32_t* out_flags;
  int32_t* status;
};

// ratio p/q of Eq. acc-sjdpp and of the confidence C (the same quantity), with the conventions for
// the corner cases: p == 0 gives 0 (never accepted, never reused); q <= 0 with p > 0 gives +inf.
__device__ __forceinline__ float likelihood_ratio(float p, float q) {
  if (p == 0.0f) return 0.0f;
  if (!(q > 0.0f)) return __int_as_float(0x7f800000);
  return __fdiv_rn(p, q);
}

constexpr int kVerifyThreads = 512;     // >= SJD_W_MAX: a thread per window row
constexpr int kVerifyShort = 4 * kVerifyThreads;  // entries of a row that is not LONG
constexpr int kVerifyStage = 8192;      // without the map: words of the previous iteration's row staged in shared memory
constexpr int kVerifyAsked = 4;         // rows of the previous iteration's distributions asked into the L2 early

struct VerifySmem {
  uint64_t warp_sum[2][kVerifyThreads / 32];
  uint64_t random;                // of the rejected row
  int first_reject;
  int status;
  int q_cnt[kVerifyThreads];      // of every window row
};
static_assert(sizeof(VerifySmem) % 16 == 0, "the map behind it is cleared sixteen bytes at a time");
// Behind it, where an id lies in the previous iteration's row.  kMapVals: a bit for every id of the vocabulary, for each word of bits the
// position of its first entry (16 bits), and the row's probabilities: a lookup is a bit, a population count and an addition.  kMap:
// without the probabilities, where they would be too much.  kNoMap (vocabularies of a million ids): the ids themselves, of a very
// long row every stride-th, to be searched by halving, and the probabilities of a row that is not LONG.
enum { kNoMap = 0, kMap = 1, kMapVals = 2 };
__host__ __device__ inline int verify_map_words(int V) { return V / 128 * 4 + 4; }
__host__ __device__ inline size_t verify_smem(int V, int kcap, bool is_long, int map) {
  if (map == kNoMap) return sizeof(VerifySmem) + (is_long ? (size_t)kVerifyStage * 4 : (size_t)kVerifyShort * 8);
  return sizeof(VerifySmem) + (size_t)verify_map_words(V) * 6 + (map == kMapVals ? (size_t)(kcap + 3) / 4 * 16 : 0);
}
// the best that fits
inline int verify_map(int V, int kcap, bool is_long, size_t limit) {
  if (kcap > 65536) return kNoMap;
  return verify_smem(V, kcap, is_long, kMapVals) <= limit ? kMapVals : is_long && verify_smem(V, kcap, is_long, kMap) <= limit ? kMap : kNoMap;
}

// One CTA per sequence.  Latency is all there is to it (it sits between two row kernels), so nothing is waited for
// that could have been asked for earlier: what does not come from the row stage is loaded, the random numbers are drawn and the
// map is cleared before the wait for that stage; both rows of the residual draw come in with one round of loads, without
// branches (a load in one is waited for where the branch ends); what does not depend on the draw is written meanwhile.  A warp
// owns consecutive entries of the rejected row, a lane every 32nd of them; only the warp that the draw falls to locates it.
//
// LONG: rows of more than 2,048 entries, a warp's taken sixteen groups of 32 at a time.
// MANY: more sequences than SMs (launch_verify()): two CTAs to an SM.  One CTA of 72 registers a thread (128 where it is LONG) fills an SM, and then
// the sequences go in rounds; where there is one round, registers shorten the only CTA's way (1,024 rows in 32 sequences 73.2 us a step with 64
// registers, 70.8 with 72; in 512 of two rows 78.7, 81.4).  LONG rows then come four groups at a time: sixteen do not fit, eight are no faster.
//
// The map, the loads without branches and the early requests against a search by halving in the row itself, from the row stage's end to a
// CTA's own, thousands of cycles: 16 rows of K=64 7.4 -> 4.9, 1,024 rows of K=2,000 11.3 -> 7.3, of K=8,192 85 -> 14.7 (a step: 77.9 -> 74.6
// us, 171 -> 142 us); 128 rows of V=131,072, K=8,192 73.2 -> 55.8 us a step; 32 rows of K=V=65,536 (without probabilities in the map) 597 -> 378 us.
template <bool LONG, int LOOK, bool MANY>
__global__ void __launch_bounds__(kVerifyThreads, MANY ? 2 : 1) verify_kernel(const VerifyArgs a) {
  constexpr int NT = kVerifyThreads, NW = NT / 32, E = LONG && !MANY ? 16 : 4;
  constexpr bool MAP = LOOK != kNoMap, VALS = LOOK == kMapVals || (LOOK == kNoMap && !LONG);  // VALS: the probabilities are staged
  extern __shared__ __align__(128) unsigned char smem_raw[];
  VerifySmem& sm = *reinterpret_cast<VerifySmem*>(smem_raw);
  const int words = MAP ? verify_map_words(a.V) : 0;
  uint32_t* const map_bits = reinterpret_cast<uint32_t*>(smem_raw + sizeof(VerifySmem));
  uint16_t* const map_first = reinterpret_cast<uint16_t*>(map_bits + words);
  int32_t* const look_id = reinterpret_cast<int32_t*>(map_bits);
  float* const look_val = MAP ? reinterpret_cast<float*>(map_first + words) : reinterpret_cast<float*>(look_id + kVerifyShort);
  const int b = blockIdx.x, i = threadIdx.x, lane = i & 31, warp = i >> 5, W = a.W, kcap = a.kcap;
  const bool draft_all = (a.flags & kFlagDraftAll) != 0;
  const bool reuse_on = (a.flags & kFlagReuse) != 0;
  const size_t base = (size_t)b * W;
  // Inputs of the call: written before the row kernel began, which waits for that itself before it lets this grid start.
  const int L = a.win_len ? min(max(a.win_len[b], 0), W) : W;
  const int pos0 = a.pos_base ? a.pos_base[b] : 0;
  const int iter = a.iteration ? a.iteration[b] : a.iteration0;
  const uint32_t seq = (uint32_t)(a.seq_base + b);
  float q_tok = 0.0f, u = 0.0f;
  int draft = -1;
  uint64_t random = 0;
  if (!draft_all && i < L) {
    q_tok = a.q_tok[base + i];
    draft = a.drafts[base + i];
    sm.q_cnt[i] = a.q_cnt[base + i];
    u = uniform24(philox4x32_10((uint32_t)(pos0 + i), seq, (uint32_t)iter, kPurposeAccept, a.seed_lo, a.seed_hi).x0);
    random = random64(philox4x32_10((uint32_t)(pos0 + i), seq, (uint32_t)iter, kPurposeResidual, a.seed_lo, a.seed_hi));
  }
  if constexpr (MAP) {
    if (!draft_all)
      for (int k = i; k < words / 4; k += NT) reinterpret_cast<uint4*>(map_bits)[k] = make_uint4(0u, 0u, 0u, 0u);
  }
  // (the draw most often falls to one of the first rows; an address that this SM has not met lately is found out as well)
  if (!draft_all && warp < min(kVerifyAsked, L)) {
    const size_t at = (base + warp) * (size_t)kcap;
    const int n = min(a.q_cnt[base + warp], kcap);
    for (int k = 32 * lane; k < n; k += 1024) {
      ask_line(a.q_ids + at + k);
      ask_line(a.q_vals + at + k);
    }
    if (lane == 0) {
      ask_line(a.p_ids + at);
      ask_line(a.p_vals + at);
    }
  }
  if (i == 0) {
    sm.first_reject = L;
    sm.status = 0;
  }
  __syncthreads();
  // Launched with programmatic stream serialisation right behind the row kernel: the grid may be scheduled while that
  // kernel's last rows are still running, and waits here until all of its writes are visible.  A no-op after an
  // ordinary launch.
  grid_dependency_wait();
  // a following kernel that waits the same way (the next step's row kernel) may set itself up meanwhile
  allow_dependent_launch();

  // Step 3: r < min(1, p(x_i)/q(x_i)) on every valid row; the counter-based generator makes the rows independent, so
  // they are all tested at once
  RowScratch rs{0.0f, -1, 0.0f, 0};
  float ratio = 0.0f;
  {
    int st = 0;
    bool rejected = false;
    if (i < L) {
      rs = a.scratch[base + i];
      if (rs.status & kRowStatusDegenerate) st |= kStatusDegenerate;
      if (rs.status & kRowStatusTimeout) st |= kStatusTimeout;
      if (rs.status & kRowStatusRedone) st |= kStatusRedone;
      if (!draft_all) {
        ratio = likelihood_ratio(rs.p_tok, q_tok);
        rejected = !(u < fminf(ratio, 1.0f));
        if (!(q_tok > 0.0f)) st |= kStatusQtok;
      }
    }
    const uint32_t votes = __ballot_sync(0xffffffffu, rejected);
    if (lane == 0 && votes != 0u) atomicMin(&sm.first_reject, i + __ffs((int)votes) - 1);
    if (st) atomicOr(&sm.status, st);
  }
  __syncthreads();
  const int acc = draft_all ? 0 : sm.first_reject;
  const bool draw = !draft_all && acc < L;

  // Step 4, the rows that do not wait for a draw, and the outputs
  auto put_rows = [&] {
    if (i < W && !(draw && i == acc)) {
      int tok = -1, flag = kOutInvalid;
      float pr = 0.0f;
      if (i < L) {
        if (draft_all) {
          tok = rs.samp_tok; pr = rs.samp_prob; flag = kOutResampled;
        } else if (i < acc) {
          tok = draft; pr = rs.p_tok; flag = kOutAccepted;
        } else if (reuse_on && rs.p_tok > 0.0f && ratio > a.tau) {  // the ratio is the confidence of Eq. (C)
          tok = draft; pr = rs.p_tok; flag = kOutReused;
        } else {
          tok = rs.samp_tok; pr = rs.samp_prob; flag = kOutResampled;
        }
      }
      a.out_tokens[base + i] = tok;
      a.out_tok_prob[base + i] = pr;
      if (a.out_flags) a.out_flags[base + i] = flag;
    }
    if (i == 0) a.out_accept_len[b] = acc;
  };
  if (!draw) {
    put_rows();
    if (i == 0 && a.status) a.status[b] = sm.status;
    return;
  }
  if (i == acc) sm.random = random;

  // Step 4, first rejected row: draw from max(0, p - q) / sum max(0, p - q).  Warp w owns 32 * per consecutive entries of p_a
  // (ascending token id).
  const size_t row = (base + acc) * (size_t)kcap;
  const int32_t* const pid = a.p_ids + row;
  const float* const pv = a.p_vals + row;
  const int32_t* const qid = a.q_ids + row;
  const float* const qv = a.q_vals + row;
  const int per = (kcap + NT - 1) / NT;  // groups of 32 per warp: up to E unless LONG
  const int own0 = warp * per * 32 + lane;
  int id[E];
  float p[E];
  auto load = [&](int j0) {
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const int k = own0 + 32 * (j0 + j);
      id[j] = -1;
      p[j] = 0.0f;
      if (j0 + j < per && k < kcap) {
        id[j] = pid[k];
        p[j] = pv[k];
      }
    }
  };
  load(0);
  // the previous iteration's row
  const int qc = sm.q_cnt[acc];
  const int n = min(max(qc, 0), kcap);  // a uniform row has no list
  int stride = 1;
  int x[E], last[E];  // ids, and (first lane) the id before them
  float y[E];
  auto load_reference = [&](int k0) {
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const int k = k0 + j * NT;
      x[j] = last[j] = -1;  // (of another word than any there is)
      y[j] = 0.0f;
      if (k < n) x[j] = qid[k];
      if (MAP && lane == 0 && k > 0 && k < n) last[j] = qid[k - 1];
      if (VALS && k < n) y[j] = qv[k];
    }
  };
  if constexpr (MAP || !LONG) load_reference(i);
  put_rows();
  if constexpr (MAP) {
    for (int k0 = i;;) {
#pragma unroll
      for (int j = 0; j < E; ++j) {
        const int k = k0 + j * NT, own = x[j];
        int before = __shfl_up_sync(0xffffffffu, own, 1);
        if (lane == 0) before = last[j];
        if (VALS && k < n) look_val[k] = y[j];
        if ((uint32_t)own < (uint32_t)a.V) {  // (-1 beyond the list's end)
          atomicOr(&map_bits[own >> 5], 1u << (own & 31));
          if ((before >> 5) != (own >> 5)) map_first[own >> 5] = (uint16_t)k;
        }
      }
      k0 += E * NT;
      if (!LONG || k0 - i >= n) break;
      load_reference(k0);
    }
  } else if constexpr (!LONG) {
#pragma unroll
    for (int j = 0; j < E; ++j) {
      look_id[i + j * NT] = x[j];
      look_val[i + j * NT] = y[j];
    }
  } else {
    stride = (n + kVerifyStage - 1) / kVerifyStage;
    for (int k = i; k * stride < n; k += NT) look_id[k] = qid[k * stride];
  }
  __syncthreads();
  const float unlisted = qc == kQUniform ? __fdiv_rn(1.0f, (float)a.V) : 0.0f;
  const int staged = n > 0 ? (n + stride - 1) / stride : 0;
  // the previous iteration's probability of a token
  auto reference = [&](int token) {
    float q = unlisted;
    if constexpr (MAP) {
      const uint32_t at_word = min((uint32_t)token, (uint32_t)a.V - 1u) >> 5, bit = 1u << (token & 31);
      const uint32_t word = map_bits[at_word];
      const int at = max(min((int)map_first[at_word] + __popc(word & (bit - 1u)), n - 1), 0);
      if constexpr (VALS) {
        const float v = look_val[at];  // (whether or not: a load is cheaper than a branch)
        q = (word & bit) != 0u ? v : q;
      } else {
        if ((word & bit) != 0u) q = qv[at];
      }
    } else if (n > 0) {
      // largest staged position whose id does not exceed the wanted one
      int at = 0;
      for (int half = 1 << (31 - __clz(staged)); half > 0; half >>= 1)
        if (at + half < staged && look_id[at + half] <= token) at += half;
      if constexpr (!LONG) {
        if (look_id[at] == token) q = look_val[at];
      } else {
        at *= stride;
        const int end = min(at + stride, n);
        while (at + 1 < end && qid[at + 1] <= token) ++at;
        if (qid[at] == token) q = qv[at];
      }
    }
    return q;
  };
  // what q leaves of the loaded entries, or p itself (nothing where there is no entry: its p is zero)
  float w[E];
  bool from_p = false;
  auto weigh = [&] {
#pragma unroll
    for (int j = 0; j < E; ++j) w[j] = from_p ? p[j] : __fsub_rn(p[j], reference(id[j]));
  };
  for (;;) {
    uint64_t local = 0;
    for (int j0 = 0; j0 < per; j0 += E) {
      if (LONG && per > E && (j0 > 0 || from_p)) load(j0);
      weigh();
#pragma unroll
      for (int j = 0; j < E; ++j) local += fixed_weight(w[j]);
    }
    local = warp_sum_u64(local);
    if (lane == 0) sm.warp_sum[from_p][warp] = local;
    __syncthreads();
    const uint64_t sum = lane < NW ? sm.warp_sum[from_p][lane] : 0ull;
    const uint64_t T = warp_sum_u64(sum);
    uint64_t before = warp_sum_u64(lane < warp ? sum : 0ull);
    if (T == 0 && !from_p) {  // the residual weights sum to zero after rounding: p itself
      from_p = true;
      continue;
    }
    if (i == 0 && a.status) a.status[b] = sm.status | (from_p ? kStatusEmptyResidual : 0);
    auto emit = [&](int token, float prob) {
      a.out_tokens[base + acc] = token;
      a.out_tok_prob[base + acc] = prob;
      if (a.out_flags) a.out_flags[base + acc] = kOutResidual;
    };
    if (T == 0) {  // nothing but zeros: the first entry
      if (i == 0) emit(pid[0], pv[0]);
      return;
    }
    const uint64_t t = __umul64hi(sm.random, T);
    if (!(t >= before && t < before + local)) return;  // the whole warp
    for (int j0 = 0; j0 < per; j0 += E) {
      if (LONG && per > E) {
        load(j0);
        weigh();
      }
      // the group of 32 that the draw falls to, then the entry
      uint64_t group[E];
#pragma unroll
      for (int j = 0; j < E; ++j) group[j] = warp_sum_u64(fixed_weight(w[j]));
      int at_id = 0;
      float at_p = 0.0f;
      uint64_t own = 0;
      bool found = false;
#pragma unroll
      for (int j = 0; j < E; ++j) {
        if (found) continue;
        found = t < before + group[j];
        if (found) {
          own = fixed_weight(w[j]);
          at_id = id[j];
          at_p = p[j];
        } else {
          before += group[j];
        }
      }
      if (!found) continue;
      uint64_t upto = own;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint64_t o = shfl_up_u64(upto, d);
        if (lane >= d) upto += o;
      }
      upto += before;
      if (t < upto && t >= upto - own) emit(at_id, at_p);
      return;
    }
  }
}

}  // namespace sjd
