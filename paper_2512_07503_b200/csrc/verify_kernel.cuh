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
constexpr int kVerifyItems = 4;         // entries of the rejected row per thread and round: 2,048 a round
constexpr int kVerifyStage = 8192;      // words of the previous iteration's row staged in shared memory

struct VerifySmem {
  uint64_t scan[2 * 32 + 8];
  // ids of the previous iteration's row (of a very long one every stride-th), and behind the first 2,048 the
  // probabilities when the whole row fits in 2,048 entries
  alignas(16) int32_t q[kVerifyStage];
  int32_t q_cnt[kVerifyThreads];  // of every window row
  int first_reject;
  int status;
  int res_tok;
  float res_prob;
};

// One CTA per sequence.  Latency is all there is to it (it sits between two row kernels), so nothing is waited for
// that could have been asked for earlier: what does not come from the row stage is loaded, and the accept tests' random
// numbers are drawn, before the wait for that stage; both rows of the residual draw come in with one round of loads; the
// lookups of a thread's four entries share one search.  16 sequences of 64 rows, K=2,000: 8.4 us under ncu
// (12.1 before), and 3 us less of a step (one window of 32 rows: 25.5 -> 21.4 us).
//
// LONG: rows of more than 2,048 entries, taken in rounds (1,024 rows of K=8,192: 294 -> 235 us a step).
template <bool LONG>
__global__ void __launch_bounds__(kVerifyThreads) verify_kernel(const VerifyArgs a) {
  constexpr int NT = kVerifyThreads, ITEMS = kVerifyItems;
  __shared__ VerifySmem sm;
  const int b = blockIdx.x, i = threadIdx.x, W = a.W;
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
  if (!draft_all && i < L) {
    q_tok = a.q_tok[base + i];
    draft = a.drafts[base + i];
    sm.q_cnt[i] = a.q_cnt[base + i];
    u = uniform24(philox4x32_10((uint32_t)(pos0 + i), seq, (uint32_t)iter, kPurposeAccept, a.seed_lo, a.seed_hi).x0);
  }
  if (i == 0) {
    sm.first_reject = L;
    sm.status = 0;
    sm.res_tok = -1;
    sm.res_prob = 0.0f;
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
  if (i < L) {
    rs = a.scratch[base + i];
    int st = (rs.status & kRowStatusDegenerate) ? kStatusDegenerate : 0;
    if (rs.status & kRowStatusTimeout) st |= kStatusTimeout;
    if (rs.status & kRowStatusRedone) st |= kStatusRedone;
    if (!draft_all) {
      ratio = likelihood_ratio(rs.p_tok, q_tok);
      if (!(u < fminf(ratio, 1.0f))) atomicMin(&sm.first_reject, i);
      if (!(q_tok > 0.0f)) st |= kStatusQtok;
    }
    if (st) atomicOr(&sm.status, st);
  }
  __syncthreads();
  const int acc = draft_all ? 0 : sm.first_reject;

  // Step 4, first rejected row: draw from max(0, p - q) / sum max(0, p - q).  Every thread owns a run of consecutive entries
  // of p_a (ascending token id), so one scan of the per-thread sums locates the draw.
  if (!draft_all && acc < L) {
    const size_t r = base + acc;
    const int kcap = a.kcap;
    const int32_t* pid = a.p_ids + r * kcap;
    const float* pv = a.p_vals + r * kcap;
    const int32_t* qid = a.q_ids + r * kcap;
    const float* qv = a.q_vals + r * kcap;
    const int qc = sm.q_cnt[acc];
    const float q_uniform = __fdiv_rn(1.0f, (float)a.V);
    const uint64_t R = random64(philox4x32_10((uint32_t)(pos0 + acc), seq, (uint32_t)iter, kPurposeResidual, a.seed_lo, a.seed_hi));
    const int rounds = LONG ? (kcap + NT * ITEMS - 1) / (NT * ITEMS) : 1;
    const int k0 = i * ITEMS * rounds;  // this thread's run of consecutive entries
    int id[ITEMS];
    float p[ITEMS], w[ITEMS];
    // whole runs of four as one load each where the arrays' alignment allows it
    const bool vec = (kcap & 3) == 0 && ((reinterpret_cast<uintptr_t>(a.p_ids) | reinterpret_cast<uintptr_t>(a.p_vals) |
                                          reinterpret_cast<uintptr_t>(a.q_ids) | reinterpret_cast<uintptr_t>(a.q_vals)) & 15u) == 0;
    auto load4 = [&](const int32_t* ids, const float* vals, int k, int len, int (&to_id)[ITEMS], float (&to_val)[ITEMS]) {
      if (vec) {
        const int4 x = k < len ? *reinterpret_cast<const int4*>(ids + k) : make_int4(-1, -1, -1, -1);
        const float4 y = k < len ? *reinterpret_cast<const float4*>(vals + k) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        to_id[0] = x.x; to_id[1] = x.y; to_id[2] = x.z; to_id[3] = x.w;
        to_val[0] = y.x; to_val[1] = y.y; to_val[2] = y.z; to_val[3] = y.w;
        return;
      }
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const bool in = k + j < len;
        to_id[j] = in ? ids[k + j] : -1;
        to_val[j] = in ? vals[k + j] : 0.0f;
      }
    };
    auto load = [&](int k) { load4(pid, pv, k, kcap, id, p); };
    const int n = min(max(qc, 0), kcap);  // a uniform row has no list
    int stride = 1;
    if (!LONG) {
      // all loads at once
      int qi[ITEMS];
      float qw[ITEMS];
      load(k0);
      load4(qid, qv, k0, n, qi, qw);
      *reinterpret_cast<int4*>(&sm.q[k0]) = make_int4(qi[0], qi[1], qi[2], qi[3]);
      *reinterpret_cast<float4*>(&sm.q[NT * ITEMS + k0]) = make_float4(qw[0], qw[1], qw[2], qw[3]);
    } else {
      stride = (n + kVerifyStage - 1) / kVerifyStage;
      for (int k = i; k * stride < n; k += NT) sm.q[k] = qid[k * stride];
    }
    __syncthreads();
    const int staged = n > 0 ? (n + stride - 1) / stride : 0;
    // weights of the four entries in id / p: what q leaves of p
    auto residual = [&](int k) {
      // largest staged position whose id does not exceed the wanted one: by halving for the first of the four, by steps
      // from there for the others: both rows ascend and hold about as many entries, so one or two steps do (four searches
      // by halving in step: 5.7 K cycles of the kernel's 14 K, this 4.7 K; a hash table 7 K and 4 K to fill; neighbouring
      // entries to neighbouring lanes 3.1 K, but more for locating the draw than that saves).  Where the other row's ids crowd
      // between two of these eight steps do not get there, and the rest goes by halving again.
      int lo[ITEMS];
      int at = 0;
      auto halve = [&](int wanted) {
        for (int half = n > 0 ? 1 << (31 - __clz(staged)) : 0; half > 0; half >>= 1)
          if (at + half < staged && sm.q[at + half] <= wanted) at += half;
      };
      halve(id[0]);
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        if (j > 0) {
          int steps = 8;
          while (at + 1 < staged && sm.q[at + 1] <= id[j] && steps > 0) ++at, --steps;
          if (steps == 0) halve(id[j]);
        }
        lo[j] = at;
      }
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        float q = qc == kQUniform ? q_uniform : 0.0f;
        if (n > 0) {
          if (!LONG) {
            if (sm.q[lo[j]] == id[j]) q = reinterpret_cast<const float*>(sm.q)[NT * ITEMS + lo[j]];
          } else {
            int at = lo[j] * stride;
            const int end = min(at + stride, n);
            while (at + 1 < end && qid[at + 1] <= id[j]) ++at;
            if (qid[at] == id[j]) q = qv[at];
          }
        }
        w[j] = k + j < kcap ? __fsub_rn(p[j], q) : 0.0f;
      }
    };
    int flip = 0;
    uint64_t T = 0, before = 0, local = 0;
    bool from_p = false;
    for (;;) {
      // residual weights first; p itself only when they sum to zero after rounding
      local = 0;
      for (int r = 0; r < rounds; ++r) {
        if (LONG) load(k0 + ITEMS * r);
        if (!from_p) residual(k0 + ITEMS * r);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
          if (from_p) w[j] = p[j];
          local += fixed_weight(w[j]);
        }
      }
      before = group_scan1<NT, 0, uint64_t>(local, i, sm.scan, flip, &T);
      if (T != 0 || from_p) break;
      if (i == 0) sm.status |= kStatusEmptyResidual;
      from_p = true;
    }
    const uint64_t t = __umul64hi(R, T);
    if (T == 0 ? i == 0 : (t >= before && t < before + local)) {
      int j = 0;
      if (T == 0) {
        load(0);  // nothing but zeros: the first entry
      } else {
        for (int r = 0; r < rounds; ++r) {
          if (LONG) {
            load(k0 + ITEMS * r);
            if (!from_p) residual(k0 + ITEMS * r);
          }
          uint64_t sum = 0;
          j = 0;
#pragma unroll
          for (int x = 0; x < ITEMS; ++x) {
            sum += fixed_weight(LONG && from_p ? p[x] : w[x]);
            if (t >= before + sum) j = x + 1;
          }
          if (j < ITEMS) break;  // comes true: t < before + local
          before += sum;
        }
      }
      sm.res_tok = j == 0 ? id[0] : j == 1 ? id[1] : j == 2 ? id[2] : id[3];
      sm.res_prob = j == 0 ? p[0] : j == 1 ? p[1] : j == 2 ? p[2] : p[3];
    }
  }
  __syncthreads();

  // Step 4, remaining rows, and the outputs
  if (i < W) {
    int tok = -1, flag = kOutInvalid;
    float pr = 0.0f;
    if (i < L) {
      if (draft_all) {
        tok = rs.samp_tok; pr = rs.samp_prob; flag = kOutResampled;
      } else if (i < acc) {
        tok = draft; pr = rs.p_tok; flag = kOutAccepted;
      } else if (i == acc) {
        tok = sm.res_tok; pr = sm.res_prob; flag = kOutResidual;
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
  if (i == 0) {
    a.out_accept_len[b] = acc;
    if (a.status) a.status[b] = sm.status;
  }
}

}  // namespace sjd
