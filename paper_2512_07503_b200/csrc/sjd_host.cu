// Host-buffer variant of the step (declared in include/sjd.h): device mirrors of every argument are
// allocated once per context; each call copies in, runs sjd_step() and copies out.
//
// The link to the host is what bounds it: 50 GB/s, and some 4 us for every copy whatever its size.  So
//   - the batch goes through in parts of whole sequences: while a part's logits are on their way in, the part before it is
//     in the kernels and the one before that on its way out (three streams; the parts use the mirrors' own ranges, and
//     sequence numbers by seq_base; a row's result does not depend on how many rows a call has, except that a row which one of
//     the row kernels has to redo agrees with the other's to rounding only);
//   - the small arrays of a call are gathered in page-locked memory, from which a kernel fetches them while the
//     first logits come in, and into which the kernels write the small results: no copies of their own;
//   - of the previous iteration's distributions one row per sequence is needed, and only the verification knows which: it
//     reads that row out of the caller's arrays if they are page-locked.  Pageable ones are copied whole.
// Pinned bf16 logits, W=32, V=16,384, K=1,000, both logit arrays: B=4 (8.4 MB of logits, 168 us of the link) 296 -> 233 us, B=32
// 1,640 -> 1,370 us (1,340 of the link).  One part only: 238 us at B=4.
#include "../../include/sjd.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>

#include "host_piece.h"

namespace {

// Every part has at least this many bytes of logits (where there is more than one): each costs two to four copies more, and hides its
// kernels and its copies out behind the others.  The case above in parts of 2, 3, 4 and 8 MB: 252, 250, 233, 238 us; B=32: at
// most four parts 1,402 us, eight 1,383.
constexpr size_t kPartBytes = 4 << 20;
constexpr int kMaxParts = 8;

}  // namespace

struct sjd_host_ctx {
  int32_t B, W, V, dtype, top_k, kcap;
  size_t rows, row_bytes;
  char* arena;  // the device mirrors, one allocation
  char *d_cond, *d_uncond;
  sjd_probs d_q, d_out;  // (only the lists: ids and vals)
  int32_t* d_small;      // window lengths, positions, iterations; drafts and their probabilities and list lengths
  int32_t *h_small, *h_results, *m_small, *m_results;  // page-locked: the same, and the small results; as the device sees them
  void* d_ws;
  size_t ws_bytes;
  cudaStream_t in, run, out;
  cudaEvent_t arrived[kMaxParts], stepped[kMaxParts];
};

namespace {

__global__ void fetch_words(const int32_t* __restrict__ from, int32_t* __restrict__ to, int n) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i < n) to[i] = from[i];
}

// The device's address of a host array that one page-locked and mapped piece of memory holds, else null.
template <typename T>
T* mapped(T* p, size_t bytes) {
  using Query = CUresult (*)(void*, CUpointer_attribute, CUdeviceptr);
  static const Query query = [] {  // (through the runtime: no link against the driver library)
    void* f = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPoint("cuPointerGetAttribute", &f, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess) f = nullptr;
    return reinterpret_cast<Query>(f);
  }();
  return static_cast<T*>(sjd::device_address_of(p, bytes, [](const void* at, sjd::HostPiece* piece) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, at) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
    if (attr.type != cudaMemoryTypeHost || !attr.devicePointer || !query) return false;
    piece->device = static_cast<char*>(attr.devicePointer);
    const CUdeviceptr d = reinterpret_cast<CUdeviceptr>(attr.devicePointer);
    return query(&piece->start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, d) == CUDA_SUCCESS &&
           query(&piece->size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, d) == CUDA_SUCCESS;
  }));
}

void drain(sjd_host_ctx* c) {
  if (c->in) cudaStreamSynchronize(c->in);
  if (c->run) cudaStreamSynchronize(c->run);
  if (c->out) cudaStreamSynchronize(c->out);
}

bool create(sjd_host_ctx* c) {
  const size_t rows = c->rows, B = (size_t)c->B, lists = rows * (size_t)c->kcap * 4, logits = rows * c->row_bytes;
  const size_t n_in = (3 * B + 3 * rows) * 4, n_out = (2 * B + 4 * rows) * 4;
  const size_t sizes[] = {logits, logits, lists, lists, lists, lists, n_in, c->ws_bytes};
  size_t at[9] = {0};
  for (int i = 0; i < 8; ++i) at[i + 1] = at[i] + ((sizes[i] + 255) & ~(size_t)255);
  if (cudaMalloc(reinterpret_cast<void**>(&c->arena), at[8]) != cudaSuccess) return false;
  auto words = [&](int i) { return reinterpret_cast<int32_t*>(c->arena + at[i]); };
  c->d_cond = c->arena;
  c->d_uncond = c->arena + at[1];
  c->d_q.ids = words(2);
  c->d_q.vals = reinterpret_cast<float*>(words(3));
  c->d_out.ids = words(4);
  c->d_out.vals = reinterpret_cast<float*>(words(5));
  c->d_small = words(6);
  c->d_ws = words(7);
  if (cudaHostAlloc(reinterpret_cast<void**>(&c->h_small), n_in + n_out, cudaHostAllocMapped) != cudaSuccess ||
      cudaHostGetDevicePointer(reinterpret_cast<void**>(&c->m_small), c->h_small, 0) != cudaSuccess)
    return false;
  c->h_results = c->h_small + n_in / 4;
  c->m_results = c->m_small + n_in / 4;
  for (cudaStream_t* st : {&c->in, &c->run, &c->out})
    if (cudaStreamCreateWithFlags(st, cudaStreamNonBlocking) != cudaSuccess) return false;
  for (int i = 0; i < kMaxParts; ++i)
    if (cudaEventCreateWithFlags(&c->arrived[i], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->stepped[i], cudaEventDisableTiming) != cudaSuccess)
      return false;
  return true;
}

#define SJD_TRY(expr)                   \
  do {                                  \
    if ((expr) != cudaSuccess) return SJD_ERR_CUDA; \
  } while (0)

// Everything that a call enqueues; the caller drains the streams whatever it returns.
int enqueue(sjd_host_ctx* c, const char* cond, const char* uncond, const int32_t* drafts, const sjd_probs* q,
            const sjd_params* P, uint64_t seed, sjd_probs* out) {
  const cudaMemcpyKind H2D = cudaMemcpyHostToDevice, D2H = cudaMemcpyDeviceToHost;
  const size_t rows = c->rows, B = (size_t)c->B, W = (size_t)c->W, kc = (size_t)c->kcap, n_logits = W * c->row_bytes;
  size_t parts = B < kMaxParts ? B : kMaxParts;
  while (parts > 1 && B / parts * n_logits * (uncond ? 2 : 1) < kPartBytes) --parts;  // (the smallest part)
  int32_t* const d_win = c->d_small;
  int32_t* const d_drafts = c->d_small + 3 * B;
  int32_t* const m_tokens = c->m_results + 2 * B;
  sjd_probs d_q = c->d_q;
  bool q_copied = false;
  for (size_t k = 0; k < parts; ++k) {
    const size_t b0 = k * B / parts, nb = (k + 1) * B / parts - b0, r0 = b0 * W, n_lists = nb * W * kc * 4;
    SJD_TRY(cudaMemcpyAsync(c->d_cond + b0 * n_logits, cond + b0 * n_logits, nb * n_logits, H2D, c->in));
    if (uncond) SJD_TRY(cudaMemcpyAsync(c->d_uncond + b0 * n_logits, uncond + b0 * n_logits, nb * n_logits, H2D, c->in));
    if (k == 0) {  // the small arrays, while the first logits are on their way
      const int n = (int)(3 * B + (q ? 3 * rows : 0));
      if (P->win_len) std::memcpy(c->h_small, P->win_len, B * 4);
      if (P->pos_base) std::memcpy(c->h_small + B, P->pos_base, B * 4);
      if (P->iteration) std::memcpy(c->h_small + 2 * B, P->iteration, B * 4);
      if (q) {
        std::memcpy(c->h_small + 3 * B, drafts, rows * 4);
        std::memcpy(c->h_small + 3 * B + rows, q->tok_prob, rows * 4);
        std::memcpy(c->h_small + 3 * B + 2 * rows, q->cnt, rows * 4);
        int32_t* const m_ids = mapped(q->ids, rows * kc * 4);
        float* const m_vals = mapped(q->vals, rows * kc * 4);
        q_copied = !m_ids || !m_vals;
        if (!q_copied) d_q.ids = m_ids, d_q.vals = m_vals;
      }
      fetch_words<<<(n + 255) / 256, 256, 0, c->run>>>(c->m_small, c->d_small, n);
      SJD_TRY(cudaGetLastError());
    }
    if (q_copied) {
      SJD_TRY(cudaMemcpyAsync(d_q.ids + r0 * kc, q->ids + r0 * kc, n_lists, H2D, c->in));
      SJD_TRY(cudaMemcpyAsync(d_q.vals + r0 * kc, q->vals + r0 * kc, n_lists, H2D, c->in));
    }
    sjd_probs part_q, part_out;
    part_q.tok_prob = reinterpret_cast<float*>(d_drafts + rows + r0);
    part_q.ids = d_q.ids + r0 * kc;
    part_q.vals = d_q.vals + r0 * kc;
    part_q.cnt = d_drafts + 2 * rows + r0;
    part_out.tok_prob = reinterpret_cast<float*>(m_tokens + rows + r0);
    part_out.ids = c->d_out.ids + r0 * kc;
    part_out.vals = c->d_out.vals + r0 * kc;
    part_out.cnt = m_tokens + 2 * rows + r0;
    SJD_TRY(cudaEventRecord(c->arrived[k], c->in));
    SJD_TRY(cudaStreamWaitEvent(c->run, c->arrived[k], 0));

    sjd_params D = *P;
    D.B = (int32_t)nb;
    D.seq_base = P->seq_base + (int32_t)b0;
    D.stride_b = (int64_t)c->W * c->V;
    D.stride_w = c->V;
    D.win_len = P->win_len ? d_win + b0 : nullptr;
    D.pos_base = P->pos_base ? d_win + B + b0 : nullptr;
    D.iteration = P->iteration ? d_win + 2 * B + b0 : nullptr;
    D.status = P->status ? c->m_results + B + b0 : nullptr;
    D.out_flags = P->out_flags ? m_tokens + 3 * rows + r0 : nullptr;
    D.workspace = c->d_ws;
    D.workspace_bytes = c->ws_bytes;
    D.stream = c->run;
    D.ev_rows_begin = nullptr;
    D.ev_rows_end = nullptr;
    const int rc = sjd_step(c->d_cond + b0 * n_logits, uncond ? c->d_uncond + b0 * n_logits : nullptr, d_drafts + r0,
                            q ? &part_q : nullptr, &D, seed, c->m_results + b0, m_tokens + r0, &part_out);
    if (rc != SJD_OK) return rc;
    SJD_TRY(cudaEventRecord(c->stepped[k], c->run));
  }
  // (Copies to pageable memory hold the caller up, so none is issued before the last part is on its way.)
  for (size_t k = 0; k < parts; ++k) {
    const size_t b0 = k * B / parts, nb = (k + 1) * B / parts - b0, r0 = b0 * W, n_lists = nb * W * kc * 4;
    SJD_TRY(cudaStreamWaitEvent(c->out, c->stepped[k], 0));
    SJD_TRY(cudaMemcpyAsync(out->ids + r0 * kc, c->d_out.ids + r0 * kc, n_lists, D2H, c->out));
    SJD_TRY(cudaMemcpyAsync(out->vals + r0 * kc, c->d_out.vals + r0 * kc, n_lists, D2H, c->out));
  }
  return SJD_OK;
}

}  // namespace

extern "C" {

int sjd_host_ctx_create(const sjd_params* s, sjd_host_ctx** out_ctx) {
  if (!s || !out_ctx) return SJD_ERR_NULL;
  *out_ctx = nullptr;
  if (s->B < 1 || s->W < 1 || s->W > SJD_W_MAX || s->V < 8 || (s->V % 8) != 0 || s->top_k < 1) return SJD_ERR_SHAPE;
  if (s->logits_dtype != SJD_F32 && s->logits_dtype != SJD_BF16 && s->logits_dtype != SJD_F16) return SJD_ERR_DTYPE;
  sjd_host_ctx* c = static_cast<sjd_host_ctx*>(std::calloc(1, sizeof(sjd_host_ctx)));
  if (!c) return SJD_ERR_CUDA;
  c->B = s->B; c->W = s->W; c->V = s->V; c->dtype = s->logits_dtype; c->top_k = s->top_k;
  c->kcap = s->top_k < s->V ? s->top_k : s->V;
  c->rows = (size_t)s->B * s->W;
  c->row_bytes = (size_t)s->V * (s->logits_dtype == SJD_F32 ? 4 : 2);
  sjd_params shape;
  std::memset(&shape, 0, sizeof(shape));
  shape.B = s->B; shape.W = s->W;
  c->ws_bytes = sjd_workspace_bytes(&shape);
  if (!create(c)) {
    sjd_host_ctx_destroy(c);
    return SJD_ERR_CUDA;
  }
  *out_ctx = c;
  return SJD_OK;
}

void sjd_host_ctx_destroy(sjd_host_ctx* c) {
  if (!c) return;
  drain(c);
  for (cudaStream_t st : {c->in, c->run, c->out})
    if (st) cudaStreamDestroy(st);
  for (int i = 0; i < kMaxParts; ++i) {
    if (c->arrived[i]) cudaEventDestroy(c->arrived[i]);
    if (c->stepped[i]) cudaEventDestroy(c->stepped[i]);
  }
  cudaFreeHost(c->h_small);
  cudaFree(c->arena);
  std::free(c);
}

int sjd_step_host(sjd_host_ctx* c, const void* logits_cond, const void* logits_uncond, const int32_t* drafts,
                  const sjd_probs* q, const sjd_params* P, uint64_t seed, int32_t* out_accept_len,
                  int32_t* out_tokens, sjd_probs* out) {
  if (!c || !P || !logits_cond || !out_accept_len || !out_tokens || !out) return SJD_ERR_NULL;
  if (!out->tok_prob || !out->ids || !out->vals || !out->cnt) return SJD_ERR_NULL;
  if (P->struct_size != (int32_t)sizeof(sjd_params)) return SJD_ERR_STRUCT;
  if (P->B != c->B || P->W != c->W || P->V != c->V || P->logits_dtype != c->dtype || P->top_k != c->top_k)
    return SJD_ERR_SHAPE;
  const bool draft_all = (P->flags & SJD_FLAG_DRAFT_ALL) != 0;
  if (!draft_all && (!drafts || !q || !q->tok_prob || !q->ids || !q->vals || !q->cnt)) return SJD_ERR_NULL;
  const int rc = enqueue(c, static_cast<const char*>(logits_cond), static_cast<const char*>(logits_uncond), drafts,
                         draft_all ? nullptr : q, P, seed, out);
  if (rc != SJD_OK) {
    drain(c);  // nothing of the caller's is touched after the return
    return rc;
  }
  SJD_TRY(cudaStreamSynchronize(c->out));  // behind every part's step, and so behind every copy in
  const size_t rows = c->rows, B = (size_t)c->B;
  const int32_t* o = c->h_results;
  std::memcpy(out_accept_len, o, B * 4);
  if (P->status) std::memcpy(P->status, o + B, B * 4);
  std::memcpy(out_tokens, o + 2 * B, rows * 4);
  std::memcpy(out->tok_prob, o + 2 * B + rows, rows * 4);
  std::memcpy(out->cnt, o + 2 * B + 2 * rows, rows * 4);
  if (P->out_flags) std::memcpy(P->out_flags, o + 2 * B + 3 * rows, rows * 4);
  return SJD_OK;
}

}  // extern "C"
