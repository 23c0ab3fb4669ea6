// Host side of the C ABI declared in include/sjd.h: argument checks and kernel launches.
// Nothing here allocates, frees or synchronises.
#include "../../include/sjd.h"

#include <cuda_runtime.h>

#include <atomic>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "device_once.h"
#include "device_utils.cuh"
#include "row_kernels.cuh"
#include "rows_pipeline.cuh"
#include "rows_sift.cuh"
#include "verify_kernel.cuh"
#include "advance_kernel.cuh"

#include <cmath>

namespace {

thread_local char g_cuda_error[256] = "";
std::atomic<uint64_t> g_launches{0};

int cuda_fail(cudaError_t e, const char* what) {
  std::snprintf(g_cuda_error, sizeof(g_cuda_error), "%s: %s", what, cudaGetErrorString(e));
  return SJD_ERR_CUDA;
}

constexpr int kGenericThreads = 512;

int current_device() {
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess ? dev : -1;
}

// SM count of the current device (cached per device ordinal).
int sm_count() {
  static sjd::DeviceValue cache;
  const int dev = current_device();
  const int n = cache.get(dev, [dev] {
    int v = 0;
    return (dev >= 0 && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) ? v : 0;
  });
  return n > 0 ? n : 148;
}

// The opt-in to more than 48 KB of dynamic shared memory belongs to the (device, kernel) pair: it is set
// once per device for each kernel instantiation (`once` is that instantiation's record).
template <typename Kern>
cudaError_t allow_large_smem(Kern kern, sjd::DeviceOnce& once, int bytes) {
  cudaError_t err = cudaSuccess;
  once.run_once(current_device(), [&] {
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return err == cudaSuccess ? 0 : 1;
  });
  return err;
}

constexpr int kFilterWarps = 8;
constexpr int kFinisherWarps = 8;
constexpr int kMaxStages = 12;
constexpr size_t kSmemLimit = 227u * 1024u;

// Decide whether the single-pass pipelined kernel can take this shape, and with which sampling
// parameters.  The sample is every SS-th 256-element tile of a row; its rank-m value (from the top)
// becomes the candidate threshold.  m is chosen 4.5 standard deviations above K/SS (sample_rank), so that
// a row with exchangeable entries almost never fails to deliver K candidates (such a row is redone by the
// any-shape path, never answered wrongly).  The on-chip lists must hold the expected number of
// candidates with a margin: four standard deviations for the row's total, and for the share of one
// filter thread (a Poisson count) a tail below 1e-6.
// Rank m of the sample element that serves as the first threshold, for an expected a = kcap / S of the row's
// kcap largest inside a sample of one S-th of the row.  The number of those that really fall in the sample
// is at most Poisson(a)-distributed (drawing without replacement only narrows it), so m = a + z sqrt(m),
// i.e. sqrt(m) = z/2 + sqrt(z^2/4 + a), leaves the threshold above the true one (too few candidates, the
// row redone by the any-shape path at many times the cost) with a probability below 4e-6 per row at z = 4.5.
int sample_rank(double a, double z = 4.5) {
  const double root = z / 2 + std::sqrt(z * z / 4 + a);
  return (int)std::ceil(root * root);
}

bool plan_pipeline(const sjd_params* P, int kcap, sjd::PipeCfg* cfg, size_t* smem) {
  const int V = P->V;
  if (kcap > sjd::kKcapMax || V % sjd::kTileElems != 0) return false;
  const int tile_bytes = sjd::kTileElems * (P->logits_dtype == SJD_F32 ? 4 : 2);
  const int tps = sjd::kStageArrayBytes / tile_bytes;
  const int tiles = V / sjd::kTileElems;
  const int vwords = V / 32;
  if (tiles > sjd::kItersMax * kFilterWarps) return false;
  for (int ss : {8, 16, 32}) {
    if (tiles % ss != 0) continue;
    const int sample_tiles = tiles / ss, tail_tiles = tiles - sample_tiles;
    const int sample_stages = (sample_tiles + tps - 1) / tps;
    // tiles of filter warp 0 per row (the most any warp gets), four hit bits each
    int iters0 = 0;
    for (int left = sample_tiles; left > 0; left -= tps) iters0 += ((left < tps ? left : tps) + kFilterWarps - 1) / kFilterWarps;
    for (int left = tail_tiles; left > 0; left -= tps) iters0 += ((left < tps ? left : tps) + kFilterWarps - 1) / kFilterWarps;
    const int mask_words = (4 * iters0 + 31) / 32;
    if (iters0 > sjd::kItersMax || mask_words > sjd::kMaskWordsMax) continue;
    const size_t fixed = sjd::pipe_smem_fixed_bytes(kFilterWarps, vwords, mask_words);
    if (fixed + (size_t)(sample_stages + 3) * 2 * sjd::kStageArrayBytes > kSmemLimit) continue;
    int ns = (int)((kSmemLimit - fixed) / (2 * (size_t)sjd::kStageArrayBytes));
    if (ns > kMaxStages) ns = kMaxStages;
    const int n_sample = V / ss;
    const double a = (double)kcap / ss;
    const int m = sample_rank(a);
    if (m > n_sample / 2 || m > 32 * sample_tiles) continue;  // the rank must exist among the group maxima too
    const double mean = (double)m * ss, sd = (double)ss * std::sqrt((double)m);
    if (mean + 4.0 * sd > (double)sjd::kDenseCap) continue;
    // sample pairs are kept against a floor somewhat below the threshold: about 2m more entries
    const double per_thread = (mean + 2.0 * m) / (32.0 * kFilterWarps);
    if (per_thread + 5.0 * std::sqrt(per_thread) + 1.0 > (double)(sjd::kListCap - 4)) continue;
    cfg->sample_stride = ss;
    cfg->sample_rank = m;
    cfg->n_stages = ns;
    cfg->vwords = vwords;
    cfg->mask_words = mask_words;
    *smem = sjd::pipe_smem_bytes(ns, kFilterWarps, vwords, mask_words);
    return true;
  }
  return false;
}

// Launch as a programmatic dependent of the stream's previous kernel: when that kernel allows it (ours do
// near their end), this grid's blocks are placed and set up early and wait inside the kernel
// (grid_dependency_wait) until the previous kernel has completed.  After a kernel that does not take part,
// an event or a copy this is an ordinary launch.
template <typename... KArgs, typename... Args>
cudaError_t launch_after(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool dependent,
                         int cluster, Args&&... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute attr[2];
  lc.attrs = attr;
  if (dependent) {
    attr[lc.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[lc.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[lc.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[lc.numAttrs].val.clusterDim.x = (unsigned)cluster;
    attr[lc.numAttrs].val.clusterDim.y = 1;
    attr[lc.numAttrs++].val.clusterDim.z = 1;
  }
  return cudaLaunchKernelEx(&lc, kern, std::forward<Args>(args)...);
}

template <int DTYPE>
cudaError_t launch_pipeline(const sjd::RowArgs& ra, const sjd::PipeCfg& cfg, size_t smem, int grid, cudaStream_t st) {
  auto kern = sjd::rows_pipeline_kernel<DTYPE, kFilterWarps, kFinisherWarps>;
  static sjd::DeviceOnce configured;  // per instantiation
  const cudaError_t e = allow_large_smem(kern, configured, (int)kSmemLimit);
  if (e != cudaSuccess) return e;
  return launch_after(kern, dim3((unsigned)grid), dim3((kFilterWarps + kFinisherWarps + 1) * 32), smem, st, true, 1, ra, cfg);
}

// ---- the kernels that sift a row by a sampled threshold (rows_sift.cuh) ----
// Share p of a row's entries to aim the threshold at, such that a row with exchangeable entries still has its
// kcap candidates when the estimate is off by 4.5 standard deviations (probability below 4e-6): p - 4.5 sd(p) =
// kcap / V.  From the n sampled elements themselves sd(p) = sqrt(p (1 - p) / n); from the maxima of N vectors of G
// elements, of which the share q = 1 - (1 - p)^G lies above the threshold, sd(p) = sqrt(q (1 - q) / N) / (dq/dp).
// (Part of every call: a handful of multiplications, no pow.)
double power(double x, int G) {  // G: 1, 2, 4 or 8
  if (G > 1) x *= x;
  if (G > 2) x *= x;
  if (G > 4) x *= x;
  return x;
}
double aimed_share(double want, double N, int G, double* sd) {
  double p = want, last = 0.0;
  for (int it = 0; it < 40 && std::fabs(p - last) > 1e-5 * p; ++it) {
    const double rest = power(1.0 - p, G), q = 1.0 - rest;
    *sd = std::sqrt(q * rest / N) * (1.0 - p) / (G * rest);
    last = p;
    p = want + 4.5 * *sd;
    if (!(p < 0.9)) return 1.0;
  }
  return p;
}

struct SiftPlan {
  sjd::SiftCfg cfg;
  int cluster;  // CTAs per row; 0: the stream kernel
  size_t smem;
};

// Segments of equal length, each with a list that holds its share of the candidates with four standard deviations of
// the threshold's estimate and four of the segment's own count to spare.  Packed screening lets some more pass.  Together the
// lists also hold what a row that crowds needs: the entries a second threshold leaves, and a word per unit.  False where they would
// be too long for 16-bit positions.
bool cut_segments(sjd::SiftCfg* c, int V, int kcap, int segs, int unit, double p, double sd, double more) {
  c->seg_len = (((V + segs - 1) / segs) + 7) & ~7;
  c->units = (c->seg_len + unit - 1) / unit;
  const double mean = c->seg_len * (p + 4.0 * sd) * more;
  int cap = (int)(mean + 4.0 * std::sqrt(mean) + 8.0);
  if (cap > c->seg_len) cap = c->seg_len;
  c->seg_cap = (cap + 7) & ~7;
  const int crowded = (kcap + 128 + segs * c->units + 7) & ~7;
  c->pool = c->seg_cap * segs > crowded ? c->seg_cap * segs : crowded;
  return c->pool <= 65528;
}

bool plan_sift(const sjd_params* P, int kcap, bool has_u, SiftPlan* plan) {
  const int V = P->V, es = P->logits_dtype == SJD_F32 ? 4 : 2, ev = 16 / es, unit = sjd::kUnitBytes / es;
  if (V < 2048 || V > 65536 * sjd::kTeamWarps) return false;
  sjd::SiftCfg& c = plan->cfg;
  std::memset(&c, 0, sizeof(c));
  c.piece_stride = (((V + sjd::kSiftPieces - 1) / sjd::kSiftPieces) + 7) & ~7;
  // the sample: vectors per piece and groups per vector that let the threshold come closest, with 1,024 groups at most
  const double want = (double)kcap / V;
  double p = 2.0, sd = 0.0;
  for (int pv = 4; pv >= 1; pv >>= 1) {
    if (pv > 1 && c.piece_stride * es < 32 * pv) continue;  // pieces take half of the row at most
    int vecs = 0;
    for (int k = 0; k < pv && k * ev < c.piece_stride; ++k) {  // pieces that have a k-th vector
      const int with = (V - k * ev + c.piece_stride - 1) / c.piece_stride;
      vecs += with < sjd::kSiftPieces ? with : sjd::kSiftPieces;
    }
    for (int g = 1; g * pv <= 4; g <<= 1) {
      double sd_g;
      const double p_g = aimed_share(want, (double)vecs * g, ev / g, &sd_g);
      if (p_g >= p) continue;
      p = p_g;
      sd = sd_g;
      c.piece_vecs = pv;
      c.groups = g;
      c.rank = (int)std::ceil(vecs * g * (1.0 - power(1.0 - p, ev / g)));
    }
  }
  if (p > 0.6) return false;
  // packed screening: 16-bit logits, an ordinary temperature, and with guidance an s that the type holds exactly, as 1 - s.
  // With guidance and bf16 logits a tenth more entries pass, which costs more than the screening saves where many are
  // kept (1,024 rows of 65,536, K=8,192: 206 us screened, 166 exact) and lists that no longer leave room for three teams
  // (K=2,000: 77.8, 74.5).
  {
    auto holds = [&](float x) {
      const float m = P->logits_dtype == SJD_F16 ? 2048.0f : 256.0f;  // significand bits
      int e;
      const float f = std::frexp(x, &e) * m;
      return x == 0.0f || (f == std::floor(f) && e > -8 && e < 8);
    };
    c.packed = P->logits_dtype != SJD_F32 && (P->logits_dtype == SJD_F16 || !has_u || p < 0.03) && P->inv_temperature > 1e-3f && P->inv_temperature < 1e3f &&
               (!has_u || (holds(P->cfg_scale) && holds(1.0f - P->cfg_scale)));
  }
  const int sms = sm_count();
  const int64_t rows = (int64_t)P->B * P->W;
  const double more = !c.packed ? 1.0 : P->logits_dtype == SJD_F16 || !has_u ? 1.05 : 1.15;
  // few rows: the fewest CTAs that hold a row, while all rows' clusters find their SMs at once (clusters of four and eight do
  // not fill the GPU: their SMs lie in one GPC).  Sharing a row costs more than it saves: every CTA takes the whole sample,
  // and the candidates, the barriers and the launch of a cluster are slow.  us a step with clusters of 1, 2, 4, 8 CTAs and by the stream
  // kernel: 16 rows of 4,096 fp32, K=64: 11.3, 13.0, 13.9, 20.7, 11.2; of 16,384 bf16, K=500: 12.2, 13.8, 14.9, 22.9, 12.9; of 65,536, K=2,000,
  // bf16 (one does not hold it): -, 16.7, 16.9, 24.7, 20.7 (32 rows: -, 16.8, 17.3, 31.4, 20.8), fp32: -, -, 16.8, 24.0, 23.8 (32 rows: -, -,
  // 17.6, 30.8, 24.6; 36 rows, two rounds of four: -, -, 23.0, 33.0, 24.8).
  for (int n_cta = 1; n_cta <= sjd::kMaxCluster; n_cta <<= 1) {
    if (rows * n_cta > (n_cta <= 2 ? sms : n_cta == 4 ? sms * 7 / 8 : sms / 2)) break;
    if (!cut_segments(&c, V, kcap, sjd::kClusterWarps * n_cta, unit, p, sd, more) || (int64_t)n_cta * c.seg_len > 65536) continue;
    c.scratch = c.seg_cap;
    plan->cluster = n_cta;
    plan->smem = sjd::sift_cluster_smem(c, n_cta, es, has_u);
    if (plan->smem > kSmemLimit) continue;
    // A row that crowds lists the ids of a unit apart from the row's list: room for all of a unit's, as far as the division of an SM's
    // memory that the row needs anyway goes (196 KB shared, or all of it: with less left to the L1 ordinary rows take up to 1 % longer).  The
    // verification's blocks need nothing kept free: beside these, 512 threads of 72 registers and more, they find no registers.  (With 36 KB
    // kept free for them rows of K=8,192 got no more room at all: 32 of 65,536 bf16 that crowd 163 us a step, now 87; 8 of fp32 144 and 106.)
    const int most = c.seg_len < unit ? c.seg_len : unit;
    const size_t division = 195u << 10;  // (a block's own kilobyte comes on top)
    const size_t limit = plan->smem <= division ? division : kSmemLimit;
    if (n_cta > 1 && most > c.scratch) {
      const int room = c.scratch + (int)((limit - plan->smem) / (2 * sjd::kClusterWarps));
      c.scratch = (room < most ? room : most) & ~7;
      plan->smem = sjd::sift_cluster_smem(c, n_cta, es, has_u);
    }
    return true;
  }
  if (!cut_segments(&c, V, kcap, sjd::kTeamWarps, unit, p, sd, more)) return false;
  c.once = rows * V * es * (has_u ? 2 : 1) > (96ll << 20) ? 1 : 0;
  plan->cluster = 0;
  static const int choices[][2] = {{3, 4}, {3, 3}, {3, 2}, {2, 2}, {2, 1}, {1, 2}, {1, 1}};
  for (const auto& ch : choices) {
    c.teams = ch[0];
    c.slots = ch[1];
    plan->smem = sjd::sift_stream_smem(c, has_u);
    if (plan->smem <= kSmemLimit) return true;
  }
  return false;
}

// Which row kernel a step takes, and how.  The tile-dealing one is only there for SJD_FLAG_FORCE_TILES: what plan_sift() refuses,
// plan_pipeline() refuses as well.
struct RowPlan {
  int path;  // SJD_PATH_*
  SiftPlan sift;
  sjd::PipeCfg tiles;
  size_t tiles_smem;
};
void plan_rows(const sjd_params* P, int kcap, bool has_u, RowPlan* plan) {
  plan->path = SJD_PATH_ANY_SHAPE;
  if (P->flags & SJD_FLAG_FORCE_GENERIC) return;
  if (!(P->flags & SJD_FLAG_FORCE_TILES) && plan_sift(P, kcap, has_u, &plan->sift))
    plan->path = plan->sift.cluster > 0 ? SJD_PATH_CLUSTER : SJD_PATH_STREAM;
  else if (plan_pipeline(P, kcap, &plan->tiles, &plan->tiles_smem))
    plan->path = SJD_PATH_TILES;
}

template <int DTYPE, bool HAS_U, bool HAS_T>
cudaError_t launch_sift_as(const sjd::RowArgs& ra, const SiftPlan& plan, cudaStream_t st) {
  const int rows = ra.B * ra.W;
  if (plan.cluster > 0) {
    auto kern = sjd::rows_cluster_kernel<DTYPE, HAS_U, HAS_T>;
    static sjd::DeviceOnce configured;
    const cudaError_t e = allow_large_smem(kern, configured, (int)kSmemLimit);
    if (e != cudaSuccess) return e;
    return launch_after(kern, dim3((unsigned)(rows * plan.cluster)), dim3(sjd::kClusterWarps * 32), plan.smem, st, true, plan.cluster, ra,
                        plan.cfg);
  }
  auto kern = sjd::rows_stream_kernel<DTYPE, HAS_U, HAS_T>;
  static sjd::DeviceOnce configured;
  cudaError_t e = allow_large_smem(kern, configured, (int)kSmemLimit);
  // a CTA takes at most kStreamRows rows per launch: larger problems go in several launches
  const int64_t per_launch = (int64_t)sjd::kStreamRows * sm_count();
  sjd::SiftCfg cfg = plan.cfg;
  for (int64_t r0 = 0; r0 < rows && e == cudaSuccess; r0 += per_launch) {
    cfg.row_begin = (int)r0;
    cfg.row_end = (int)(r0 + per_launch < rows ? r0 + per_launch : rows);
    const int n = cfg.row_end - cfg.row_begin;
    e = launch_after(kern, dim3((unsigned)(n < sm_count() ? n : sm_count())), dim3((unsigned)(cfg.teams * (sjd::kTeamThreads + 32))), plan.smem, st,
                     true, 1, ra, cfg);
    if (e == cudaSuccess && r0 > 0) ++g_launches;
  }
  return e;
}

template <int DTYPE>
cudaError_t launch_sift(const sjd::RowArgs& ra, const SiftPlan& plan, cudaStream_t st) {
  const bool t = ra.inv_T != 1.0f;
  if (ra.uncond != nullptr) return t ? launch_sift_as<DTYPE, true, true>(ra, plan, st) : launch_sift_as<DTYPE, true, false>(ra, plan, st);
  return t ? launch_sift_as<DTYPE, false, true>(ra, plan, st) : launch_sift_as<DTYPE, false, false>(ra, plan, st);
}

template <bool LONG, int LOOK, bool MANY>
cudaError_t launch_verify_as(const sjd::VerifyArgs& va, cudaStream_t st, bool dependent) {
  auto kern = sjd::verify_kernel<LONG, LOOK, MANY>;
  static sjd::DeviceOnce configured;
  const cudaError_t e = allow_large_smem(kern, configured, (int)kSmemLimit);
  if (e != cudaSuccess) return e;
  return launch_after(kern, dim3((unsigned)va.B), dim3(sjd::kVerifyThreads), sjd::verify_smem(va.V, va.kcap, LONG, LOOK), st, dependent, 1, va);
}
template <bool LONG, int LOOK>
cudaError_t launch_verify_of(const sjd::VerifyArgs& va, cudaStream_t st, bool dependent) {
  // Two CTAs to an SM where they would go in rounds otherwise, us a step (V, K, sequences x rows; one to an SM, two): 4,096, 64, 170 x 1: 14.0, 14.0;
  // 300 x 1: 16.8, 15.3; 1,024 x 1: 39.2, 33.1; 1,024, 64, 2,048 x 1: 98.0, 85.6; 65,536, 2,000, 200 x 4: 64.6, 63.2; 4,096, 2,100, 1,024 x 1: 68.0, 52.6;
  // 65,536, 8,192, 200 x 4: 129.4, 124.1.  A few more than one to an SM end about as early the one way as the other: 4,096, 64, 149 x 1: 13.7, 13.8;
  // 524,288, 2,000, 150 x 1: 133.1, 135.0.
  const int sms = sm_count();
  return va.B > sms + sms / 8 ? launch_verify_as<LONG, LOOK, true>(va, st, dependent) : launch_verify_as<LONG, LOOK, false>(va, st, dependent);
}
cudaError_t launch_verify(const sjd::VerifyArgs& va, cudaStream_t st, bool dependent) {
  const bool is_long = va.kcap > sjd::kVerifyShort;
  const int look = sjd::verify_map(va.V, va.kcap, is_long, kSmemLimit);
  if (!is_long) return look == sjd::kMapVals ? launch_verify_of<false, sjd::kMapVals>(va, st, dependent) : launch_verify_of<false, sjd::kNoMap>(va, st, dependent);
  return look == sjd::kMapVals ? launch_verify_of<true, sjd::kMapVals>(va, st, dependent)
         : look == sjd::kMap   ? launch_verify_of<true, sjd::kMap>(va, st, dependent)
                               : launch_verify_of<true, sjd::kNoMap>(va, st, dependent);
}

// Scratch of sjd_step_static(): lives in the library's device image, so every GPU that loads the library
// holds these bytes until the process exits.  Sized for SJD_STATIC_MAX_ROWS rows of RowScratch.
constexpr size_t kStaticScratchBytes = (((size_t)SJD_STATIC_MAX_ROWS * sizeof(sjd::RowScratch) + 256) + 255) & ~(size_t)255;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

using sjd::kMaxDevices;
std::mutex g_static_mutex;
void* g_static_scratch_addr[kMaxDevices] = {};  // device address of g_static_scratch, per device ordinal

// Device address of the static scratch on the CURRENT device.  In host code the symbol's name is only a
// handle; the address a kernel can use comes from cudaGetSymbolAddress(), asked once per device.
int static_scratch_address(void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return SJD_ERR_CAPACITY;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (g_static_scratch_addr[dev] == nullptr) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(static scratch)");
    if (p == nullptr || (reinterpret_cast<uintptr_t>(p) & 255u) != 0) return SJD_ERR_WORKSPACE;
    g_static_scratch_addr[dev] = p;
  }
  *out = g_static_scratch_addr[dev];
  return SJD_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_probs(const sjd_probs* p) {
  if (!p || !p->tok_prob || !p->ids || !p->vals || !p->cnt) return SJD_ERR_NULL;
  return SJD_OK;
}

}  // namespace

extern "C" {

int sjd_version(void) { return SJD_VERSION; }

const char* sjd_status_string(int code) {
  switch (code) {
    case SJD_OK: return "ok";
    case SJD_ERR_NULL: return "a required pointer is NULL";
    case SJD_ERR_SHAPE: return "bad shape: need B >= 0, 1 <= W <= SJD_W_MAX, V >= 8 and V % 8 == 0, top_k >= 1";
    case SJD_ERR_ALIGN: return "logits base address or strides are not 16-byte aligned";
    case SJD_ERR_DTYPE: return "unknown logits dtype";
    case SJD_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case SJD_ERR_STRUCT: return "struct_size does not match this library";
    case SJD_ERR_CUDA: return "CUDA runtime error";
    case SJD_ERR_CAPACITY: return "problem exceeds the fixed capacity of this entry point";
    default: return "unknown status";
  }
}

const char* sjd_last_cuda_error(void) { return g_cuda_error; }

uint64_t sjd_launch_count(void) { return g_launches.load(); }

size_t sjd_workspace_bytes(const sjd_params* p) {
  if (!p || p->B < 0 || p->W < 1) return 0;
  const size_t rows = (size_t)p->B * (size_t)p->W;
  const size_t bytes = rows * sizeof(sjd::RowScratch) + 256;
  return (bytes + 255) & ~(size_t)255;
}

int sjd_step(const void* logits_cond, const void* logits_uncond, const int32_t* drafts, const sjd_probs* draft_probs,
             const sjd_params* P, uint64_t philox_seed, int32_t* out_accept_len, int32_t* out_tokens,
             sjd_probs* out_probs) {
  if (!P) return SJD_ERR_NULL;
  if (P->struct_size != (int32_t)sizeof(sjd_params)) return SJD_ERR_STRUCT;
  if (!logits_cond || !out_accept_len || !out_tokens) return SJD_ERR_NULL;
  if (check_probs(out_probs) != SJD_OK) return SJD_ERR_NULL;
  const bool draft_all = (P->flags & SJD_FLAG_DRAFT_ALL) != 0;
  if (!draft_all && (!drafts || check_probs(draft_probs) != SJD_OK)) return SJD_ERR_NULL;
  if (P->B < 0 || P->W < 1 || P->W > SJD_W_MAX || P->V < 8 || (P->V % 8) != 0 || P->top_k < 1) return SJD_ERR_SHAPE;
  if (P->logits_dtype != SJD_F32 && P->logits_dtype != SJD_BF16 && P->logits_dtype != SJD_F16) return SJD_ERR_DTYPE;
  const int64_t esize = P->logits_dtype == SJD_F32 ? 4 : 2;
  if (!aligned16(logits_cond) || (logits_uncond && !aligned16(logits_uncond)) || (P->stride_b * esize) % 16 != 0 ||
      (P->stride_w * esize) % 16 != 0 || P->stride_w < P->V || P->stride_b < 0)
    return SJD_ERR_ALIGN;
  if (!P->workspace || (reinterpret_cast<uintptr_t>(P->workspace) & 255u) != 0 ||
      P->workspace_bytes < sjd_workspace_bytes(P))
    return SJD_ERR_WORKSPACE;
  if (P->B == 0) return SJD_OK;

  cudaStream_t stream = static_cast<cudaStream_t>(P->stream);
  const int kcap = P->top_k < P->V ? P->top_k : P->V;
  const int rows = P->B * P->W;

  sjd::RowArgs ra;
  ra.cond = logits_cond;
  ra.uncond = logits_uncond;
  ra.stride_b = P->stride_b;
  ra.stride_w = P->stride_w;
  ra.B = P->B; ra.W = P->W; ra.V = P->V; ra.kcap = kcap;
  ra.s = P->cfg_scale;
  ra.inv_T = P->inv_temperature;
  ra.win_len = P->win_len;
  ra.pos_base = P->pos_base;
  ra.iteration = P->iteration;
  ra.iteration0 = P->iteration0;
  ra.seq_base = P->seq_base;
  ra.drafts = draft_all ? nullptr : drafts;
  ra.seed_lo = (uint32_t)(philox_seed & 0xffffffffu);
  ra.seed_hi = (uint32_t)(philox_seed >> 32);
  ra.purpose = draft_all ? sjd::kPurposeInit : sjd::kPurposeRedraft;
  ra.out_ids = out_probs->ids;
  ra.out_vals = out_probs->vals;
  ra.out_cnt = out_probs->cnt;
  ra.scratch = static_cast<sjd::RowScratch*>(P->workspace);

  if (P->ev_rows_begin) {
    const cudaError_t e = cudaEventRecord(static_cast<cudaEvent_t>(P->ev_rows_begin), stream);
    if (e != cudaSuccess) return cuda_fail(e, "event record");
  }
  {
    RowPlan plan;
    cudaError_t e;
    plan_rows(P, kcap, logits_uncond != nullptr, &plan);
    if (plan.path == SJD_PATH_STREAM || plan.path == SJD_PATH_CLUSTER) {
      e = P->logits_dtype == SJD_BF16  ? launch_sift<1>(ra, plan.sift, stream)
          : P->logits_dtype == SJD_F16 ? launch_sift<2>(ra, plan.sift, stream)
                                       : launch_sift<0>(ra, plan.sift, stream);
    } else if (plan.path == SJD_PATH_TILES) {
      const int grid = rows < sm_count() ? rows : sm_count();
      e = P->logits_dtype == SJD_BF16  ? launch_pipeline<1>(ra, plan.tiles, plan.tiles_smem, grid, stream)
          : P->logits_dtype == SJD_F16 ? launch_pipeline<2>(ra, plan.tiles, plan.tiles_smem, grid, stream)
                                       : launch_pipeline<0>(ra, plan.tiles, plan.tiles_smem, grid, stream);
    } else {
      const int grid = rows < 4 * sm_count() ? rows : 4 * sm_count();
      e = P->logits_dtype == SJD_BF16
              ? launch_after(sjd::rows_generic_kernel<1, kGenericThreads>, dim3((unsigned)grid), dim3(kGenericThreads), 0, stream, true, 1, ra)
          : P->logits_dtype == SJD_F16
              ? launch_after(sjd::rows_generic_kernel<2, kGenericThreads>, dim3((unsigned)grid), dim3(kGenericThreads), 0, stream, true, 1, ra)
              : launch_after(sjd::rows_generic_kernel<0, kGenericThreads>, dim3((unsigned)grid), dim3(kGenericThreads), 0, stream, true, 1, ra);
    }
    if (e != cudaSuccess) return cuda_fail(e, "row kernel launch");
    ++g_launches;
  }
  if (P->ev_rows_end) {
    const cudaError_t e = cudaEventRecord(static_cast<cudaEvent_t>(P->ev_rows_end), stream);
    if (e != cudaSuccess) return cuda_fail(e, "event record");
  }

  sjd::VerifyArgs va;
  va.B = P->B; va.W = P->W; va.V = P->V; va.kcap = kcap;
  va.flags = P->flags;
  va.tau = P->reuse_tau;
  va.win_len = P->win_len;
  va.pos_base = P->pos_base;
  va.iteration = P->iteration;
  va.iteration0 = P->iteration0;
  va.seq_base = P->seq_base;
  va.seed_lo = ra.seed_lo;
  va.seed_hi = ra.seed_hi;
  va.drafts = drafts;
  va.q_tok = draft_all ? nullptr : draft_probs->tok_prob;
  va.q_ids = draft_all ? nullptr : draft_probs->ids;
  va.q_vals = draft_all ? nullptr : draft_probs->vals;
  va.q_cnt = draft_all ? nullptr : draft_probs->cnt;
  va.p_ids = out_probs->ids;
  va.p_vals = out_probs->vals;
  va.scratch = ra.scratch;
  va.out_accept_len = out_accept_len;
  va.out_tokens = out_tokens;
  va.out_tok_prob = out_probs->tok_prob;
  va.out_flags = P->out_flags;
  va.status = P->status;
  {
    // directly behind the row kernel the verification grid is launched as its programmatic dependent: its
    // blocks are placed as the row kernel's last blocks retire and wait inside the kernel for its completion.
    // An event recorded in between makes it an ordinary launch.
    const cudaError_t e = launch_verify(va, stream, P->ev_rows_end == nullptr);
    if (e != cudaSuccess) return cuda_fail(e, "verify kernel launch");
    ++g_launches;
  }
  return SJD_OK;
}

int sjd_step_static(const void* logits_cond, const void* logits_uncond, const int32_t* drafts,
                    const sjd_probs* draft_probs, const sjd_params* P, uint64_t philox_seed, int32_t* out_accept_len,
                    int32_t* out_tokens, sjd_probs* out_probs) {
  if (!P) return SJD_ERR_NULL;
  if (P->struct_size != (int32_t)sizeof(sjd_params)) return SJD_ERR_STRUCT;
  if (P->B < 0 || P->W < 1 || P->W > SJD_W_MAX) return SJD_ERR_SHAPE;
  if ((int64_t)P->B * (int64_t)P->W > (int64_t)SJD_STATIC_MAX_ROWS) return SJD_ERR_CAPACITY;
  void* scratch = nullptr;
  const int rc = static_scratch_address(&scratch);
  if (rc != SJD_OK) return rc;
  sjd_params Q = *P;
  Q.workspace = scratch;
  Q.workspace_bytes = kStaticScratchBytes;
  return sjd_step(logits_cond, logits_uncond, drafts, draft_probs, &Q, philox_seed, out_accept_len, out_tokens, out_probs);
}

}  // extern "C"

namespace {
int fill_advance(sjd::AdvanceArgs* a, const sjd_params* P, int32_t n_total, uint64_t seed, int32_t* win_len,
                 int32_t* pos_base, int32_t* iteration, int32_t* next_drafts, sjd_probs* next_probs) {
  if (!P) return SJD_ERR_NULL;
  if (P->struct_size != (int32_t)sizeof(sjd_params)) return SJD_ERR_STRUCT;
  if (!win_len || !pos_base || !iteration || !next_drafts || check_probs(next_probs) != SJD_OK) return SJD_ERR_NULL;
  if (P->B < 0 || P->W < 1 || P->W > SJD_W_MAX || P->V < 1 || P->top_k < 1 || n_total < 0) return SJD_ERR_SHAPE;
  if (P->init_mode < SJD_INIT_RANDOM || P->init_mode > SJD_INIT_SAMPLE_ABOVE) return SJD_ERR_SHAPE;
  if (P->init_mode != SJD_INIT_RANDOM && P->grid_width < 1) return SJD_ERR_SHAPE;
  std::memset(a, 0, sizeof(*a));
  a->B = P->B; a->W = P->W; a->V = P->V;
  a->kcap = P->top_k < P->V ? P->top_k : P->V;
  a->n_total = n_total;
  a->seq_base = P->seq_base;
  a->init_mode = P->init_mode;
  a->grid_width = P->grid_width > 0 ? P->grid_width : 1;
  a->no_refine = (P->flags & SJD_FLAG_NO_REFINE) ? 1 : 0;
  a->seed_lo = (uint32_t)(seed & 0xffffffffu);
  a->seed_hi = (uint32_t)(seed >> 32);
  a->win_len = win_len; a->pos_base = pos_base; a->iteration = iteration;
  a->next_drafts = next_drafts;
  a->next_tok_prob = next_probs->tok_prob; a->next_ids = next_probs->ids; a->next_vals = next_probs->vals;
  a->next_cnt = next_probs->cnt;
  return SJD_OK;
}
}  // namespace

extern "C" {

int sjd_row_path(const sjd_params* P, int guidance) {
  if (!P) return SJD_ERR_NULL;
  if (P->struct_size != (int32_t)sizeof(sjd_params)) return SJD_ERR_STRUCT;
  if (P->B < 0 || P->W < 1 || P->W > SJD_W_MAX || P->V < 8 || (P->V % 8) != 0 || P->top_k < 1) return SJD_ERR_SHAPE;
  if (P->logits_dtype != SJD_F32 && P->logits_dtype != SJD_BF16 && P->logits_dtype != SJD_F16) return SJD_ERR_DTYPE;
  const int64_t esize = P->logits_dtype == SJD_F32 ? 4 : 2;
  if ((P->stride_b * esize) % 16 != 0 || (P->stride_w * esize) % 16 != 0 || P->stride_w < P->V || P->stride_b < 0)
    return SJD_ERR_ALIGN;
  RowPlan plan;
  plan_rows(P, P->top_k < P->V ? P->top_k : P->V, guidance != 0, &plan);
  return plan.path;
}

int sjd_row_kernel(const sjd_params* P) {
  const int path = sjd_row_path(P, 1);
  if (path != SJD_PATH_STREAM && path != SJD_PATH_CLUSTER) return path;  // (the two names' values agree)
  return (P->top_k < P->V ? P->top_k : P->V) <= sjd::kKcapMax ? SJD_ROWS_RANGES : SJD_ROWS_GENERIC;
}

int sjd_window_init(const sjd_params* P, int32_t n_total, uint64_t philox_seed, int32_t* win_len, int32_t* pos_base,
                    int32_t* iteration, int32_t* drafts, sjd_probs* draft_probs) {
  sjd::AdvanceArgs a;
  const int rc = fill_advance(&a, P, n_total, philox_seed, win_len, pos_base, iteration, drafts, draft_probs);
  if (rc != SJD_OK) return rc;
  if (P->B == 0) return SJD_OK;
  const int rows = P->B * P->W;
  sjd::init_window_kernel<<<(rows + 255) / 256, 256, 0, static_cast<cudaStream_t>(P->stream)>>>(a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "window init launch");
  ++g_launches;
  return SJD_OK;
}

int sjd_window_advance(const sjd_params* P, int32_t n_total, uint64_t philox_seed, const int32_t* accept_len,
                       const int32_t* step_tokens, const sjd_probs* step_probs, int32_t* win_len, int32_t* pos_base,
                       int32_t* iteration, int32_t* next_drafts, sjd_probs* next_probs, int32_t* committed,
                       int32_t* n_committed) {
  sjd::AdvanceArgs a;
  const int rc = fill_advance(&a, P, n_total, philox_seed, win_len, pos_base, iteration, next_drafts, next_probs);
  if (rc != SJD_OK) return rc;
  if (!accept_len || !step_tokens || !committed || check_probs(const_cast<sjd_probs*>(step_probs)) != SJD_OK) return SJD_ERR_NULL;
  if (P->B == 0) return SJD_OK;
  a.accept_len = accept_len;
  a.step_tokens = step_tokens;
  a.step_tok_prob = step_probs->tok_prob; a.step_ids = step_probs->ids; a.step_vals = step_probs->vals;
  a.step_cnt = step_probs->cnt;
  a.committed = committed;
  a.n_committed = n_committed;
  cudaStream_t st = static_cast<cudaStream_t>(P->stream);
  cudaError_t e = launch_after(sjd::advance_rows_kernel<256>, dim3((unsigned)(P->B * P->W)), dim3(256), 0, st, true, 1, a);
  if (e != cudaSuccess) return cuda_fail(e, "window advance launch");
  ++g_launches;
  e = launch_after(sjd::advance_state_kernel, dim3((unsigned)((P->B + 127) / 128)), dim3(128), 0, st, true, 1, a);
  if (e != cudaSuccess) return cuda_fail(e, "window state launch");
  ++g_launches;
  return SJD_OK;
}

}  // extern "C"
