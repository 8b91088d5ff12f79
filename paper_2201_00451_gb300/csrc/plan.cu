// C ABI of libfstat: plan lifetime, data upload, template scheduling.
//
// fstat_compute groups templates by sky position (alpha, delta).  Per sky it
// runs the per-sky kernels once (Sec. 3 steps iii-v, which the paper notes
// are reused across spindown templates, Sec. 4.1), then two FFT kernels per
// template (steps vi-vii).  Everything is enqueued on the caller's stream;
// the only host<->device traffic per call is the template list.

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <new>
#include <numeric>
#include <string>
#include <vector>

#include "ascent.cuh"
#include "fstat_internal.cuh"
#include "reduce_peaks.cuh"
#include "sft.cuh"

using namespace fstat;

namespace fstat {
int fft_default_c(int log2_len, int pass_b, int precision);  // fft_shapes.cu
}

namespace {
constexpr double kTabStep = 30.0;  // s, spacing of the timing table
}

struct EventPair {
  cudaEvent_t a, b;
};

struct fstat_plan {
  fstat_plan_desc d;
  Geo geo;
  int device = 0;
  int log2n = 0, log2n1 = 0, log2n2 = 0;
  int64_t n1 = 0, n2 = 0;
  GCol gc{};
  size_t pair_bytes = 16;
  void* xh[kMaxDet] = {};
  int dtype[kMaxDet] = {};
  bool have[kMaxDet] = {};
  double sigma[kMaxDet] = {};
  double sigma_ref = 1.0;        // common rescaling of the series (see sky.cu)
  void* G = nullptr;
  void* Z = nullptr;
  // templates rotate over nstream streams (the caller's + plan-owned side
  // streams), each with its own intermediate, so FFT passes of consecutive
  // templates overlap
  static constexpr int kMaxStreams = 8;
  int nstream = 2;
  // n_z intermediates one behind the other from Z on.  batched (FP32 plans):
  // templates share launches over them (see template_batch), and the first call
  // with enough templates takes more (grow_z, once); captured: a batch holds their
  // addresses, so that the block before that stays (old_z)
  int n_z = 0;
  bool batched = false, grown = false, captured = false;
  std::vector<void*> old_z;
  void* Zs[kMaxStreams] = {};      // Zs[0] aliases Z, Zs[k < n_z] lie in its block
  cudaStream_t side[kMaxStreams] = {};
  cudaEvent_t fork = nullptr;
  cudaEvent_t join[kMaxStreams] = {};
  void* partials = nullptr;      // sums of the resampling's blocks (sky.cu)
  ResTab* rtab = nullptr;        // its constants (geo.rtab)
  TimeTab* tab = nullptr;        // timing table and rotation cubics (geo.tab, geo.rot)
  Cubic* tm_tab = nullptr;       // per-sky Roemer delay cubics (geo.tm_tab)
  SkyNode* nodes = nullptr;      // per-sky timing nodes (geo.nodes)
  NodeF32* nodes32 = nullptr;  // the same nodes in FP32 (geo.nodes32)
  SkyConst* sky = nullptr;
  void* tw = nullptr;            // FP64 plans: twiddle tables for the current split
  TwiddleTables tt{};
  int ca = 0, cb = 0;            // CTA shapes of pass A / pass B (0 = default)
  int cb_pk = -1, vb_pk = -1;    // pass B of the peaks mode when tuned apart (-1: cb, vb)
  int va = 0, vb = 0;            // schedule codes of pass A / pass B (fstat_set_cta)
  int ra = 0, rb = 0;            // persistent CTAs per SM of pass A / pass B (0 = all resident)
  int* d_err = nullptr;   // [0] sticky kernel error, [1] scratch for input checks
  int* h_err = nullptr;   // pinned
  fstat_template* d_tmpl = nullptr;
  int* d_order = nullptr;
  TmplCoef* d_coef = nullptr;
  fstat_template* h_tmpl = nullptr;  // pinned staging
  int* h_order = nullptr;            // pinned staging
  int64_t cap = 0;
  cudaEvent_t staged = nullptr;
  cudaEvent_t done = nullptr;
  bool staged_pending = false;
  bool sky_valid = false;
  double sky_alpha = 0, sky_delta = 0;
  SkyPos pos{};                  // of that sky position
  // refinement: sample tables (built lazily), candidate staging, scratch
  void* gtab = nullptr;
  bool gtab_valid = false;
  fstat_candidate* h_cand = nullptr;  // pinned
  fstat_candidate* d_cand = nullptr;
  int64_t ccap = 0;
  void* gscratch = nullptr;
  size_t gscratch_bytes = 0;
  void* rbuf = nullptr;   // fstat_refine's ascent state and 2F history
  size_t rbuf_bytes = 0;
  cudaEvent_t cand_staged = nullptr;
  bool cand_pending = false;
  // profiling (kernel kinds 0 = pass A, 1 = pass B, 2 = per-sky work,
  // 3 = fused launch of both passes)
  bool prof = false;
  std::vector<EventPair> ev[4];
  std::vector<EventPair> pool;
  int64_t launches[4] = {0, 0, 0, 0};
  // peaks mode: band keys [templates of the call][n_bands]
  unsigned long long* keys = nullptr;
  int64_t keys_cap = 0;
  // device memory this plan has allocated over its life, and the cap on it
  // (0 = none) read at creation from FSTAT_DEVICE_BYTES_CAP
  size_t alloc_bytes = 0, alloc_cap = 0;
  // polls of the first wait for a pass-B tile's bulk copies (< 0: default)
  int wait_limit = -1;
  int64_t n_launches = 0;  // kernel launches enqueued (fstat_launch_count)
  // one persistent launch of both FFT passes per sky group and chunk of
  // templates (FP32 plans, splits with a compiled fused shape)
  bool fused = false;
  int* fq = nullptr;       // launch state of the fused kernel
};

namespace {

int cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return FSTAT_OK;
  if (e == cudaErrorMemoryAllocation) return FSTAT_ERR_OOM;
  return FSTAT_ERR_CUDA;
}

#define CK(call)                                 \
  do {                                           \
    cudaError_t e_ = (call);                     \
    if (e_ != cudaSuccess) return cuda_status(e_); \
  } while (0)

// Plan-owned device allocation, counted against the plan's cap: a cap that
// the request would pass fails like an exhausted device (FSTAT_ERR_OOM).
template <typename Ptr>
cudaError_t palloc(fstat_plan* p, Ptr** ptr, size_t bytes) {
  if (p->alloc_cap && p->alloc_bytes + bytes > p->alloc_cap) return cudaErrorMemoryAllocation;
  void* v = nullptr;
  const cudaError_t e = cudaMalloc(&v, bytes);
  if (e != cudaSuccess) return e;
  *ptr = static_cast<Ptr*>(v);
  p->alloc_bytes += bytes;
  return cudaSuccess;
}

int ilog2_exact(int64_t v) {
  if (v <= 0 || (v & (v - 1))) return -1;
  int k = 0;
  while ((int64_t(1) << k) < v) ++k;
  return k;
}

void free_all(fstat_plan* p) {
  for (int X = 0; X < kMaxDet; ++X) if (p->xh[X]) cudaFree(p->xh[X]);
  if (p->G) cudaFree(p->G);
  if (p->Z) cudaFree(p->Z);
  for (int k = 1; k < fstat_plan::kMaxStreams; ++k) {
    if (p->Zs[k] && k >= p->n_z) cudaFree(p->Zs[k]);
    if (p->side[k]) cudaStreamDestroy(p->side[k]);
    if (p->join[k]) cudaEventDestroy(p->join[k]);
  }
  for (void* z : p->old_z) cudaFree(z);
  if (p->fork) cudaEventDestroy(p->fork);
  if (p->partials) cudaFree(p->partials);
  if (p->rtab) cudaFree(p->rtab);
  if (p->tab) cudaFree(p->tab);
  if (p->tm_tab) cudaFree(p->tm_tab);
  if (p->nodes) cudaFree(p->nodes);
  if (p->nodes32) cudaFree(p->nodes32);
  if (p->sky) cudaFree(p->sky);
  if (p->tw) cudaFree(p->tw);
  if (p->d_err) cudaFree(p->d_err);
  if (p->h_err) cudaFreeHost(p->h_err);
  if (p->d_tmpl) cudaFree(p->d_tmpl);
  if (p->d_order) cudaFree(p->d_order);
  if (p->d_coef) cudaFree(p->d_coef);
  if (p->h_tmpl) cudaFreeHost(p->h_tmpl);
  if (p->h_order) cudaFreeHost(p->h_order);
  if (p->gtab) cudaFree(p->gtab);
  if (p->h_cand) cudaFreeHost(p->h_cand);
  if (p->d_cand) cudaFree(p->d_cand);
  if (p->gscratch) cudaFree(p->gscratch);
  if (p->rbuf) cudaFree(p->rbuf);
  if (p->keys) cudaFree(p->keys);
  if (p->fq) cudaFree(p->fq);
  if (p->cand_staged) cudaEventDestroy(p->cand_staged);
  if (p->staged) cudaEventDestroy(p->staged);
  if (p->done) cudaEventDestroy(p->done);
  for (auto& v : p->ev)
    for (auto& e : v) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
  for (auto& e : p->pool) { cudaEventDestroy(e.a); cudaEventDestroy(e.b); }
}

int ensure_capacity(fstat_plan* p, int64_t n) {
  if (n <= p->cap) return FSTAT_OK;
  if (p->staged_pending) { CK(cudaEventSynchronize(p->staged)); p->staged_pending = false; }
  CK(cudaDeviceSynchronize());
  int64_t c = std::max<int64_t>(n, std::max<int64_t>(1024, 2 * p->cap));
  if (p->d_tmpl) cudaFree(p->d_tmpl);
  if (p->d_order) cudaFree(p->d_order);
  if (p->d_coef) cudaFree(p->d_coef);
  if (p->h_tmpl) cudaFreeHost(p->h_tmpl);
  if (p->h_order) cudaFreeHost(p->h_order);
  p->d_tmpl = nullptr; p->d_order = nullptr; p->d_coef = nullptr; p->h_tmpl = nullptr; p->h_order = nullptr;
  p->cap = 0;
  CK(palloc(p, &p->d_tmpl, c * sizeof(fstat_template)));
  CK(palloc(p, &p->d_order, c * sizeof(int)));
  CK(palloc(p, &p->d_coef, c * sizeof(TmplCoef)));
  CK(cudaMallocHost(&p->h_tmpl, c * sizeof(fstat_template)));
  CK(cudaMallocHost(&p->h_order, c * sizeof(int)));
  p->cap = c;
  return FSTAT_OK;
}

EventPair get_events(fstat_plan* p) {
  if (!p->pool.empty()) { EventPair e = p->pool.back(); p->pool.pop_back(); return e; }
  EventPair e{};
  cudaEventCreate(&e.a);
  cudaEventCreate(&e.b);
  return e;
}

// Intermediates.  A plan starts with one per template stream.  One pass of one
// short transform leaves most of the GPU idle and lasts as long as its chain of
// loads, barriers and stores (~8 us), so FP32 plans give one launch several
// templates where their intermediates stay in L2 (64 MB; 128 MB at 2^21, where the
// block is one of two per stream): at the first call whose launches would take
// more than there are, since a process may hold many plans with small banks.
// Above 2^21 a template fills the GPU, and two streams overlap consecutive passes.
int z_shared(int64_t n_fft) {
  if (n_fft > (int64_t(1) << 21)) return 2;
  return (int)std::min<int64_t>(32, std::max<int64_t>(4, (int64_t(1) << 22) / n_fft));
}
// where templates do not share launches (FP64, segment sums): four template
// streams up to n_fft = 2^19 (2^18 runs 1.6x faster with four than with two),
// two above (2^21: four are 8% slower)
int default_streams(int64_t n_fft) { return n_fft <= (int64_t(1) << 19) ? 4 : 2; }
// streams of launches that share templates (template_batch)
int shared_streams(int64_t n_fft) { return n_fft <= (int64_t(1) << 16) ? 1 : 2; }

cudaError_t alloc_z(fstat_plan* p, int n) {
  const size_t one = (size_t)p->d.n_fft * p->pair_bytes;
  void* z = nullptr;
  const cudaError_t e = palloc(p, &z, n * one);
  if (e != cudaSuccess) return e;
  p->Z = z;
  p->n_z = n;
  for (int k = 0; k < n && k < fstat_plan::kMaxStreams; ++k) p->Zs[k] = (char*)z + k * one;
  return e;
}

// Intermediates for groups of n templates of one sky position.  The plan keeps
// what it has where there is no memory for more (and a plan with a cap on its
// memory never takes more).
int grow_z(fstat_plan* p, int64_t n) {
  const int ns = shared_streams(p->d.n_fft), most = z_shared(p->d.n_fft);
  if (!p->batched || p->grown || p->alloc_cap || std::min<int64_t>(most, ns * ((n + ns - 1) / ns)) <= p->n_z)
    return FSTAT_OK;
  CK(cudaDeviceSynchronize());
  void* own[fstat_plan::kMaxStreams] = {p->Z};  // the block, and what other calls added to it
  for (int k = p->n_z; k < fstat_plan::kMaxStreams && k < most; ++k) own[k] = p->Zs[k];
  p->grown = true;
  if (alloc_z(p, most) != cudaSuccess) {
    cudaGetLastError();
    return FSTAT_OK;
  }
  for (void* z : own)
    if (z && p->captured) p->old_z.push_back(z);
    else if (z) cudaFree(z);
  return FSTAT_OK;
}

// Templates per launch of a group of n, and the streams that the launches rotate
// over.  Up to 2^16 one stream: a launch of many templates fills the GPU, and
// the fork and join would cost more than the overlap of the two passes gives.
// us per call of 16 templates, one per launch over four streams (two from 2^20
// on) -> so: 2^13 117 -> 56, 2^16 115 -> 66, 2^18 134 -> 101, 2^19 164 -> 150,
// 2^20 254 -> 236, 2^21 447 -> 441; of 4 templates: 2^13 62 -> 55, 2^18 82 -> 77.
//
// ring: fewer output rows than templates, 0 = a row each.  Later templates replace
// earlier ones there, so a launch's rows differ and a row stays with one stream:
// rows in order (ord ascending by one), and the streams' launches together
// divide the ring; otherwise one template after the other.
int template_batch(const fstat_plan* p, const int* ord, int64_t n, int64_t ring, int* streams) {
  *streams = (int)std::min<int64_t>(p->nstream, n);
  if (ring) {
    while (ring % *streams) --*streams;
    for (int64_t k = 1; k < n && *streams > 1; ++k)
      if (ord[k] != ord[k - 1] + 1) *streams = 1;
  }
  if (!p->batched) return 1;
  const int ns = shared_streams(p->d.n_fft);
  int T = (int)std::min<int64_t>(p->n_z / ns, (n + ns - 1) / ns);
  if (ring) {
    while (T & (T - 1)) T &= T - 1;
    while (T > 1 && ring % (T * ns)) T >>= 1;
    for (int64_t k = 1; k < n && T > 1; ++k)
      if (ord[k] != ord[k - 1] + 1) T = 1;
    if (T == 1) return 1;
  }
  *streams = (int)std::min<int64_t>(ns, n);
  return T;
}

double spin_spacing(const fstat_plan* p) { return (double)pass_a_spacing(p->log2n, p->log2n2); }

// Per-sky work and the spindown coefficients of sorted templates
// [first, first + count) (none for count 0).
int run_sky(fstat_plan* p, double alpha, double delta, const CoefJob& job, cudaStream_t st) {
  EventPair e{};
  if (p->prof) { e = get_events(p); cudaEventRecord(e.a, st); }
  const void* xh[kMaxDet];
  for (int X = 0; X < kMaxDet; ++X) xh[X] = p->xh[X];
  p->pos = sky_position(p->geo, alpha, delta);
  launch_sky(p->geo, p->d.precision, p->pos, xh, p->dtype, p->G, (int)p->n1, p->gc, p->partials, p->sky, p->d_err, job,
             st);
  CK(cudaGetLastError());
  p->n_launches += 3;  // delay table; nodes; resampling, sums and coefficients
  if (p->prof) { cudaEventRecord(e.b, st); p->ev[2].push_back(e); p->launches[2]++; }
  p->sky_valid = true;
  p->sky_alpha = alpha;
  p->sky_delta = delta;
  return FSTAT_OK;
}

// The same where the plan may hold this sky position's series already.
int run_group(fstat_plan* p, const fstat_template& t, bool force, const CoefJob& job, cudaStream_t st) {
  if (force || !(p->sky_valid && p->sky_alpha == t.alpha && p->sky_delta == t.delta))
    return run_sky(p, t.alpha, t.delta, job, st);
  launch_tmpl_coef(p->pos, p->geo, job, st);
  ++p->n_launches;
  CK(cudaGetLastError());
  return FSTAT_OK;
}

int set_split(fstat_plan* p, int log2n1) {
  int log2n2 = p->log2n - log2n1;
  const int max2 = p->d.precision == FSTAT_FP64 ? kMaxLog2 : kMaxLog2A;
  if (log2n1 < kMinLog2 || log2n1 > kMaxLog2 || log2n2 < kMinLog2 || log2n2 > max2)
    return FSTAT_ERR_UNSUPPORTED;
  p->log2n1 = log2n1;
  p->log2n2 = log2n2;
  p->n1 = int64_t(1) << log2n1;
  p->n2 = int64_t(1) << log2n2;
  p->gc = g_columns(p->d.n_samples, p->n1, p->d.precision == FSTAT_FP64 ? 0 : wpass_a_residues_log2(log2n2));
  p->sky_valid = false;
  if (p->tw) {
    p->tt = twiddle_layout(log2n1, log2n2, p->tw);
    CK(build_twiddles(log2n1, log2n2, p->tw, 0));
    CK(cudaStreamSynchronize(0));
  }
  return FSTAT_OK;
}

// FP32 plans run the warp-local passes whatever the schedule code (the codes
// name schedules of the CTA-wide passes, which they beat throughout; lengths
// and shapes those were never compiled for stay refused).
bool warp_passes(const fstat_plan* p) { return p->d.precision != FSTAT_FP64; }

// cb: rows per tile of the pass B that follows
// T > 1 (FP32 plans): templates coef[0 .. T) in one launch, intermediates from Z on.
cudaError_t launch_a(fstat_plan* p, int ca, int va, int cb, const TmplCoef* coef, cudaStream_t st,
                     void* Z = nullptr, int res = -1, int T = 1) {
  if (!Z) Z = p->Z;
  if (res < 0) res = p->ra;
  ++p->n_launches;
  if (warp_passes(p)) {
    if (!pass_a_shape(p->log2n2, ca, va)) return cudaErrorInvalidConfiguration;
    const int staging = va >= 16 ? 1 : va == 2 ? 2 : 0;  // staged columns asked for; none asked for
    return launch_wpass_a(p->log2n2, staging, p->G, p->gc, p->d.n_samples, (int)p->n1, coef, Z,
                          wpass_z_layout(p->log2n1, cb), T, p->d_err, p->wait_limit, st, res);
  }
  return launch_pass_a_f64(p->log2n2, ca, va, p->G, p->gc, p->d.n_samples, (int)p->n1, p->tt.a, coef, Z, st, res);
}

// T > 1: rows ord[0 .. T) mod out_rows of out (their band keys from
// pk->band_key + ord n_bands, pk->tmpl + ord; see launch_wpass_b*).
cudaError_t launch_b(fstat_plan* p, int cb, int vb, float* out, cudaStream_t st, void* Z = nullptr,
                     const PeakArgs* pk = nullptr, int res = -1, int T = 1, const int* ord = nullptr,
                     int64_t out_rows = 1) {
  if (!Z) Z = p->Z;
  if (res < 0) res = p->rb;
  ++p->n_launches;
  if (warp_passes(p)) {
    if (!pass_b_shape(p->log2n1, cb, vb)) return cudaErrorInvalidConfiguration;
    if (pk)
      return launch_wpass_b_peak(p->log2n1, cb, Z, T, (int)p->n2, p->sky, ord,
                                 pk->band_key ? (int)(p->d.n_fft >> pk->log2_band) : 0, *pk, p->d_err, p->wait_limit, st,
                                 res);
    return launch_wpass_b(p->log2n1, cb, Z, T, (int)p->n2, p->sky, out, ord, out_rows, p->d_err, p->wait_limit, st, res);
  }
  return launch_pass_b_f64(p->log2n1, cb, vb, Z, (int)p->n2, p->tt.b, p->sky, out, st, pk, res);
}

cudaError_t launch_b_acc(fstat_plan* p, float* out, int shift, bool first, cudaStream_t st, void* Z) {
  ++p->n_launches;
  if (warp_passes(p)) {
    if (!pass_b_shape(p->log2n1, p->cb, p->vb)) return cudaErrorInvalidConfiguration;
    return launch_wpass_b_acc(p->log2n1, p->cb, Z, (int)p->n2, p->sky, out, shift, first, p->d_err, p->wait_limit, st, p->rb);
  }
  return launch_pass_b_acc_f64(p->log2n1, p->cb, p->vb, Z, (int)p->n2, p->tt.b, p->sky, out, shift, first, st, p->rb);
}

}  // namespace

extern "C" {

const char* fstat_strerror(int code) {
  switch (code) {
    case FSTAT_OK: return "ok";
    case FSTAT_ERR_INVALID_ARG: return "invalid argument";
    case FSTAT_ERR_OOM: return "out of memory";
    case FSTAT_ERR_CUDA: return "CUDA error";
    case FSTAT_ERR_DEGENERATE: return "degenerate antenna-pattern matrix (D <= 0)";
    case FSTAT_ERR_NONFINITE: return "non-finite value in input series";
    case FSTAT_ERR_NOT_READY: return "not every detector has data";
    case FSTAT_ERR_UNSUPPORTED: return "size or phase range outside the supported limits";
    case FSTAT_ERR_TIMEOUT: return "a kernel's bounded wait for its own copies ran out";
    default: return "unknown error";
  }
}

int fstat_plan_create(const fstat_plan_desc* desc, fstat_plan** out) {
  if (!desc || !out) return FSTAT_ERR_INVALID_ARG;
  *out = nullptr;
  const fstat_plan_desc& d = *desc;
  if (d.n_det < 1 || d.n_det > FSTAT_MAX_DET || d.dterms < 1 || d.dterms > 32 ||
      (d.precision != FSTAT_MIXED && d.precision != FSTAT_FP64) || d.interp < FSTAT_INTERP_TAPERED || d.interp > FSTAT_INTERP_PERIODIC ||
      !(d.dt > 0.0) || !std::isfinite(d.t0) || !std::isfinite(d.f_het) || d.n_samples < 1 ||
      d.n_samples >= (int64_t(1) << 24) || !(d.ephem.c > 0.0) || !std::isfinite(d.ephem.au) ||
      (!std::isnan(d.t_ref) && !std::isfinite(d.t_ref)))
    return FSTAT_ERR_INVALID_ARG;
  int log2n = ilog2_exact(d.n_fft);
  if (log2n < 0) return FSTAT_ERR_INVALID_ARG;
  if (log2n < 2 * kMinLog2 || log2n > 2 * kMaxLog2) return FSTAT_ERR_UNSUPPORTED;
  if (d.n_fft < d.n_samples) return FSTAT_ERR_INVALID_ARG;

  fstat_plan* p = new (std::nothrow) fstat_plan();
  if (!p) return FSTAT_ERR_OOM;
  p->d = d;
  if (const char* cap = std::getenv("FSTAT_DEVICE_BYTES_CAP")) p->alloc_cap = (size_t)std::strtoull(cap, nullptr, 10);
  cudaGetDevice(&p->device);
  p->log2n = log2n;
  set_split(p, log2n / 2);
  p->pair_bytes = d.precision == FSTAT_FP64 ? 32 : 16;

  Geo& g = p->geo;
  std::memset(&g, 0, sizeof(g));
  g.c = d.ephem.c;
  g.au = d.ephem.au;
  g.r_earth = d.ephem.r_earth;
  g.w_rot = d.ephem.omega_rot;
  g.w_orb = d.ephem.omega_orb;
  g.cos_obl = std::cos(d.ephem.obliquity);
  g.sin_obl = std::sin(d.ephem.obliquity);
  g.orb_ph0 = d.ephem.orb_phase0;
  g.sid_ph0 = d.ephem.sidereal_phase0;
  for (int X = 0; X < d.n_det; ++X) {
    g.lat[X] = d.det[X].lat_rad;
    g.lon[X] = d.det[X].lon_rad;
    g.gam[X] = d.det[X].gamma_rad;
    g.s2g[X] = std::sin(2.0 * g.gam[X]);
    g.c2g[X] = std::cos(2.0 * g.gam[X]);
    g.sl[X] = std::sin(g.lat[X]);
    g.cl[X] = std::cos(g.lat[X]);
    g.s2l[X] = std::sin(2.0 * g.lat[X]);
    g.c2l[X] = std::cos(2.0 * g.lat[X]);
    g.rcl[X] = d.ephem.r_earth * std::cos(d.det[X].lat_rad);
    g.rsl[X] = d.ephem.r_earth * std::sin(d.det[X].lat_rad);
    g.clon[X] = std::cos(d.det[X].lon_rad);
    g.slon[X] = std::sin(d.det[X].lon_rad);
    g.w[X] = 0.0;
  }
  g.t0 = d.t0;
  g.dt = d.dt;
  g.f_het = d.f_het;
  g.t_ref = std::isnan(d.t_ref) ? d.t0 + (double)(d.n_samples / 2) * d.dt : d.t_ref;
  g.n = d.n_samples;
  g.tap_c2 = (float)(9.8696044010893586 / 6.0 / ((double)g.n * (double)g.n));
  g.n_det = d.n_det;
  g.dterms = d.dterms;
  g.interp = d.interp;

  const int64_t N = d.n_samples;
  cudaError_t e = cudaSuccess;
  // whole columns of whole residues: up to N1 RL <= 2^12 x 16 pairs of padding
  if (e == cudaSuccess)
    e = palloc(p, &p->G, (size_t)(N + (int64_t(1) << (kMaxLog2 + (d.precision == FSTAT_FP64 ? 0 : 4)))) * p->pair_bytes);
  p->nstream = default_streams(d.n_fft);
  p->batched = d.precision != FSTAT_FP64 && !p->alloc_cap;
  if (e == cudaSuccess) e = alloc_z(p, p->nstream);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->fork, cudaEventDisableTiming);
  for (int k = 1; k < p->nstream && e == cudaSuccess; ++k) {
    e = cudaStreamCreateWithFlags(&p->side[k], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->join[k], cudaEventDisableTiming);
  }
  // timing table over every epoch the timing can reach: the data span
  // widened by the largest delay (|t_m| <= (au + r_earth)/c) plus margin
  {
    // (and the timing nodes, which extend two node steps before the data
    // and up to three node steps past it)
    g.node_log2 = node_step_log2(d.dt, d.ephem.omega_rot, d.precision);
    const double step = (double)(1 << g.node_log2);
    const double reach = (d.ephem.au + d.ephem.r_earth) / d.ephem.c + 100.0;
    const double lo = d.t0 - 2.0 * reach - 2.0 * kTabStep - 2.0 * step * d.dt;
    const double hi = d.t0 + (double)N * d.dt + 2.0 * reach + 2.0 * kTabStep + 4.0 * step * d.dt;
    g.tab_n = time_table_entries(lo, hi, kTabStep);
    g.tab_t0 = lo;
    g.tab_inv_h = 1.0 / kTabStep;
    TimeTab* tab = nullptr;
    if (e == cudaSuccess) e = palloc(p, &tab, (size_t)g.tab_n * (sizeof(TimeTab) + sizeof(RotCell)));
    RotCell* rot = reinterpret_cast<RotCell*>(tab + g.tab_n);
    p->tab = tab;
    g.tab = tab;
    g.rot = rot;
    g.inv_dt = 1.0 / d.dt;
    if (e == cudaSuccess) e = palloc(p, &p->tm_tab, (size_t)g.tab_n * d.n_det * sizeof(Cubic));
    g.tm_tab = p->tm_tab;
    g.n_nodes = sky_nodes(N, g.node_log2);
    if (e == cudaSuccess) e = palloc(p, &p->nodes, (size_t)g.n_nodes * d.n_det * sizeof(SkyNode));
    if (e == cudaSuccess) e = palloc(p, &p->nodes32, (size_t)g.n_nodes * d.n_det * sizeof(NodeF32));
    g.nodes = p->nodes;
    g.nodes32 = p->nodes32;
    if (e == cudaSuccess) e = launch_time_table(g, tab, rot, 0);
    if (e == cudaSuccess) e = palloc(p, &p->rtab, resample_table_bytes());
    if (e == cudaSuccess) e = launch_resample_table(g, p->rtab, 0);
    g.rtab = p->rtab;
  }
  if (e == cudaSuccess) e = palloc(p, &p->partials, sky_partials_bytes(N));
  if (e == cudaSuccess) e = cudaMemset(p->partials, 0, sky_partials_bytes(N));
  if (e == cudaSuccess) e = palloc(p, &p->sky, sizeof(SkyConst));
  if (e == cudaSuccess && d.precision == FSTAT_FP64) e = palloc(p, &p->tw, (size_t)6 * (size_t(1) << kMaxLog2) * 16);
  if (e == cudaSuccess) e = palloc(p, &p->d_err, 2 * sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(p->d_err, 0, 2 * sizeof(int));
  if (e == cudaSuccess) e = cudaMallocHost(&p->h_err, 2 * sizeof(int));
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->staged, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->done, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->cand_staged, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    free_all(p);
    delete p;
    return cuda_status(e);
  }
  // the tables are complete before any call, on whatever stream, reads them
  int rc = set_split(p, p->log2n1);
  if (!rc) rc = cuda_status(cudaStreamSynchronize(0));
  if (rc) {
    free_all(p);
    delete p;
    return rc;
  }
  *out = p;
  return FSTAT_OK;
}

void fstat_plan_destroy(fstat_plan* p) {
  if (!p) return;
  cudaDeviceSynchronize();
  free_all(p);
  delete p;
}

}  // extern "C"

namespace {

// Device storage for detector `det`'s series in `dtype`; marks the series
// (and everything derived from it) stale.
int prepare_series(fstat_plan* p, int det, int dtype, cudaStream_t st) {
  const size_t eb = dtype == FSTAT_C128 ? 16 : 8;
  if (p->xh[det] && p->dtype[det] != dtype) {
    CK(cudaStreamSynchronize(st));
    cudaFree(p->xh[det]);
    p->xh[det] = nullptr;
  }
  if (!p->xh[det]) CK(palloc(p, &p->xh[det], (size_t)p->d.n_samples * eb));
  p->dtype[det] = dtype;
  p->have[det] = false;
  p->sky_valid = false;
  p->gtab_valid = false;
  return FSTAT_OK;
}

// Read the finiteness check that `st` has left in d_err[1] (synchronises) and
// update the noise weights: common rescaling by the smallest sigma among the
// detectors with data.
int finish_series(fstat_plan* p, int det, double sigma, cudaStream_t st) {
  CK(cudaMemcpyAsync(p->h_err + 1, p->d_err + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (p->h_err[1] != 0) return p->h_err[1];
  p->sigma[det] = sigma;
  p->have[det] = true;
  double ref = 0.0;
  for (int X = 0; X < p->d.n_det; ++X)
    if (p->have[X] && (ref == 0.0 || p->sigma[X] < ref)) ref = p->sigma[X];
  p->sigma_ref = ref;
  p->geo.inv_sigma_ref = 1.0 / ref;
  p->geo.isf = (float)p->geo.inv_sigma_ref;
  for (int X = 0; X < p->d.n_det; ++X) {
    p->geo.w[X] = p->have[X] ? ref * ref / (2.0 * p->sigma[X] * p->sigma[X]) : 0.0;
    p->geo.wf[X] = (float)p->geo.w[X];
  }
  return FSTAT_OK;
}

}  // namespace

extern "C" {

int fstat_set_data(fstat_plan* p, int det, const void* xh, int dtype, int64_t n, double sigma,
                   void* stream) {
  if (!p || !xh || det < 0 || det >= p->d.n_det || n != p->d.n_samples || !(sigma > 0.0) ||
      !std::isfinite(sigma) || (dtype != FSTAT_C64 && dtype != FSTAT_C128))
    return FSTAT_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = prepare_series(p, det, dtype, st);
  if (rc) return rc;
  CK(cudaMemcpyAsync(p->xh[det], xh, (size_t)n * (dtype == FSTAT_C128 ? 16 : 8), cudaMemcpyDefault, st));
  CK(cudaMemsetAsync(p->d_err + 1, 0, sizeof(int), st));
  launch_check_finite(p->xh[det], dtype, n, p->d_err + 1, st);
  CK(cudaGetLastError());
  return finish_series(p, det, sigma, st);
}

int fstat_set_sfts(fstat_plan* p, int det, const void* bins, int dtype, int64_t n_sft, int64_t n_bins,
                   int64_t q0, double t_sft, int64_t m_raw, double sigma, void* stream) {
  if (!p || !bins || det < 0 || det >= p->d.n_det || (dtype != FSTAT_C64 && dtype != FSTAT_C128) ||
      n_sft < 1 || n_sft > 65535 || n_bins < 2 || n_bins > INT32_MAX || m_raw < n_bins ||
      !(t_sft > 0.0) || !std::isfinite(t_sft) || !(sigma > 0.0) || !std::isfinite(sigma) ||
      n_sft * n_bins != p->d.n_samples)
    return FSTAT_ERR_INVALID_ARG;
  // the output grid is the plan's: dt = t_sft / n_bins, starting at t0
  if (std::fabs(t_sft / (double)n_bins - p->d.dt) > 1e-12 * p->d.dt) return FSTAT_ERR_INVALID_ARG;
  // the band is the n_bins bins centred on f_het, which lies on the SFT grid
  const double qh = p->d.f_het * t_sft;
  if (std::fabs(qh - std::rint(qh)) > 1e-6 || (int64_t)std::rint(qh) - n_bins / 2 != q0)
    return FSTAT_ERR_INVALID_ARG;
  if (sft_smem_bytes((int)n_bins, p->d.precision) > (size_t)220 * 1024) return FSTAT_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  const int out_dtype = p->d.precision == FSTAT_FP64 ? FSTAT_C128 : FSTAT_C64;
  int rc = prepare_series(p, det, out_dtype, st);
  if (rc) return rc;
  // the per-sky series and the FFT intermediate are stale from here on: they
  // hold the host bins (n complex values of either type fit the n pairs of
  // G) and the roots of unity, once the plan's earlier work has read them
  CK(cudaStreamWaitEvent(st, p->done, 0));
  const void* src = bins;
  cudaPointerAttributes at{};
  int dev = -1;
  const size_t eb = dtype == FSTAT_C128 ? 16 : 8;
  const bool on_device = cudaPointerGetAttributes(&at, bins) == cudaSuccess && at.type == cudaMemoryTypeDevice &&
                         cudaGetDevice(&dev) == cudaSuccess && at.device == dev && ((uintptr_t)bins & (eb - 1)) == 0;
  if (!on_device) {
    cudaGetLastError();
    src = p->G;
    CK(cudaMemcpyAsync(p->G, bins, (size_t)p->d.n_samples * eb, cudaMemcpyDefault, st));
  }
  CK(cudaMemsetAsync(p->d_err + 1, 0, sizeof(int), st));
  CK(launch_sft_to_xh(p->d.precision, dtype, src, n_sft, (int)n_bins, p->d.f_het, p->d.t0, t_sft, m_raw, p->Z,
                      p->xh[det], p->d_err + 1, st));
  return finish_series(p, det, sigma, st);
}

int fstat_export_data(fstat_plan* p, int det, void* out, void* stream) {
  if (!p || !out || det < 0 || det >= p->d.n_det) return FSTAT_ERR_INVALID_ARG;
  if (!p->have[det]) return FSTAT_ERR_NOT_READY;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t eb = p->dtype[det] == FSTAT_C128 ? 16 : 8;
  CK(cudaMemcpyAsync(out, p->xh[det], (size_t)p->d.n_samples * eb, cudaMemcpyDefault, st));
  CK(cudaStreamSynchronize(st));
  return p->dtype[det];
}

}  // extern "C"

namespace {

// Templates per fused launch (bounds the launch state and the int item count).
constexpr int64_t kFusedMaxT = 1 << 15;

bool fused_ok(const fstat_plan* p) {
  return p->d.precision == FSTAT_MIXED && fused_supported(p->log2n1, p->log2n2);
}

// The fused launch's ring of intermediates and its launch state (256 KB, for the
// most templates of one launch: a captured batch keeps its address, so a later
// call with more templates must not replace it).
int fused_buffers(fstat_plan* p) {
  for (int r = 0; r < kRing; ++r)
    if (!p->Zs[r]) CK(palloc(p, &p->Zs[r], (size_t)p->d.n_fft * p->pair_bytes));
  if (!p->fq) CK(palloc(p, &p->fq, queue_ints((int)kFusedMaxT) * sizeof(int)));
  return FSTAT_OK;
}

// Steps (vi)-(vii) for sorted templates [i, j) of one sky group as fused
// launches of up to kFusedMaxT templates each.
int enqueue_fused(fstat_plan* p, int64_t i, int64_t j, const int* d_ord, const TmplCoef* d_coef, float* twoF,
                  int64_t out_rows, cudaStream_t st, bool prof) {
  int rc = fused_buffers(p);
  if (rc) return rc;
  for (int64_t k0 = i; k0 < j; k0 += kFusedMaxT) {
    const int T = (int)std::min<int64_t>(kFusedMaxT, j - k0);
    FusedArgs a{};
    a.G = (const float4*)p->G;
    a.gc = p->gc;
    a.n = (int)p->d.n_samples;
    a.n1 = (int)p->n1;
    a.n2 = (int)p->n2;
    a.coef = d_coef + k0;
    a.ord = d_ord + k0;
    a.out_rows = out_rows;
    a.out = twoF;
    a.sky = p->sky;
    for (int r = 0; r < kRing; ++r) a.Z[r] = (float4*)p->Zs[r];
    a.q = p->fq;
    a.T = T;
    a.err = p->d_err;
    a.wait_set = p->wait_limit >= 0;
    a.wait_limit = p->wait_limit >= 0 ? p->wait_limit : 0;
    // a.na, a.nb, a.total: filled by the launcher from its compiled shape
    CK(cudaMemsetAsync(p->fq, 0, queue_ints(T) * sizeof(int), st));
    EventPair e{};
    if (prof) { e = get_events(p); cudaEventRecord(e.a, st); }
    cudaError_t ce = launch_fused_f32(p->log2n1, p->log2n2, a, st);
    if (ce != cudaSuccess) return cuda_status(ce);
    ++p->n_launches;
    if (prof) { cudaEventRecord(e.b, st); p->ev[3].push_back(e); p->launches[3]++; }
  }
  return FSTAT_OK;
}

// Enqueue steps (iii)-(vii) for n templates on `st`.  h_tmpl/h_ord (host)
// give the sky grouping; d_tmpl/d_ord/d_coef are the device copies the
// kernels read.  force_sky: always redo the per-sky work (graph capture).
// po != nullptr: peaks mode, 2F reduced into po's list and the plan's band
// keys instead of written to twoF.
int enqueue_compute(fstat_plan* p, const fstat_template* h_tmpl, const int* h_ord, int64_t n,
                    const fstat_template* d_tmpl, const int* d_ord, TmplCoef* d_coef, float* twoF,
                    int64_t out_rows, cudaStream_t st, bool force_sky, bool prof,
                    const fstat_peak_out* po = nullptr) {
  int log2_band = 0;
  if (po && po->n_bands > 0) log2_band = ilog2_exact(p->d.n_fft / po->n_bands);
  const int64_t nfft = p->d.n_fft;
  int64_t i = 0;
  while (i < n) {
    const fstat_template& t0 = h_tmpl[h_ord[i]];
    int64_t j = i + 1;
    while (j < n && h_tmpl[h_ord[j]].alpha == t0.alpha && h_tmpl[h_ord[j]].delta == t0.delta) ++j;
    int rc = po || !(p->fused && fused_ok(p)) ? grow_z(p, j - i) : FSTAT_OK;
    if (rc) return rc;
    rc = run_group(p, t0, force_sky, CoefJob{d_tmpl, d_ord, (int)i, (int)(j - i), spin_spacing(p), d_coef}, st);
    if (rc) return rc;
    if (!po && p->fused && fused_ok(p)) {
      rc = enqueue_fused(p, i, j, d_ord, d_coef, twoF, out_rows, st, prof);
      if (rc) return rc;
      i = j;
      continue;
    }
    // Launches of tmax templates rotate over `st` and the plan's side streams, each
    // with its own intermediates, so that consecutive passes overlap; the
    // side streams join back before the next sky position overwrites the
    // per-sky series.
    int ns = 0;
    const int tmax = template_batch(p, h_ord + i, j - i, po || out_rows >= n ? 0 : out_rows, &ns);
    if (ns > 1) {
      CK(cudaEventRecord(p->fork, st));
      for (int q = 1; q < ns; ++q) CK(cudaStreamWaitEvent(p->side[q], p->fork, 0));
    }
    for (int64_t k = i, b = 0; k < j; k += tmax, ++b) {
      const int T = (int)std::min<int64_t>(tmax, j - k), q = (int)(b % ns);
      // one template: its own row; more: the rows of the device's order
      float* out = po ? nullptr : T > 1 ? twoF : twoF + ((int64_t)h_ord[k] % out_rows) * nfft;
      const int* ord = T > 1 ? d_ord + k : nullptr;
      PeakArgs pk{};
      if (po) {
        const int64_t own = T > 1 ? 0 : h_ord[k];
        pk.band_key = po->n_bands > 0 ? p->keys + own * po->n_bands : nullptr;
        pk.peaks = po->peaks;
        pk.count = po->n_peaks;
        pk.cap = po->n_peaks ? po->capacity : 0;
        pk.tmpl = po->tmpl_offset + own;
        pk.thr = po->threshold;
        pk.log2_band = log2_band;
      }
      const TmplCoef* coef = d_coef + k;
      cudaStream_t s = q ? p->side[q] : st;
      void* Zb = tmax > 1 ? (char*)p->Z + (size_t)q * tmax * nfft * p->pair_bytes : p->Zs[q];
      EventPair ea{}, eb{};
      if (prof) { ea = get_events(p); cudaEventRecord(ea.a, s); }
      const bool own = po && p->cb_pk >= 0;  // the peaks mode's own pass-B shape
      const int cb = own ? p->cb_pk : p->cb, vb = own ? p->vb_pk : p->vb;
      cudaError_t e = launch_a(p, p->ca, p->va, cb, coef, s, Zb, -1, T);
      if (e != cudaSuccess) return cuda_status(e);
      if (prof) {
        cudaEventRecord(ea.b, s); p->ev[0].push_back(ea); p->launches[0]++;
        eb = get_events(p); cudaEventRecord(eb.a, s);
      }
      e = launch_b(p, cb, vb, out, s, Zb, po ? &pk : nullptr, -1, T, ord, out_rows);
      if (e != cudaSuccess) return cuda_status(e);
      if (prof) { cudaEventRecord(eb.b, s); p->ev[1].push_back(eb); p->launches[1]++; }
    }
    for (int q = 1; q < ns; ++q) {
      CK(cudaEventRecord(p->join[q], p->side[q]));
      CK(cudaStreamWaitEvent(st, p->join[q], 0));
    }
    i = j;
  }
  return FSTAT_OK;
}

// Largest |tau| = |t_b - t_ref| over the data samples of any sky position:
// the SSB grid starts within the orbital Roemer delay (au / c) of t0.
double spin_tau_max(const fstat_plan* p) {
  const double t_last = p->d.t0 + (double)(p->d.n_samples - 1) * p->d.dt;
  return std::max(std::fabs(p->d.t0 - p->geo.t_ref), std::fabs(t_last - p->geo.t_ref)) +
         p->d.ephem.au / p->d.ephem.c + p->d.dt;
}

int validate_templates(const fstat_plan* p, const fstat_template* tmpl, int64_t n) {
  if (n < 0 || (n > 0 && !tmpl) || n > INT32_MAX) return FSTAT_ERR_INVALID_ARG;
  for (int X = 0; X < p->d.n_det; ++X)
    if (!p->have[X]) return FSTAT_ERR_NOT_READY;
  for (int64_t i = 0; i < n; ++i)
    if (!std::isfinite(tmpl[i].alpha) || !std::isfinite(tmpl[i].delta) ||
        !std::isfinite(tmpl[i].f1dot) || !std::isfinite(tmpl[i].f2dot))
      return FSTAT_ERR_INVALID_ARG;
  // spindown phase excursion within what the phase evaluation reduces exactly
  const double tmax = spin_tau_max(p);
  for (int64_t i = 0; i < n; ++i)
    if (!spin_in_range(tmax, tmpl[i].f1dot, tmpl[i].f2dot)) return FSTAT_ERR_UNSUPPORTED;
  return FSTAT_OK;
}

void sky_order(const fstat_template* tmpl, int64_t n, int* ord) {
  std::iota(ord, ord + n, 0);
  std::stable_sort(ord, ord + n, [&](int a, int b) {
    if (tmpl[a].alpha != tmpl[b].alpha) return tmpl[a].alpha < tmpl[b].alpha;
    return tmpl[a].delta < tmpl[b].delta;
  });
}

}  // namespace

extern "C" {

int fstat_compute(fstat_plan* p, const fstat_template* tmpl, int64_t n_tmpl, float* twoF,
                  void* stream) {
  if (!p || (n_tmpl > 0 && !twoF)) return FSTAT_ERR_INVALID_ARG;
  int rc = validate_templates(p, tmpl, n_tmpl);
  if (rc) return rc;
  if (n_tmpl == 0) return FSTAT_OK;
  cudaStream_t st = (cudaStream_t)stream;
  rc = ensure_capacity(p, n_tmpl);
  if (rc) return rc;
  if (p->staged_pending) { CK(cudaEventSynchronize(p->staged)); p->staged_pending = false; }
  std::memcpy(p->h_tmpl, tmpl, (size_t)n_tmpl * sizeof(fstat_template));
  sky_order(tmpl, n_tmpl, p->h_order);
  CK(cudaMemcpyAsync(p->d_tmpl, p->h_tmpl, (size_t)n_tmpl * sizeof(fstat_template),
                     cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(p->d_order, p->h_order, (size_t)n_tmpl * sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaEventRecord(p->staged, st));
  p->staged_pending = true;
  rc = enqueue_compute(p, tmpl, p->h_order, n_tmpl, p->d_tmpl, p->d_order, p->d_coef, twoF, n_tmpl, st,
                       false, p->prof);
  if (rc) return rc;
  CK(cudaEventRecord(p->done, st));
  return FSTAT_OK;
}

int fstat_semicoherent(fstat_plan* const* seg, int n_seg, const fstat_template* tmpl, int64_t n_tmpl,
                       double t_ref, float* twoF, void* stream) {
  if (!seg || n_seg < 1 || n_seg > FSTAT_MAX_SEGMENTS || !std::isfinite(t_ref) || (n_tmpl > 0 && !twoF))
    return FSTAT_ERR_INVALID_ARG;
  fstat_plan* p0 = seg[0];
  for (int s = 0; s < n_seg; ++s) {
    fstat_plan* p = seg[s];
    if (!p || p->d.precision != p0->d.precision || p->d.dt != p0->d.dt || p->d.f_het != p0->d.f_het ||
        p->d.n_fft != p0->d.n_fft)
      return FSTAT_ERR_INVALID_ARG;
    for (int r = 0; r < s; ++r)
      if (seg[r] == p) return FSTAT_ERR_INVALID_ARG;
    int rc = validate_templates(p, tmpl, n_tmpl);
    if (rc) return rc;
  }
  if (n_tmpl == 0) return FSTAT_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t n = n_tmpl, nfft = p0->d.n_fft;
  const double df = 1.0 / ((double)nfft * p0->d.dt);
  std::vector<int> ord(n);
  sky_order(tmpl, n, ord.data());
  // per segment: templates with f1dot carried to the segment's reference
  // time, and the bin offset of its frequency axis (nearest bin)
  std::vector<int> shift((size_t)n_seg * n);
  int ns = fstat_plan::kMaxStreams;
  for (int s = 0; s < n_seg; ++s) {
    fstat_plan* p = seg[s];
    int rc = ensure_capacity(p, n);
    if (rc) return rc;
    if (p->staged_pending) { CK(cudaEventSynchronize(p->staged)); p->staged_pending = false; }
    const double d_ref = p->geo.t_ref - t_ref;
    for (int64_t i = 0; i < n; ++i) {
      fstat_template t = tmpl[i];
      const double sh = std::rint((t.f1dot * d_ref + 0.5 * t.f2dot * d_ref * d_ref) / df);
      if (!(std::fabs(sh) < 1e9)) return FSTAT_ERR_INVALID_ARG;
      shift[(size_t)s * n + i] = (int)sh;
      t.f1dot += t.f2dot * d_ref;
      if (!spin_in_range(spin_tau_max(p), t.f1dot, t.f2dot)) return FSTAT_ERR_UNSUPPORTED;
      p->h_tmpl[i] = t;
      p->h_order[i] = ord[i];
    }
    CK(cudaMemcpyAsync(p->d_tmpl, p->h_tmpl, (size_t)n * sizeof(fstat_template), cudaMemcpyHostToDevice, st));
    CK(cudaMemcpyAsync(p->d_order, p->h_order, (size_t)n * sizeof(int), cudaMemcpyHostToDevice, st));
    CK(cudaEventRecord(p->staged, st));
    p->staged_pending = true;
    ns = std::min(ns, p->nstream);
  }
  // Templates rotate over the first plan's streams; every segment of one
  // template runs on the same stream, so its additions to the output row
  // are ordered, and all segments use the first plan's intermediate for that
  // stream, one after the other: fewer lines to evict from L2 than with one per
  // segment (four segments at 2^22, whole call: 1566 -> 1555 us).
  int64_t i = 0;
  while (i < n) {
    const fstat_template& t0 = tmpl[ord[i]];
    int64_t j = i + 1;
    while (j < n && tmpl[ord[j]].alpha == t0.alpha && tmpl[ord[j]].delta == t0.delta) ++j;
    for (int s = 0; s < n_seg; ++s) {
      fstat_plan* p = seg[s];
      const int rc = run_group(p, t0, false,
                               CoefJob{p->d_tmpl, p->d_order, (int)i, (int)(j - i), spin_spacing(p), p->d_coef}, st);
      if (rc) return rc;
    }
    const int nq = (int)std::min<int64_t>(ns, j - i);
    if (nq > 1) {
      CK(cudaEventRecord(p0->fork, st));
      for (int q = 1; q < nq; ++q) CK(cudaStreamWaitEvent(p0->side[q], p0->fork, 0));
    }
    for (int64_t k = i; k < j; ++k) {
      const int q = (int)((k - i) % nq);
      cudaStream_t sq = q ? p0->side[q] : st;
      float* out = twoF + (int64_t)ord[k] * nfft;
      for (int s = 0; s < n_seg; ++s) {
        fstat_plan* p = seg[s];
        cudaError_t e = launch_a(p, p->ca, p->va, p->cb, p->d_coef + k, sq, p0->Zs[q]);
        if (e == cudaSuccess) e = launch_b_acc(p, out, shift[(size_t)s * n + ord[k]], s == 0, sq, p0->Zs[q]);
        if (e != cudaSuccess) return cuda_status(e);
      }
    }
    for (int q = 1; q < nq; ++q) {
      CK(cudaEventRecord(p0->join[q], p0->side[q]));
      CK(cudaStreamWaitEvent(st, p0->join[q], 0));
    }
    i = j;
  }
  for (int s = 0; s < n_seg; ++s) CK(cudaEventRecord(seg[s]->done, st));
  return FSTAT_OK;
}

namespace {

// Checks of a peaks request shared by fstat_compute_peaks and
// fstat_reduce_peaks, and the band-key scratch for n_rows rows.
int peaks_request(fstat_plan* p, const fstat_peak_out* po, int64_t n_rows, int64_t* nkeys) {
  if (!po) return FSTAT_ERR_INVALID_ARG;
  const bool list = po->n_peaks != nullptr;
  const bool bands = po->n_bands != 0;
  if (!list && !bands) return FSTAT_ERR_INVALID_ARG;
  if (list && (std::isnan(po->threshold) || po->capacity < 0 || (po->capacity > 0 && !po->peaks)))
    return FSTAT_ERR_INVALID_ARG;
  if (bands && (po->n_bands < 0 || po->n_bands > p->d.n_fft || ilog2_exact(po->n_bands) < 0 ||
                (n_rows > 0 && !po->band_max)))
    return FSTAT_ERR_INVALID_ARG;
  *nkeys = bands ? n_rows * (int64_t)po->n_bands : 0;
  if (*nkeys > p->keys_cap) {
    CK(cudaDeviceSynchronize());
    if (p->keys) cudaFree(p->keys);
    p->keys = nullptr;
    p->keys_cap = 0;
    CK(palloc(p, &p->keys, (size_t)*nkeys * sizeof(unsigned long long)));
    p->keys_cap = *nkeys;
  }
  return FSTAT_OK;
}

}  // namespace

int fstat_reduce_peaks(fstat_plan* p, const float* twoF, int64_t n_rows, const fstat_peak_out* po,
                       void* stream) {
  if (!p || n_rows < 0 || (n_rows > 0 && !twoF) || ((uintptr_t)twoF & 15)) return FSTAT_ERR_INVALID_ARG;
  if (p->d.n_fft % 4096) return FSTAT_ERR_UNSUPPORTED;
  int64_t nkeys = 0;
  int rc = peaks_request(p, po, n_rows, &nkeys);
  if (rc || n_rows == 0) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (nkeys) CK(cudaMemsetAsync(p->keys, 0, (size_t)nkeys * sizeof(unsigned long long), st));
  PeakArgs pk{};
  pk.band_key = nkeys ? p->keys : nullptr;
  pk.peaks = po->peaks;
  pk.count = po->n_peaks;
  pk.cap = po->n_peaks ? po->capacity : 0;
  pk.tmpl = po->tmpl_offset;
  pk.thr = po->threshold;
  pk.log2_band = po->n_bands > 0 ? ilog2_exact(p->d.n_fft / po->n_bands) : 0;
  CK(launch_reduce_peaks(twoF, n_rows, p->d.n_fft, pk, po->n_bands, st));
  if (nkeys) CK(launch_band_decode(p->keys, nkeys, po->band_max, po->band_bin, st));
  CK(cudaEventRecord(p->done, st));
  return FSTAT_OK;
}

int fstat_compute_peaks(fstat_plan* p, const fstat_template* tmpl, int64_t n_tmpl, const fstat_peak_out* po,
                        void* stream) {
  if (!p || !po) return FSTAT_ERR_INVALID_ARG;
  int rc = validate_templates(p, tmpl, n_tmpl);
  if (rc) return rc;
  int64_t nkeys = 0;
  rc = peaks_request(p, po, n_tmpl, &nkeys);
  if (rc) return rc;
  if (n_tmpl == 0) return FSTAT_OK;
  cudaStream_t st = (cudaStream_t)stream;
  rc = ensure_capacity(p, n_tmpl);
  if (rc) return rc;
  if (p->staged_pending) { CK(cudaEventSynchronize(p->staged)); p->staged_pending = false; }
  std::memcpy(p->h_tmpl, tmpl, (size_t)n_tmpl * sizeof(fstat_template));
  sky_order(tmpl, n_tmpl, p->h_order);
  CK(cudaMemcpyAsync(p->d_tmpl, p->h_tmpl, (size_t)n_tmpl * sizeof(fstat_template),
                     cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(p->d_order, p->h_order, (size_t)n_tmpl * sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaEventRecord(p->staged, st));
  p->staged_pending = true;
  if (nkeys) CK(cudaMemsetAsync(p->keys, 0, (size_t)nkeys * sizeof(unsigned long long), st));
  rc = enqueue_compute(p, tmpl, p->h_order, n_tmpl, p->d_tmpl, p->d_order, p->d_coef, nullptr, n_tmpl, st,
                       false, p->prof, po);
  if (rc) return rc;
  if (nkeys) CK(launch_band_decode(p->keys, nkeys, po->band_max, po->band_bin, st));
  CK(cudaEventRecord(p->done, st));
  return FSTAT_OK;
}

static bool candidates_finite(const fstat_candidate* cand, int64_t n) {
  for (int64_t i = 0; i < n; ++i)
    if (!std::isfinite(cand[i].f) || !std::isfinite(cand[i].f1dot) || !std::isfinite(cand[i].alpha) ||
        !std::isfinite(cand[i].delta) || !std::isfinite(cand[i].f2dot))
      return false;
  return true;
}

// the gradient's sample tables (built once per data set) and scratch for n
// candidates
static int grad_prepare(fstat_plan* p, int64_t n, cudaStream_t st) {
  if (!p->gtab) CK(palloc(p, &p->gtab, grad_table_bytes(p->geo)));
  if (!p->gtab_valid) {
    const void* xh[kMaxDet];
    for (int X = 0; X < kMaxDet; ++X) xh[X] = p->xh[X];
    CK(launch_grad_tables(p->geo, xh, p->dtype, p->gtab, st));
    p->gtab_valid = true;
  }
  const size_t need = grad_scratch_bytes((int)n, p->geo);
  if (need > p->gscratch_bytes) {
    CK(cudaDeviceSynchronize());
    if (p->gscratch) cudaFree(p->gscratch);
    p->alloc_bytes -= p->gscratch_bytes;
    p->gscratch = nullptr;
    p->gscratch_bytes = 0;
    CK(palloc(p, &p->gscratch, need));
    p->gscratch_bytes = need;
  }
  return FSTAT_OK;
}

int fstat_grad(fstat_plan* p, const fstat_candidate* cand, int64_t n, float* twoF, float* grad,
               void* stream) {
  if (!p || n < 0 || (n > 0 && (!cand || !twoF || !grad)) || n > INT32_MAX) return FSTAT_ERR_INVALID_ARG;
  for (int X = 0; X < p->d.n_det; ++X)
    if (!p->have[X]) return FSTAT_ERR_NOT_READY;
  if (!candidates_finite(cand, n)) return FSTAT_ERR_INVALID_ARG;
  if (n == 0) return FSTAT_OK;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = grad_prepare(p, n, st);
  if (rc) return rc;
  if (p->cand_pending) { CK(cudaEventSynchronize(p->cand_staged)); p->cand_pending = false; }
  if (n > p->ccap) {
    CK(cudaDeviceSynchronize());
    if (p->h_cand) cudaFreeHost(p->h_cand);
    if (p->d_cand) cudaFree(p->d_cand);
    p->h_cand = nullptr;
    p->d_cand = nullptr;
    p->ccap = 0;
    int64_t c = std::max<int64_t>(n, 256);
    CK(cudaMallocHost(&p->h_cand, c * sizeof(fstat_candidate)));
    CK(palloc(p, &p->d_cand, c * sizeof(fstat_candidate)));
    p->ccap = c;
  }
  std::memcpy(p->h_cand, cand, (size_t)n * sizeof(fstat_candidate));
  CK(cudaMemcpyAsync(p->d_cand, p->h_cand, (size_t)n * sizeof(fstat_candidate), cudaMemcpyHostToDevice, st));
  CK(cudaEventRecord(p->cand_staged, st));
  p->cand_pending = true;
  CK(launch_grad(p->geo, p->gtab, p->d_cand, (int)n, p->gscratch, twoF, grad, st));
  CK(cudaEventRecord(p->done, st));
  return FSTAT_OK;
}

int fstat_refine(fstat_plan* p, const fstat_candidate* cand, int64_t n, const double* scales, int steps,
                 double step0, fstat_candidate* out, float* hist, void* stream) {
  if (!p || n < 0 || n > INT32_MAX || (n > 0 && (!cand || !out)) || !scales || steps < 0 || steps > 100000 ||
      !std::isfinite(step0) || !(step0 > 0.0))
    return FSTAT_ERR_INVALID_ARG;
  for (int j = 0; j < 4; ++j)
    if (!std::isfinite(scales[j]) || !(scales[j] > 0.0)) return FSTAT_ERR_INVALID_ARG;
  for (int X = 0; X < p->d.n_det; ++X)
    if (!p->have[X]) return FSTAT_ERR_NOT_READY;
  if (!candidates_finite(cand, n)) return FSTAT_ERR_INVALID_ARG;
  if (n == 0) return FSTAT_OK;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = grad_prepare(p, n, st);
  if (rc) return rc;
  // one block: theta, trial | cur, val | g, gt | eta | 2F history
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t nc = up((size_t)n * sizeof(fstat_candidate)), nf = up((size_t)n * sizeof(float));
  const size_t n4 = up((size_t)n * 4 * sizeof(float)), nd = up((size_t)n * sizeof(double));
  const size_t nh = up((size_t)(steps + 1) * n * sizeof(float));
  const size_t need = 2 * nc + 2 * nf + 2 * n4 + nd + nh;
  if (need > p->rbuf_bytes) {
    CK(cudaDeviceSynchronize());
    if (p->rbuf) cudaFree(p->rbuf);
    p->alloc_bytes -= p->rbuf_bytes;
    p->rbuf = nullptr;
    p->rbuf_bytes = 0;
    CK(palloc(p, &p->rbuf, need));
    p->rbuf_bytes = need;
  }
  char* b = (char*)p->rbuf;
  AscentState s;
  s.n = (int)n;
  s.theta = (fstat_candidate*)b; b += nc;
  s.trial = (fstat_candidate*)b; b += nc;
  s.cur = (float*)b; b += nf;
  s.val = (float*)b; b += nf;
  s.g = (float*)b; b += n4;
  s.gt = (float*)b; b += n4;
  s.eta = (double*)b; b += nd;
  float* h = (float*)b;
  CK(cudaMemcpyAsync(s.theta, cand, (size_t)n * sizeof(fstat_candidate), cudaMemcpyHostToDevice, st));
  CK(launch_grad(p->geo, p->gtab, s.theta, (int)n, p->gscratch, s.cur, s.g, st));
  CK(launch_ascent_init(s, step0, h, st));
  for (int k = 0; k < steps; ++k) {
    CK(launch_ascent_trial(s, scales, st));
    CK(launch_grad(p->geo, p->gtab, s.trial, (int)n, p->gscratch, s.val, s.gt, st));
    CK(launch_ascent_accept(s, h + (size_t)(k + 1) * n, st));
  }
  // the evaluations, trial and accept per step, init
  p->n_launches += 1 + 2 * (int64_t)steps + (1 + (int64_t)steps) * grad_launches((int)n, p->geo);
  CK(cudaMemcpyAsync(out, s.theta, (size_t)n * sizeof(fstat_candidate), cudaMemcpyDeviceToHost, st));
  if (hist) CK(cudaMemcpyAsync(hist, h, (size_t)(steps + 1) * n * sizeof(float), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  return FSTAT_OK;
}

int fstat_freq_axis(const fstat_plan* p, double* f0, double* df) {
  if (!p || !f0 || !df) return FSTAT_ERR_INVALID_ARG;
  *df = 1.0 / ((double)p->d.n_fft * p->d.dt);
  *f0 = p->d.f_het - (double)(p->d.n_fft / 2) * *df;
  return FSTAT_OK;
}

int fstat_invalidate_sky(fstat_plan* p) {
  if (!p) return FSTAT_ERR_INVALID_ARG;
  p->sky_valid = false;
  return FSTAT_OK;
}

int fstat_sync(fstat_plan* p) {
  if (!p) return FSTAT_ERR_INVALID_ARG;
  CK(cudaEventSynchronize(p->done));
  CK(cudaDeviceSynchronize());
  CK(cudaMemcpy(p->h_err, p->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  int e = p->h_err[0];
  if (e) CK(cudaMemset(p->d_err, 0, sizeof(int)));
  return e;
}

int fstat_export_sky(fstat_plan* p, double alpha, double delta, double* ga, double* gb,
                     double* abcd, void* stream) {
  if (!p || !std::isfinite(alpha) || !std::isfinite(delta)) return FSTAT_ERR_INVALID_ARG;
  for (int X = 0; X < p->d.n_det; ++X)
    if (!p->have[X]) return FSTAT_ERR_NOT_READY;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = run_sky(p, alpha, delta, CoefJob{}, st);
  if (rc) return rc;
  const int64_t N = p->d.n_samples;
  std::vector<unsigned char> buf((size_t)(p->n1 * p->gc.lc) * p->pair_bytes);
  CK(cudaMemcpyAsync(buf.data(), p->G, buf.size(), cudaMemcpyDeviceToHost, st));
  SkyConst sc;
  CK(cudaMemcpyAsync(&sc, p->sky, sizeof(sc), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  for (int64_t j = 0; j < N; ++j) {
    int64_t pos = (j % p->n1) * p->gc.lc + p->gc.at((int)(j / p->n1));
    double v[4];
    if (p->pair_bytes == 16) {
      const float* f = reinterpret_cast<const float*>(buf.data()) + 4 * pos;
      for (int q = 0; q < 4; ++q) v[q] = f[q];
    } else {
      const double* f = reinterpret_cast<const double*>(buf.data()) + 4 * pos;
      for (int q = 0; q < 4; ++q) v[q] = f[q];
    }
    // back to the documented units: G = sum w a z with w = 1/(2 sigma^2)
    const double g = 1.0 / p->sigma_ref;
    if (ga) { ga[2 * j] = v[0] * g; ga[2 * j + 1] = v[1] * g; }
    if (gb) { gb[2 * j] = v[2] * g; gb[2 * j + 1] = v[3] * g; }
  }
  const double g2 = 1.0 / (p->sigma_ref * p->sigma_ref);
  if (abcd) { abcd[0] = sc.A * g2; abcd[1] = sc.B * g2; abcd[2] = sc.C * g2; abcd[3] = sc.D * g2 * g2; }
  return FSTAT_OK;
}

int fstat_set_profiling(fstat_plan* p, int enable) {
  if (!p) return FSTAT_ERR_INVALID_ARG;
  CK(cudaDeviceSynchronize());
  for (auto& v : p->ev) {
    for (auto& e : v) p->pool.push_back(e);
    v.clear();
  }
  for (auto& l : p->launches) l = 0;
  p->prof = enable != 0;
  return FSTAT_OK;
}

int fstat_kernel_stats(fstat_plan* p, int kernel, int64_t* launches, double* total_ms) {
  if (!p || kernel < 0 || kernel > 3 || !launches || !total_ms) return FSTAT_ERR_INVALID_ARG;
  CK(cudaDeviceSynchronize());
  double tot = 0.0;
  for (auto& e : p->ev[kernel]) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, e.a, e.b));
    tot += ms;
  }
  *launches = p->launches[kernel];
  *total_ms = tot;
  return FSTAT_OK;
}

int fstat_get_split(const fstat_plan* p, int64_t* n1, int64_t* n2) {
  if (!p || !n1 || !n2) return FSTAT_ERR_INVALID_ARG;
  *n1 = p->n1;
  *n2 = p->n2;
  return FSTAT_OK;
}

int fstat_set_split(fstat_plan* p, int64_t n1) {
  if (!p) return FSTAT_ERR_INVALID_ARG;
  int l = ilog2_exact(n1);
  if (l < 0) return FSTAT_ERR_INVALID_ARG;
  CK(cudaDeviceSynchronize());
  return set_split(p, l);
}

int fstat_set_streams(fstat_plan* p, int n) {
  if (!p || n < 1 || n > fstat_plan::kMaxStreams) return FSTAT_ERR_INVALID_ARG;
  CK(cudaDeviceSynchronize());
  for (int k = 1; k < n; ++k) {
    if (!p->Zs[k]) CK(palloc(p, &p->Zs[k], (size_t)p->d.n_fft * p->pair_bytes));
    if (!p->side[k]) CK(cudaStreamCreateWithFlags(&p->side[k], cudaStreamNonBlocking));
    if (!p->join[k]) CK(cudaEventCreateWithFlags(&p->join[k], cudaEventDisableTiming));
  }
  p->nstream = n;
  // the default count: as at creation; others: one template per launch, over these streams
  p->batched = n == default_streams(p->d.n_fft) && p->d.precision != FSTAT_FP64 && !p->alloc_cap;
  return FSTAT_OK;
}

int fstat_get_cta(const fstat_plan* p, int* ca, int* va, int* cb, int* vb) {
  if (!p || !ca || !va || !cb || !vb) return FSTAT_ERR_INVALID_ARG;
  // the shape the passes run with: 0 resolved to the length's default
  *ca = p->ca > 0 ? p->ca : fft_default_c(p->log2n2, 0, p->d.precision);
  *va = p->va;
  *cb = p->cb > 0 ? p->cb : fft_default_c(p->log2n1, 1, p->d.precision);
  *vb = p->vb;
  return FSTAT_OK;
}

int fstat_get_peaks_cta(const fstat_plan* p, int* cb, int* vb) {
  if (!p || !cb || !vb) return FSTAT_ERR_INVALID_ARG;
  const int c = p->cb_pk >= 0 ? p->cb_pk : p->cb;
  *cb = c > 0 ? c : fft_default_c(p->log2n1, 1, p->d.precision);
  *vb = p->cb_pk >= 0 ? p->vb_pk : p->vb;
  return FSTAT_OK;
}

int fstat_set_residency(fstat_plan* p, int ra, int rb) {
  if (!p || ra < 0 || rb < 0 || ra > 32 || rb > 32) return FSTAT_ERR_INVALID_ARG;
  p->ra = ra;
  p->rb = rb;
  return FSTAT_OK;
}

int fstat_get_residency(const fstat_plan* p, int* ra, int* rb) {
  if (!p || !ra || !rb) return FSTAT_ERR_INVALID_ARG;
  *ra = p->ra;
  *rb = p->rb;
  return FSTAT_OK;
}

int fstat_set_fused(fstat_plan* p, int enable) {
  if (!p) return FSTAT_ERR_INVALID_ARG;
  if (enable && !fused_ok(p)) return FSTAT_ERR_UNSUPPORTED;
  p->fused = enable != 0;
  return FSTAT_OK;
}

int fstat_get_fused(const fstat_plan* p, int* enabled) {
  if (!p || !enabled) return FSTAT_ERR_INVALID_ARG;
  *enabled = p->fused && fused_ok(p);
  return FSTAT_OK;
}

int fstat_launch_count(const fstat_plan* p, int64_t* launches) {
  if (!p || !launches) return FSTAT_ERR_INVALID_ARG;
  *launches = p->n_launches;
  return FSTAT_OK;
}

int fstat_set_wait_limit(fstat_plan* p, int polls) {
  if (!p) return FSTAT_ERR_INVALID_ARG;
  p->wait_limit = polls < 0 ? -1 : polls;
  return FSTAT_OK;
}

int fstat_set_cta(fstat_plan* p, int ca, int va, int cb, int vb) {
  if (!p || ca < 0 || cb < 0 || ca > 32 || cb > 32 || va < 0 || (va > 3 && va != 10 && va != 16 && va != 18) || vb < 0 ||
      vb > 8)
    return FSTAT_ERR_INVALID_ARG;
  p->ca = ca;
  p->va = va;
  p->cb = cb;
  p->vb = vb;
  p->cb_pk = p->vb_pk = -1;  // the peaks mode follows the set shape
  return FSTAT_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ autotune
namespace {

struct Choice {
  int l1, ca, va, cb, vb, fused;
  int cbp = -1, vbp = -1;  // pass B of the peaks mode
};
std::mutex g_tune_mu;
std::map<std::string, Choice> g_tune_cache;
bool g_tune_file_loaded = false;

std::string tune_key(const fstat_plan* p) {
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, p->device) != cudaSuccess) prop.name[0] = 0;
  char buf[400];
  std::snprintf(buf, sizeof buf, "v6|%s|N=%lld|nfft=%lld|prec=%d|ndet=%d|ns=%d%s", prop.name,
                (long long)p->d.n_samples, (long long)p->d.n_fft, p->d.precision, p->d.n_det, p->nstream, p->batched ? "b" : "");
  for (char* c = buf; *c; ++c)
    if (*c == ' ' || *c == '\t') *c = '_';
  return buf;
}

void load_tune_file() {
  if (g_tune_file_loaded) return;
  g_tune_file_loaded = true;
  const char* f = std::getenv("FSTAT_AUTOTUNE_CACHE");
  if (!f) return;
  std::ifstream in(f);
  std::string key;
  Choice c;
  while (in >> key >> c.l1 >> c.ca >> c.va >> c.cb >> c.vb >> c.fused >> c.cbp >> c.vbp) g_tune_cache[key] = c;
}

void save_tune(const std::string& key, const Choice& c) {
  g_tune_cache[key] = c;
  const char* f = std::getenv("FSTAT_AUTOTUNE_CACHE");
  if (!f) return;
  std::ofstream out(f, std::ios::app);
  out << key << " " << c.l1 << " " << c.ca << " " << c.va << " " << c.cb << " " << c.vb << " " << c.fused << " "
      << c.cbp << " " << c.vbp << "\n";
}

constexpr int kTunePipe = 32;  // templates in the autotuner's pipeline timings

// mean time (ms) of `reps` launches of pass A (which = 0) or pass B (which = 1)
float time_pass(fstat_plan* p, int which, int c, int v, const TmplCoef* coef, float* out, cudaStream_t st,
                cudaEvent_t e0, cudaEvent_t e1) {
  const int reps = 5;
  cudaError_t e = which == 0 ? launch_a(p, c, v, p->cb, coef, st) : launch_b(p, c, v, out, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return -1.f;
  }
  cudaEventRecord(e0, st);
  for (int r = 0; r < reps; ++r) {
    if (which == 0) launch_a(p, c, v, p->cb, coef, st);
    else launch_b(p, c, v, out, st);
  }
  cudaEventRecord(e1, st);
  if (cudaEventSynchronize(e1) != cudaSuccess) return -1.f;
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  return ms / reps;
}

// The pass-B shape of the peaks mode (256 whole-row bands and the threshold
// 70 of Sec. 5.4) at the current split and pass-A shape: without the 2F store
// its best shape can differ from the dense pass's.  FP32 plans time every
// compiled row count in the overlapped template pipeline, since pass A's
// stores follow the row count; FP64 has one shape.  (-1, -1): the dense pass's.
template <typename Run>
void tune_peaks(fstat_plan* p, cudaStream_t st, const Run& pipeline, int* cbp, int* vbp) {
  *cbp = *vbp = -1;
  if (p->d.precision == FSTAT_FP64 || p->d.n_fft < (1 << 14)) return;
  unsigned long long* keys = nullptr;
  fstat_peak* list = nullptr;
  if (cudaMalloc(&keys, (kTunePipe * 256 + 1) * sizeof(unsigned long long)) != cudaSuccess) return;
  if (cudaMalloc(&list, 1024 * sizeof(fstat_peak)) != cudaSuccess) { cudaFree(keys); return; }
  cudaMemsetAsync(keys, 0, (kTunePipe * 256 + 1) * sizeof(unsigned long long), st);
  fstat_peak_out po{};
  po.threshold = 70.f;
  po.n_bands = 256;
  po.peaks = list;
  po.capacity = 1024;
  po.n_peaks = keys + kTunePipe * 256;
  unsigned long long* const own = p->keys;
  p->keys = keys;
  float best = 1e30f;
  int best_cb = -1;
  for (int c : {1, 2, 4, 8}) {
    if (!pass_b_shape(p->log2n1, c, 0) || wpass_b_rows(p->log2n1, c) != c) continue;
    p->cb_pk = c;
    p->vb_pk = 0;
    const float ms = pipeline(&po);
    if (ms > 0.f && ms < best) { best = ms; best_cb = c; }
  }
  p->keys = own;
  p->cb_pk = p->vb_pk = -1;
  if (best_cb > 0) { *cbp = best_cb; *vbp = 0; }
  cudaFree(keys);
  cudaFree(list);
}

}  // namespace

extern "C" int fstat_autotune(fstat_plan* p, void* stream) {
  if (!p) return FSTAT_ERR_INVALID_ARG;
  for (int X = 0; X < p->d.n_det; ++X)
    if (!p->have[X]) return FSTAT_ERR_NOT_READY;
  cudaStream_t st = (cudaStream_t)stream;
  const std::string key = tune_key(p);
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    load_tune_file();
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) {
      CK(cudaDeviceSynchronize());
      int rc = set_split(p, it->second.l1);
      if (rc) return rc;
      p->ca = it->second.ca;
      p->va = it->second.va;
      p->cb = it->second.cb;
      p->vb = it->second.vb;
      p->fused = it->second.fused != 0 && fused_ok(p);
      p->cb_pk = it->second.cbp;
      p->vb_pk = it->second.vbp;
      return FSTAT_OK;
    }
  }
  const int kPipe = kTunePipe;
  int rc = ensure_capacity(p, kPipe);
  if (rc) return rc;
  if (p->staged_pending) { CK(cudaEventSynchronize(p->staged)); p->staged_pending = false; }
  for (int k = 0; k < kPipe; ++k) {
    p->h_tmpl[k] = fstat_template{0.3, -0.5, -1e-10 * (k + 1), 0.0};
    p->h_order[k] = k;
  }
  CK(cudaMemcpyAsync(p->d_tmpl, p->h_tmpl, kPipe * sizeof(fstat_template), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(p->d_order, p->h_order, kPipe * sizeof(int), cudaMemcpyHostToDevice, st));
  CK(cudaStreamSynchronize(st));
  std::vector<fstat_template> ht(p->h_tmpl, p->h_tmpl + kPipe);
  std::vector<int> ho(p->h_order, p->h_order + kPipe);
  float* out = nullptr;
  rc = grow_z(p, kPipe);
  if (rc) return rc;
  int64_t rows = p->batched ? p->n_z : p->nstream;  // a row per template in flight
  if (cudaMalloc(&out, (size_t)rows * p->d.n_fft * sizeof(float)) != cudaSuccess) {
    cudaGetLastError();
    rows = 1;
    CK(cudaMalloc(&out, (size_t)p->d.n_fft * sizeof(float)));
  }
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int max2 = p->d.precision == FSTAT_FP64 ? kMaxLog2 : kMaxLog2A;
  const int lo = std::max(kMinLog2, p->log2n - max2), hi = std::min(kMaxLog2, p->log2n - kMinLog2);
  Choice best{p->log2n1, 0, 0, 0, 0, 0};
  float best_ms = 1e30f;
  p->fused = false;
  const bool saved_prof = p->prof;
  p->prof = false;
  p->cb_pk = p->vb_pk = -1;
  // ms per template of the overlapped pipeline with the plan's current shapes
  // (po: the peaks mode); < 0 where they do not run, rc set on a CUDA error.
  // Best of three trials of two pipelines each: shapes differ by a few
  // percent, about the spread of a single short trial.
  auto pipeline = [&](const fstat_peak_out* po) -> float {
    auto once = [&] {
      return enqueue_compute(p, ht.data(), ho.data(), kPipe, p->d_tmpl, p->d_order, p->d_coef, out, rows, st, false, false,
                             po);
    };
    if (once()) { cudaGetLastError(); return -1.f; }
    float ms = 1e30f;
    for (int trial = 0; trial < 3; ++trial) {
      cudaEventRecord(e0, st);
      for (int rep = 0; rep < 2; ++rep) once();
      cudaEventRecord(e1, st);
      if (cudaEventSynchronize(e1) != cudaSuccess) { rc = FSTAT_ERR_CUDA; return -1.f; }
      float t = 0.f;
      cudaEventElapsedTime(&t, e0, e1);
      ms = std::min(ms, t / (2 * kPipe));
    }
    return ms;
  };
  for (int l1 = lo; l1 <= hi && rc == FSTAT_OK; ++l1) {
    rc = set_split(p, l1);
    if (rc) break;
    rc = run_sky(p, 0.3, -0.5, CoefJob{p->d_tmpl, p->d_order, 0, kPipe, spin_spacing(p), p->d_coef}, st);
    if (rc) break;
    // isolated timings of every distinct shape of each pass: for FP32 plans
    // pass A with columns staged where that costs no occupancy (0) or never
    // (2), pass B with 1 to 8 rows per tile; FP64 has one of each
    std::vector<std::pair<float, std::pair<int, int>>> ta, tb;
    for (int v : {0, 2}) {
      if (v && (!warp_passes(p) || !pass_a_shape(p->log2n2, 0, v))) continue;
      const float ms = time_pass(p, 0, 0, v, p->d_coef, out, st, e0, e1);
      if (ms > 0.f) ta.push_back({ms, {0, v}});
    }
    for (int c : {0, 1, 2, 4, 8}) {
      if (c && (!warp_passes(p) || !pass_b_shape(p->log2n1, c, 0) || wpass_b_rows(p->log2n1, c) != c ||
                c == wpass_b_rows(p->log2n1, 0)))
        continue;
      const float ms = time_pass(p, 1, c, 0, p->d_coef, out, st, e0, e1);
      if (ms > 0.f) tb.push_back({ms, {c, 0}});
    }
    std::sort(ta.begin(), ta.end());
    std::sort(tb.begin(), tb.end());
    // the best few of each, paired in the overlapped template pipeline
    for (size_t ia = 0; ia < ta.size(); ++ia) {
      for (size_t ib = 0; ib < std::min<size_t>(3, tb.size()); ++ib) {
        p->ca = ta[ia].second.first;
        p->va = ta[ia].second.second;
        p->cb = tb[ib].second.first;
        p->vb = tb[ib].second.second;
        const float ms = pipeline(nullptr);
        if (rc) break;
        if (ms > 0.f && ms < best_ms) { best_ms = ms; best = Choice{l1, p->ca, p->va, p->cb, p->vb, 0}; }
      }
      if (rc) break;
    }
    // the persistent launch of both passes over the same templates
    if (rc == FSTAT_OK && fused_ok(p)) {
      p->fused = true;
      const float ms = pipeline(nullptr);
      if (rc == FSTAT_OK && ms > 0.f && ms < best_ms) {
        best_ms = ms;
        best = Choice{l1, p->ca, p->va, p->cb, p->vb, 1};
      }
      p->fused = false;
    }
  }
  if (rc == FSTAT_OK) rc = set_split(p, best.l1);
  if (rc == FSTAT_OK) {
    p->ca = best.ca;
    p->va = best.va;
    p->cb = best.cb;
    p->vb = best.vb;
    p->fused = best.fused != 0 && fused_ok(p);
    rc = run_sky(p, 0.3, -0.5, CoefJob{p->d_tmpl, p->d_order, 0, kPipe, spin_spacing(p), p->d_coef}, st);
    if (rc == FSTAT_OK) tune_peaks(p, st, pipeline, &best.cbp, &best.vbp);
    p->cb_pk = best.cbp;
    p->vb_pk = best.vbp;
  }
  cudaFree(out);
  p->prof = saved_prof;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  std::lock_guard<std::mutex> lock(g_tune_mu);
  save_tune(key, best);
  return FSTAT_OK;
}

// ------------------------------------------------------------------- batch
struct BatchEntry {
  fstat_plan* p = nullptr;
  std::vector<fstat_template> tmpl;
  std::vector<int> ord;
  float* twoF = nullptr;
  int64_t out_rows = 0;
  fstat_template* d_tmpl = nullptr;
  int* d_ord = nullptr;
  TmplCoef* d_coef = nullptr;
  cudaStream_t s = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};

struct fstat_batch {
  std::vector<BatchEntry> e;
  cudaStream_t cap = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  size_t nodes = 0;
};

namespace {

void batch_release(fstat_batch* b) {
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->exec = nullptr;
  b->graph = nullptr;
  for (auto& x : b->e) {
    if (x.d_tmpl) cudaFree(x.d_tmpl);
    if (x.d_ord) cudaFree(x.d_ord);
    if (x.d_coef) cudaFree(x.d_coef);
    if (x.s) cudaStreamDestroy(x.s);
    if (x.fork) cudaEventDestroy(x.fork);
    if (x.join) cudaEventDestroy(x.join);
    x.d_tmpl = nullptr; x.d_ord = nullptr; x.d_coef = nullptr;
    x.s = nullptr; x.fork = nullptr; x.join = nullptr;
  }
  if (b->cap) cudaStreamDestroy(b->cap);
  b->cap = nullptr;
}

}  // namespace

extern "C" {

int fstat_batch_create(fstat_batch** out) {
  if (!out) return FSTAT_ERR_INVALID_ARG;
  *out = new (std::nothrow) fstat_batch();
  return *out ? FSTAT_OK : FSTAT_ERR_OOM;
}

int fstat_batch_add(fstat_batch* b, fstat_plan* p, const fstat_template* tmpl, int64_t n, float* twoF,
                    int64_t out_rows) {
  if (!b || !p || n < 1 || !twoF || out_rows < 0 || b->exec) return FSTAT_ERR_INVALID_ARG;
  for (auto& x : b->e)
    if (x.p == p) return FSTAT_ERR_INVALID_ARG;  // one entry per plan (shared buffers)
  int rc = validate_templates(p, tmpl, n);
  if (rc) return rc;
  BatchEntry x;
  x.p = p;
  x.tmpl.assign(tmpl, tmpl + n);
  x.ord.resize(n);
  sky_order(tmpl, n, x.ord.data());
  x.twoF = twoF;
  x.out_rows = out_rows ? out_rows : n;
  b->e.push_back(std::move(x));
  return FSTAT_OK;
}

int fstat_batch_instantiate(fstat_batch* b, void* stream) {
  if (!b || b->e.empty() || b->exec) return FSTAT_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int rc = FSTAT_OK;
  auto fail = [&](int code) { batch_release(b); return code; };
  for (auto& x : b->e) {
    const int64_t n = (int64_t)x.tmpl.size();
    if (cudaMalloc(&x.d_tmpl, n * sizeof(fstat_template)) != cudaSuccess ||
        cudaMalloc(&x.d_ord, n * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&x.d_coef, n * sizeof(TmplCoef)) != cudaSuccess)
      return fail(FSTAT_ERR_OOM);
    if (cudaMemcpy(x.d_tmpl, x.tmpl.data(), n * sizeof(fstat_template), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(x.d_ord, x.ord.data(), n * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
      return fail(FSTAT_ERR_CUDA);
    if (cudaStreamCreateWithFlags(&x.s, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&x.fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&x.join, cudaEventDisableTiming) != cudaSuccess)
      return fail(FSTAT_ERR_CUDA);
    // one ordinary run first: sets kernel attributes and takes memory outside the capture
    rc = enqueue_compute(x.p, x.tmpl.data(), x.ord.data(), n, x.d_tmpl, x.d_ord, x.d_coef, x.twoF, x.out_rows,
                         st, true, false);
    if (rc) return fail(rc);
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) return fail(FSTAT_ERR_CUDA);
  if (cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking) != cudaSuccess) return fail(FSTAT_ERR_CUDA);
  std::vector<bool> prof;
  for (auto& x : b->e) { prof.push_back(x.p->prof); x.p->prof = false; }  // no timing events in the graph
  if (cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return fail(FSTAT_ERR_CUDA);
  for (auto& x : b->e) {
    cudaEventRecord(x.fork, b->cap);
    cudaStreamWaitEvent(x.s, x.fork, 0);
    rc = enqueue_compute(x.p, x.tmpl.data(), x.ord.data(), (int64_t)x.tmpl.size(), x.d_tmpl, x.d_ord, x.d_coef,
                         x.twoF, x.out_rows, x.s, true, false);
    if (rc) break;
    cudaEventRecord(x.join, x.s);
    cudaStreamWaitEvent(b->cap, x.join, 0);
  }
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamEndCapture(b->cap, &g);
  for (size_t k = 0; k < b->e.size(); ++k) b->e[k].p->prof = prof[k];
  if (rc || e != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return fail(rc ? rc : FSTAT_ERR_CUDA);
  }
  b->graph = g;
  if (cudaGraphInstantiate(&b->exec, b->graph, 0) != cudaSuccess) return fail(FSTAT_ERR_CUDA);
  cudaGraphGetNodes(b->graph, nullptr, &b->nodes);
  for (auto& x : b->e) {
    x.p->sky_valid = false;
    x.p->captured = true;
  }
  return FSTAT_OK;
}

int fstat_batch_launch(fstat_batch* b, void* stream) {
  if (!b || !b->exec) return FSTAT_ERR_INVALID_ARG;
  CK(cudaGraphLaunch(b->exec, (cudaStream_t)stream));
  for (auto& x : b->e) {
    x.p->sky_valid = false;
    CK(cudaEventRecord(x.p->done, (cudaStream_t)stream));
  }
  return FSTAT_OK;
}

int fstat_batch_nodes(const fstat_batch* b, int64_t* nodes) {
  if (!b || !nodes) return FSTAT_ERR_INVALID_ARG;
  *nodes = (int64_t)b->nodes;
  return FSTAT_OK;
}

void fstat_batch_destroy(fstat_batch* b) {
  if (!b) return;
  cudaDeviceSynchronize();
  batch_release(b);
  delete b;
}

}  // extern "C"
