// Internal types and device helpers shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/fstat.h"

namespace fstat {

// ---------------------------------------------------------------- constants
constexpr int kMaxDet = FSTAT_MAX_DET;
constexpr int kSkyBlock = 256;      // threads per block of the per-SSB-sample kernel
constexpr int kMinLog2 = 5;         // FFT pass lengths 32 .. 4096 (pass B rows)
constexpr int kMaxLog2 = 12;
constexpr int kMaxLog2A = 13;       // pass A columns up to 8192 (FP32 plans)

// Per-sky results in device memory (k_resample's sums): the antenna-pattern
// integrals and the weights of eq. (Fstat), 2A/D, 2B/D, 4C/D
// (2F = kB|Fa|^2 + kA|Fb|^2 - kC Re FaFb*).
struct SkyConst {
  double A, B, C, D;
  double kA, kB, kC;
  float kAf, kBf, kCf;
};

// What the per-sky kernels take from the sky position alone, formed on the
// host (kernel argument, by value).
struct SkyPos {
  double t_b0;                // start of the SSB grid
  double j_ref;               // (t_ref - t_b0) / dt
  // t_m,X = ox cos(orbit) + oy sin(orbit) + rx cos(rotation) + ry sin(rotation) + rz
  double ox, oy;
  double rx[kMaxDet], ry[kMaxDet], rz[kMaxDet];
  // antenna patterns a = c0 + c1 cH^2 + c2 sH cH + c3 cH + c4 sH, likewise b, with
  // cH, sH = cos, sin(H), H = (alpha - lon) - rotation; cos, sin(alpha - lon)
  double cx[kMaxDet], sx[kMaxDet];
  double ca[kMaxDet][5];
  double cb[kMaxDet][5];
};

struct TmplCoef;

// Templates whose spindown coefficients a per-sky group needs: entries
// [first, first + count) of order, into out at the same places.
struct CoefJob {
  const fstat_template* tmpl;
  const int* order;
  int first, count;
  double spacing;  // TmplCoef's D
  TmplCoef* out;
};

// Per-template spindown phase polynomial in x = j - J (J = rint(j_ref)):
// phi(x) = p0 + p1 x + p2 x^2 + p3 x^3 cycles, and its differences over pass
// A's sample spacing D (the samples of one butterfly),
//   d1(x) = phi(x + D) - phi(x)     = q0 + q1 x + q2 x^2
//   d2(x) = d1(x + D) - d1(x)       = r0 + r1 x
//   d3    = d2(x + D) - d2(x)
// FP32 path: double-float coefficients (hi + lo carries ~48 bits) and d3 in
// units of 2^-32 cycles; FP64 path: phi's coefficients in doubles.
struct TmplCoef {
  float phi[4][2], d1[3][2], d2[2][2];  // [power][hi, lo]
  int d3, J;
  double p[4];
};

// Spindown phase polynomial of one template (eqs. Fa, Fb: Phi_s =
// 2 pi (f1dot tau^2/2 + f2dot tau^3/6)) for samples j with tau_j = (j - jr) dt,
// expanded in x = j - J.  J is the integer nearest jr clamped into the data
// [0, n - 1], so |x| <= 2^24 stays exact in FP32 wherever the reference time
// lies; p0, a phase common to every sample that cancels in 2F, is reduced mod
// 1, as are the other coefficients (x is an integer) where they reach a cycle.
__device__ inline TmplCoef spin_coef(double jr, int64_t n, double dt, double f1dot, double f2dot, double D) {
  double J = rint(jr);
  if (!(J >= 0.0)) J = 0.0;
  if (J > (double)(n - 1)) J = (double)(n - 1);
  const double e = jr - J;  // tau_j = (x - e) dt
  const double c2 = f1dot * dt * dt / 2.0;
  const double c3 = f2dot * dt * dt * dt / 6.0;
  TmplCoef c;
  c.p[3] = c3;
  c.p[2] = c2 - 3.0 * c3 * e;
  c.p[1] = -2.0 * c2 * e + 3.0 * c3 * e * e;
  c.p[0] = c2 * e * e - c3 * e * e * e;
  double d1[3] = {D * (c.p[1] + D * (c.p[2] + D * c.p[3])), D * (2.0 * c.p[2] + D * 3.0 * c.p[3]), D * 3.0 * c.p[3]};
  double d2[2] = {D * D * (2.0 * c.p[2] + D * 6.0 * c.p[3]), D * D * 6.0 * c.p[3]};
  auto split = [](double* v, float (*f)[2], int m) {
    for (int q = 0; q < m; ++q) {
      if (q == 0 || fabs(v[q]) >= 1.0) v[q] -= rint(v[q]);
      f[q][0] = (float)v[q];
      f[q][1] = (float)(v[q] - (double)f[q][0]);
    }
  };
  double d3 = D * D * D * 6.0 * c.p[3];
  d3 -= rint(d3);
  split(c.p, c.phi, 4);
  split(d1, c.d1, 3);
  split(d2, c.d2, 2);
  c.d3 = (int)(unsigned)(long long)rint(d3 * 4294967296.0);
  c.J = (int)J;
  return c;
}

// Largest spindown phase excursion over the data (cycles) that the FP32
// path's double-float evaluation reduces mod 1 exactly (its reduced phase
// then stays within [-0.57, 0.57] cycles).  tmax bounds |tau| over the data
// samples; twice max |Phi_s| / 2 pi bounds the excursion.
constexpr double kMaxSpinCycles = 1048576.0;  // 2^20
inline bool spin_in_range(double tmax, double f1dot, double f2dot) {
  const double b = fabs(f1dot) * tmax * tmax + fabs(f2dot) * tmax * tmax * tmax / 3.0;
  return b < kMaxSpinCycles;
}

// Streaming multiprocessors of the current device (host; cached per device).
int device_sm_count();

// One entry of the sky-independent timing table (sky.cu): cos, sin of the
// orbital phase and of the sidereal rotation angle.
struct alignas(32) TimeTab {
  double co, so, cq, sq;
};
// Between two entries: c0 + c1 f + c2 f^2 + c3 f^3 at the fraction f of the
// way, the cubic through the four nearest entries.
struct alignas(32) Cubic {
  double c0, c1, c2, c3;
};
struct RotCell {
  Cubic c, s;  // cos, sin of the rotation angle
};

// Per-sky timing at one node (see Geo::nodes).
struct alignas(32) SkyNode {
  double tm_det;  // t_m,X(t0 + j dt)
  double v;       // (T - t0) / dt - j, T + t_m,X(T) = t_b^j
  double a, b;    // antenna patterns at T
};
// The same nodes for the FP32 (mixed-precision) path: v = vi + vf with
// vi = rint(v) exact and |vf| <= 1/2 in FP32, dv = v(next node) - v (small:
// the delay's change over a node step), a, b in FP32; and the step-iii phase
// f_h t_m at the detector-time node, formed in FP64: ph its fraction and rate its
// change per sample up to the next node in units of 2^-32 cycles (both modulo a
// cycle, so that a sample's multiple of rate is exact), curv the change from that
// step's phase difference to the next step's, in half cycles (~1e-4).
// vi_inner = 2 vi + inner; inner: the step that starts at this node is a whole
// one and every sample of it certainly valid (k0 inside the data), from the
// delays of the cubic's four nodes with room for its overshoot.
struct alignas(32) NodeF32 {
  float a, b, vf, dv;
  int vi_inner;
  unsigned ph, rate;
  float curv;
};
// Samples between timing nodes, 4 .. 64 (a resampling block holds whole steps):
// the most for which a step lasts at most 32 s of the Earth's rotation, over
// which cubics are exact to ~1e-14 s and ~5e-12 in a, b (four samples, the fewest,
// pass 32 s above dt = 8 s: the errors grow as the fourth power of the step, to
// 2e-9 in a, b at 30 s).  FP64 plans, whose series keeps a, b in FP64: at most 16.
inline int node_step_log2(double dt, double w_rot, int precision) {
  const int most = precision == FSTAT_FP64 ? 4 : 6;
  int l = 2;
  while (l < most && (2 << l) * dt <= 32.0 && fabs(w_rot) * (2 << l) * dt <= 2.4e-3) ++l;
  return l;
}
// A step's six nearest nodes begin two steps before it and end three after.
constexpr int kNodeLead = 2;
inline int sky_nodes(int64_t n, int step_log2) { return (int)((n + (1 << step_log2) - 1) >> step_log2) + 5; }

// Geometry constants for one plan (kernel argument, by value).
struct Geo {
  double c, au, r_earth, w_rot, w_orb, cos_obl, sin_obl, orb_ph0, sid_ph0;
  double lat[kMaxDet], lon[kMaxDet], gam[kMaxDet];
  double s2g[kMaxDet], c2g[kMaxDet], sl[kMaxDet], cl[kMaxDet], s2l[kMaxDet], c2l[kMaxDet];  // of 2 gam, lat, 2 lat
  double rcl[kMaxDet], rsl[kMaxDet];   // r_earth cos(lat), r_earth sin(lat)
  double w[kMaxDet];                   // noise weights of the rescaled series, sigma_ref^2 / (2 sigma_X^2)
  double inv_sigma_ref;                // z is formed divided by sigma_ref (smallest sigma_X)
  float isf, wf[kMaxDet];              // inv_sigma_ref and w in FP32
  float tap_c2;                        // (pi / N)^2 / 6, series form of the tap weights (sky.cu)
  double t0, dt, f_het, t_ref;
  int64_t n;                           // samples per detector
  int n_det, dterms;
  int interp;                          // FSTAT_INTERP_*
  double clon[kMaxDet], slon[kMaxDet]; // cos, sin of the longitudes
  // Sky-independent timing table (sky.cu): cos, sin of the orbital phase and
  // of the sidereal rotation angle at t = tab_t0 + i / tab_inv_h.
  const TimeTab* tab;
  const RotCell* rot;                  // cubics of the rotation's cos, sin, same grid
  double tab_t0, tab_inv_h, inv_dt;
  int tab_n;
  // Roemer delay t_m of the current sky position for each detector as cubics on
  // the same grid, [X * tab_n + i] (rewritten by every per-sky run)
  Cubic* tm_tab;
  // Per-sky timing nodes every 2^node_log2 samples (sky.cu), [X * n_nodes + m]
  // for sample j = (m - kNodeLead) 2^node_log2: t_m at the detector time, and at the
  // SSB epoch the delay correction v = u - j and the antenna patterns a, b
  SkyNode* nodes;
  NodeF32* nodes32;                    // the same nodes in FP32 (mixed path)
  int n_nodes, node_log2;
  const struct ResTab* rtab;           // the resampling's constants (sky.cu)
};

// ---------------------------------------------------- pair of complex values
// The two transforms Fa and Fb of one template share every index and
// twiddle, so kernels carry them together: (a.re, a.im, b.re, b.im).
template <typename T> struct Pair { T ar, ai, br, bi; };

template <typename T> __device__ __forceinline__ Pair<T> padd(const Pair<T>& x, const Pair<T>& y) {
  return {x.ar + y.ar, x.ai + y.ai, x.br + y.br, x.bi + y.bi};
}
template <typename T> __device__ __forceinline__ Pair<T> psub(const Pair<T>& x, const Pair<T>& y) {
  return {x.ar - y.ar, x.ai - y.ai, x.br - y.br, x.bi - y.bi};
}
// (fused explicitly, here and in the transforms, so that every kernel that
// shares this arithmetic gives the same bits)
__device__ __forceinline__ float fmadd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmadd(double a, double b, double c) { return fma(a, b, c); }
// multiply both members by the complex number (c, s)
template <typename T> __device__ __forceinline__ Pair<T> pmul(const Pair<T>& x, T c, T s) {
  return {fmadd(x.ar, c, -(x.ai * s)), fmadd(x.ar, s, x.ai * c), fmadd(x.br, c, -(x.bi * s)), fmadd(x.br, s, x.bi * c)};
}
// eq. (Fstat) from the two transforms at one bin
template <typename T> __device__ __forceinline__ T two_f(const Pair<T>& x, T kA, T kB, T kC) {
  const T fa2 = fmadd(x.ar, x.ar, x.ai * x.ai);
  const T fb2 = fmadd(x.br, x.br, x.bi * x.bi);
  const T re = fmadd(x.ar, x.br, x.ai * x.bi);
  return fmadd(kB, fa2, fmadd(kA, fb2, -(kC * re)));
}
// multiply by -i
template <typename T> __device__ __forceinline__ Pair<T> pmul_mi(const Pair<T>& x) {
  return {x.ai, -x.ar, x.bi, -x.br};
}
template <typename T> __device__ __forceinline__ Pair<T> pzero() { return {T(0), T(0), T(0), T(0)}; }

// memory images: float pair = float4 (16 B); double pair = 2 x double2 (32 B)
template <typename T> struct PairMem;
template <> struct PairMem<float> { using type = float4; };
template <> struct PairMem<double> { struct alignas(16) type { double2 a, b; }; };

__device__ __forceinline__ Pair<float> pload(const float4* p) {
  float4 v = *p; return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ void pstore(float4* p, const Pair<float>& x) {
  *p = make_float4(x.ar, x.ai, x.br, x.bi);
}
__device__ __forceinline__ Pair<double> pload(const PairMem<double>::type* p) {
  double2 a = p->a, b = p->b; return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void pstore(PairMem<double>::type* p, const Pair<double>& x) {
  p->a = make_double2(x.ar, x.ai); p->b = make_double2(x.br, x.bi);
}
__device__ __forceinline__ Pair<float> pload_g(const float4* __restrict__ p) {
  float4 v = __ldg(p); return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Pair<double> pload_g(const PairMem<double>::type* __restrict__ p) {
  double2 a = __ldg(&p->a), b = __ldg(&p->b); return {a.x, a.y, b.x, b.y};
}

__device__ __forceinline__ float sinpi_t(float x) { return sinpif(x); }
__device__ __forceinline__ double sinpi_t(double x) { return sinpi(x); }
__device__ __forceinline__ void sincospi_t(float x, float* s, float* c) { sincospif(x, s, c); }
__device__ __forceinline__ void sincospi_t(double x, double* s, double* c) { sincospi(x, s, c); }

// Column layout of the resampled series G for pass A: column n1 = j mod N1
// takes lc pairs, its sample n2 = j / N1 at (n2 mod RL) lcs + n2 / RL, RL = 2^rl
// residues of lcs = ceil(samples per column / RL) pairs each.
struct GCol {
  int64_t lc;
  int lcs, rl;
  __host__ __device__ __forceinline__ int at(int n2) const { return (n2 & ((1 << rl) - 1)) * lcs + (n2 >> rl); }
};
inline GCol g_columns(int64_t n, int64_t n1, int rl) {
  const int64_t m = (n + n1 - 1) / n1;
  const int lcs = (int)((m + (1 << rl) - 1) >> rl);
  return GCol{(int64_t)lcs << rl, lcs, rl};
}

// ------------------------------------------------------------ host helpers
SkyPos sky_position(const Geo& g, double alpha, double delta);
// Blocks of the resampling kernel for n samples (its A, B, C partial sums).
size_t sky_partials_bytes(int64_t n);  // (zeroed once)
size_t resample_table_bytes();
cudaError_t launch_resample_table(const Geo& g, struct ResTab* t, cudaStream_t st);
// Steps (iii)-(v) for one sky position, and the spindown coefficients of job's
// templates (count 0: none).  Three launches.
void launch_sky(const Geo& g, int precision, const SkyPos& pos, const void* const* xh, const int* xh_dtype, void* G,
                int n1, GCol gc, void* partials, SkyConst* sky, int* err, const CoefJob& job, cudaStream_t st);
// Timing table: entries needed to cover [t_lo, t_hi] at spacing h, and the
// kernel that fills them (FP64 sincos, once per plan).
int time_table_entries(double t_lo, double t_hi, double h);
cudaError_t launch_time_table(const Geo& g, TimeTab* tab, RotCell* rot, cudaStream_t st);
void launch_tmpl_coef(const SkyPos& pos, const Geo& g, const CoefJob& job, cudaStream_t st);
// samples between the inputs of one of pass A's first butterflies
int64_t pass_a_spacing(int log2n, int log2_n2);
void launch_check_finite(const void* x, int dtype, int64_t n, int* err, cudaStream_t st);
// Gradient (adjoint.cu): per-plan sample tables and per-call scratch.
size_t grad_table_bytes(const Geo& g);
cudaError_t launch_grad_tables(const Geo& g, const void* const* xh, const int* dtype, void* base,
                               cudaStream_t st);
size_t grad_scratch_bytes(int n_cand, const Geo& g);
int grad_launches(int n_cand, const Geo& g);  // kernels of one launch_grad
cudaError_t launch_grad(const Geo& g, const void* tables, const fstat_candidate* cand_dev, int n_cand,
                        void* scratch, float* twoF, float* grad, cudaStream_t st);

// Twiddle tables of FP64 plans (tables.cu): pointers into one device block.
struct TwiddleTables {
  const void* a;   // pass A: Stockham roots, N2 entries
  const void* b;   // pass B: Stockham roots, N1 entries, then the twists
  size_t bytes;
};
TwiddleTables twiddle_layout(int log2n1, int log2n2, void* base);
cudaError_t build_twiddles(int log2n1, int log2n2, void* base, cudaStream_t st);

// Arguments of pass B's other epilogues: peaks mode reduces one template's
// 2F in the kernel instead of writing it bin by bin (fstat_compute_peaks);
// accumulate mode adds it to a row at a bin offset (fstat_semicoherent).
struct PeakArgs {
  unsigned long long* band_key;  // this template's row of band keys, or nullptr
  fstat_peak* peaks;             // crossing list [cap]
  unsigned long long* count;     // list counter, or nullptr (no list)
  long long cap;
  long long tmpl;                // template index stored with each crossing
  float thr;
  int log2_band;                 // log2(bins per band)
  int shift;                     // accumulate: bin m adds to bin m - shift
  int first;                     // accumulate: the sum starts here (every bin is written)
  int* err;                      // where a pass records FSTAT_ERR_TIMEOUT, or nullptr
  int wait_limit;                // polls of a tile's first bulk-copy wait (<= 0 with
                                 // wait_set: give up at once; unset: the default)
  int wait_set;
};

// Band key: order-preserving image of the float 2F in the high word, the
// complement of the bin in the low word, so an unsigned maximum picks the
// largest 2F and, among equal values, the smallest bin.  0 = no value.
__device__ __forceinline__ unsigned long long band_key(float v, unsigned bin) {
  unsigned u = __float_as_uint(v);
  u ^= (u & 0x80000000u) ? 0xffffffffu : 0x80000000u;
  return ((unsigned long long)u << 32) | (unsigned long long)(0xffffffffu - bin);
}

// CTA-wide FFT passes of FP64 plans; ca / cb = columns / rows per CTA and va /
// vb = schedule (0, the length's default, is the one compiled).  res > 0:
// persistent grid of at most res CTAs per SM (0 = every resident CTA).
cudaError_t launch_pass_a_f64(int log2_n2, int ca, int va, const void* G, GCol gc, int64_t n, int n1, const void* twA,
                              const TmplCoef* coef, void* Z, cudaStream_t st, int res);
// pk == nullptr: write 2F to out[n_fft]; otherwise reduce it as pk says.
cudaError_t launch_pass_b_f64(int log2_n1, int cb, int vb, const void* Z, int n2, const void* twB,
                              const SkyConst* sky, float* out, cudaStream_t st, const PeakArgs* pk, int res);
cudaError_t launch_pass_b_peak_f64(int log2_n1, int cb, int vb, const void* Z, int n2, const void* twB,
                                   const SkyConst* sky, const PeakArgs& pk, cudaStream_t st, int res);
// Accumulate mode: out[m - shift] += 2F[m] for 0 <= m - shift < n_fft; first:
// the sum starts with this term (0 where no m reaches).
cudaError_t launch_pass_b_acc_f64(int log2_n1, int cb, int vb, const void* Z, int n2, const void* twB,
                                  const SkyConst* sky, float* out, int shift, bool first, cudaStream_t st, int res);
// PeakArgs' wait fields from a plan's setting (< 0: the default limit)
inline void set_wait(PeakArgs& a, int wait_limit) {
  a.wait_set = wait_limit >= 0;
  a.wait_limit = wait_limit >= 0 ? wait_limit : 0;
}
// The warp-local FP32 passes (fft_warp.cuh).  Z: the intermediates of the
// launch's n_tmpl templates, one behind the other; coef[0..]: their coefficients;
// pass B writes template k to row ord[k] mod out_rows of out (ord == nullptr:
// one template, to out).  staging: pass A's columns staged in shared memory
// where that costs no occupancy (0), always (1; an error where they do not
// fit) or never (2).
// whether (ca, va) / (cb, vb) names a shape of the length
bool pass_a_shape(int log2_n2, int ca, int va);
bool pass_b_shape(int log2_n1, int cb, int vb);
// Layout of their intermediate for pass B's tiles of 2^cb rows: element
// (n1 = r + 2^rl j, k2) at ((k2 >> cb) N1 + r sub + j) 2^cb + k2 mod 2^cb.
struct ZLayout { int cb, rl, sub; };
ZLayout wpass_z_layout(int log2_n1, int cb);  // cb: rows per tile asked of pass B (0 = default)
int wpass_b_rows(int log2_n1, int cb);        // and what it runs with
cudaError_t launch_wpass_a(int log2_n2, int staging, const void* G, GCol gc, int64_t n, int n1, const TmplCoef* coef,
                           void* Z, ZLayout zy, int n_tmpl, int* err, int wait_limit, cudaStream_t st, int res);
int wpass_a_residues_log2(int log2_n2);  // GCol::rl for pass A of this length
cudaError_t launch_wpass_b(int log2_n1, int cb, void* Z, int n_tmpl, int n2, const SkyConst* sky, float* out,
                           const int* ord, int64_t out_rows, int* err, int wait_limit, cudaStream_t st, int res);
cudaError_t launch_wpass_b_acc(int log2_n1, int cb, void* Z, int n2, const SkyConst* sky, float* out, int shift,
                               bool first, int* err, int wait_limit, cudaStream_t st, int res);
cudaError_t launch_wpass_b_peak(int log2_n1, int cb, void* Z, int n_tmpl, int n2, const SkyConst* sky,
                                const int* ord, int n_bands, const PeakArgs& pk, int* err, int wait_limit,
                                cudaStream_t st, int res);

// One persistent launch of both FFT passes over T templates of one sky
// group (fft_fused.cuh).  kRing intermediates in flight; launch state of
// queue_ints(T) ints, zeroed before every launch.
constexpr int kRing = 3;
constexpr int kQueueHead = 4;
inline size_t queue_ints(int T) { return (size_t)kQueueHead + 2 * (size_t)T; }

struct FusedArgs {
  const float4* G;        // column-major resampled pairs (per-sky work)
  GCol gc;                // layout of G
  int n;                  // samples
  int n1, n2;             // split: n1 columns of n2 points (pass A), n2 rows of n1 points (pass B)
  const TmplCoef* coef;   // [T] spindown coefficients of the launch's templates
  const int* ord;         // [T] caller's template index of each (row = ord mod out_rows)
  int64_t out_rows;
  float* out;             // 2F rows of n1 * n2 floats
  const SkyConst* sky;
  float4* Z[kRing];       // intermediates
  int* q;                 // launch state (queue_ints(T) ints)
  int T;
  int na, nb, total;      // tiles per template of pass A, of pass B; items in the launch
  int* err;               // sticky error of the plan
  int wait_limit;         // polls of the first waits (when wait_set), else the defaults
  int wait_set;
};

// The fused launch for FP32 plans, compiled for the splits fused_supported
// names (cudaErrorInvalidConfiguration otherwise).
bool fused_supported(int log2n1, int log2n2);
cudaError_t launch_fused_f32(int log2n1, int log2n2, const FusedArgs& a, cudaStream_t st);

// Band keys of n rows x n_bands -> maximum 2F and its bin (band_bin may be null).
cudaError_t launch_band_decode(const unsigned long long* keys, int64_t count, float* band_max,
                               int32_t* band_bin, cudaStream_t st);

}  // namespace fstat
