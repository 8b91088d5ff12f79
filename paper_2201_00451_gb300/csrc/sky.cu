// Per-sky kernels: Sec. 3 steps (iii), (iv), (v) of the resampling method,
// antenna weighting, the noise-weighted detector sum, and the antenna-pattern
// integrals A, B, C, D of eq. (Fstat).  The result G = (G_a, G_b) is stored
// in the column-major layout the FFT pass A reads (GCol).
//
// Three launches per sky position: the delay table; the timing nodes; the
// resampling (step iii applied as the detector samples are staged), beside it
// A, B, C, D and the templates' spindown coefficients.  Trigonometry of the sky
// position alone is done on the host.
//
// Timing (t_m, the inversion T + t_m(T) = t_b, u = (T - t0)/dt) is FP64 in
// both precisions; f_h t_m is reduced mod 1 in FP64 before the sincos.

#include <math.h>

#include <algorithm>
#include <cmath>

#include "fstat_internal.cuh"

// Negative control for the parity tests (never in the regular build): with
// FSTAT_NEGCTRL_FP32_TIMING defined, f_h t_m and the sample position
// u = (T - t0) / dt are formed in FP32 instead of FP64, the precision loss
// the FP64 timing exists to prevent.  A test builds this variant separately
// and checks that its 2F fails the tolerance the regular build meets.
#ifdef FSTAT_NEGCTRL_FP32_TIMING
constexpr bool kNegCtrlFp32 = true;
#else
constexpr bool kNegCtrlFp32 = false;
#endif

namespace fstat {

namespace {

// The orbital phase and the sidereal rotation angle enter the timing only
// through their cosines and sines, which the plan tabulates every 30 s
// (k_time_table, FP64 sincos once per entry) over the span the timing can
// reach.  Per sky position the Roemer delay of each detector is then
// tabulated at the same epochs (k_sky_table), and every timing evaluation
// is the cubic through the four nearest entries, stored by its coefficients:
// the per-sky kernels are bound by the FP64 pipe (two operations per clock and
// SM), and a cubic takes 3 of its operations where the Lagrange weights of an
// epoch take 12 and their sum 4.  The interpolation error in t_m is ~1e-14 s
// (rotation term: (w_rot h)^4 * 9/16/24 * R_E/c at h = 30 s), below the FP64
// rounding of t_m itself.
struct TabPos {
  int i;     // entry before the epoch
  double f;  // fraction of the way to the next
};

__device__ __forceinline__ TabPos tab_pos(const Geo& g, double t) {
  const double x = (t - g.tab_t0) * g.tab_inv_h;
  int i = __double2int_rd(x);
  i = i < 1 ? 1 : (i > g.tab_n - 3 ? g.tab_n - 3 : i);
  return TabPos{i, x - (double)i};
}

// the cubic through values at -1, 0, 1, 2 (the differences are exact to their own
// rounding, so the small coefficients are as good as the values)
__device__ __forceinline__ Cubic cubic_through(double v0, double v1, double v2, double v3) {
  const double d0 = v1 - v0, d1 = v2 - v1, d2 = v3 - v2;
  const double s0 = d1 - d0, third = (d2 - d1) - s0;
  Cubic c;
  c.c0 = v1;
  c.c2 = 0.5 * s0;
  c.c3 = third * (1.0 / 6.0);
  c.c1 = d1 - c.c2 - c.c3;
  return c;
}
__device__ __forceinline__ double cubic_at(const Cubic& c, double f) {
  return fma(f, fma(f, fma(f, c.c3, c.c2), c.c1), c.c0);
}

__global__ void k_time_table(Geo g, TimeTab* __restrict__ tab) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.tab_n; i += gridDim.x * blockDim.x) {
    const double t = g.tab_t0 + (double)i / g.tab_inv_h;
    double so, co, sq, cq;
    sincos(g.orb_ph0 + g.w_orb * t, &so, &co);
    sincos(g.sid_ph0 + g.w_rot * t, &sq, &cq);
    tab[i] = TimeTab{co, so, cq, sq};
  }
}

// The rotation's cosine and sine by cubics of their own: about a cell's middle, y in
// [-Y, Y], cos y = 1 - y^2/2 + y^4/24 and sin y = y - y^3/6 with y^4 replaced by
// Y^2 y^2 - Y^4/8 (its best lower approximation): 8e-15 at 30 s, where the cubics
// through four entries leave 5e-13 of one sign, and 1.4e-12 of A and B.
__global__ void k_rot_cells(Geo g, RotCell* __restrict__ rot) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 1 || i > g.tab_n - 3) return;
  const double x = g.w_rot / g.tab_inv_h, Y = 0.5 * x, t = g.tab_t0 + ((double)i + 0.5) / g.tab_inv_h;
  double S, C;
  sincos(g.sid_ph0 + g.w_rot * t, &S, &C);
  const double e0 = 1.0 - Y * Y * Y * Y / 192.0, e2 = Y * Y / 24.0 - 0.5;
  auto cubic = [&](double k0, double k1, double k2, double k3) {  // in y = x f - Y
    Cubic c;
    c.c0 = k0 - Y * (k1 - Y * (k2 - Y * k3));
    c.c1 = x * (k1 - Y * (2.0 * k2 - 3.0 * Y * k3));
    c.c2 = x * x * (k2 - 3.0 * Y * k3);
    c.c3 = x * x * x * k3;
    return c;
  };
  rot[i] = RotCell{cubic(C * e0, -S, C * e2, S / 6.0), cubic(S * e0, C, S * e2, -C / 6.0)};
}

// t_m = (r_orb + r_rot) . n / c at every entry and the cubics between them, for
// every detector.  A block forms three entries more than it has cells.
constexpr int kTabThreads = 256, kTabOut = kTabThreads - 3;
__global__ void __launch_bounds__(kTabThreads) k_sky_table(const __grid_constant__ Geo g, const __grid_constant__ SkyPos s) {
  __shared__ double s_tm[kMaxDet][kTabThreads];
  const int t = threadIdx.x;
  const int i = (int)blockIdx.x * kTabOut + t;  // entry; cell i - 1 .. from threads 1 .. kTabOut
  if (i < g.tab_n) {
    const TimeTab e = g.tab[i];
    const double orb = s.ox * e.co + s.oy * e.so;
    for (int X = 0; X < g.n_det; ++X) s_tm[X][t] = orb + (s.rx[X] * e.cq + s.ry[X] * e.sq + s.rz[X]);
  }
  __syncthreads();
  if (t < 1 || t > kTabOut || i > g.tab_n - 3) return;
  for (int X = 0; X < g.n_det; ++X)
    g.tm_tab[(int64_t)X * g.tab_n + i] = cubic_through(s_tm[X][t - 1], s_tm[X][t], s_tm[X][t + 1], s_tm[X][t + 2]);
}

// FP32 tap weights of the general form: the quotient by the hardware reciprocal (2 ulp; its
// denominator len sin(pi (d - m)/len) lies between ~pi |d - m| and D + 1),
// and the Hamming taper's sine and cosine of an angle within +-pi/2 by the
// hardware unit (~4e-7 absolute on a factor near 1).  The Dirichlet sines
// themselves keep the accurate sincospi (their arguments can be tiny).  FP64
// keeps exact division and sincospi throughout.
__device__ __forceinline__ float tap_div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double tap_div(double a, double b) { return a / b; }
__device__ __forceinline__ void taper_sincospi(float x, float* s, float* c) {
  __sincosf(3.14159265358979323846f * x, s, c);
}
__device__ __forceinline__ void taper_sincospi(double x, double* s, double* c) { sincospi(x, s, c); }

// Per-tap constants of the interpolation kernel, one aligned entry per tap
// m = -D..D: cos, sin(pi m / len) (the Dirichlet denominator by angle
// addition) and cos, sin(pi m / (D + 1)) (the taper).
template <typename T> struct alignas(4 * sizeof(T)) TapK {
  T c, s, tc, ts;
};

// Cubic Lagrange weights at f = r / step between nodes 0 and 1 of nodes at
// -1, 0, 1, 2 (dyadic f: exact in FP64 but for the factors 1/6).
__device__ __forceinline__ void node_weights(int r, int step_log2, double* w) {
  const double f = (double)r / (double)(1 << step_log2);
  const double fm = f - 1.0, fp = f + 1.0, f2 = f - 2.0;
  w[0] = -f * fm * f2 * (1.0 / 6.0);
  w[1] = fp * fm * f2 * 0.5;
  w[2] = -fp * f * f2 * 0.5;
  w[3] = fp * f * fm * (1.0 / 6.0);
}
constexpr int kMaxStep = 64, kMaxD = 32;

}  // namespace

// What a resampling block would otherwise form again for every launch: node
// weights by j mod step, the step matrix M of A, B, C, the taps' constants.
struct ResTab {
  double w[kMaxStep][4], m[4][4];
  double fourth;  // see sum_abc
  alignas(16) float wf[kMaxStep][4];  // (read as float4)
  TapK<float> tf[2 * kMaxD + 1];
  TapK<double> td[2 * kMaxD + 1];
  float2 tt[kMaxD + 1];  // series form, see series_taps
};

namespace {

__device__ __forceinline__ const TapK<float>* taps_of(const ResTab* t, float) { return t->tf; }
__device__ __forceinline__ const TapK<double>* taps_of(const ResTab* t, double) { return t->td; }

// Dirichlet kernel of the full series (length N) or of the 2D + 1 taps themselves
template <typename T> __device__ __forceinline__ T kernel_len(const Geo& g) {
  return g.interp == FSTAT_INTERP_PERIODIC ? (T)(2 * g.dterms + 1) : (T)g.n;
}
template <typename T> __device__ void form_tap(const Geo& g, int m, TapK<T>* out) {
  T sn, cs;
  TapK<T> q;
  sincospi_t((T)m / kernel_len<T>(g), &sn, &cs);
  q.c = cs;
  q.s = sn;
  sincospi_t((T)m * ((T)1 / (T)(g.dterms + 1)), &sn, &cs);
  q.tc = cs;
  q.ts = sn;
  *out = q;
}
__global__ void k_resample_table(Geo g, ResTab* t) {
  const int i = threadIdx.x, step = 1 << g.node_log2, D = g.dterms;
  if (i < step) {
    node_weights(i, g.node_log2, t->w[i]);
    for (int q = 0; q < 4; ++q) t->wf[i][q] = (float)t->w[i][q];
  }
  if (i <= 2 * D) {
    form_tap(g, i - D, &t->tf[i]);
    form_tap(g, i - D, &t->td[i]);
    const float h = g.interp == FSTAT_INTERP_TAPERED ? (i - D) & 1 ? -0.46f : 0.46f : 0.f;
    if (i >= D) t->tt[i - D] = make_float2(h * t->tf[i].tc, h * t->tf[i].ts);
  }
  __syncthreads();
  if (i < 16) {
    double m = 0.0;
    for (int r = 0; r < step; ++r) m += t->w[r][i >> 2] * t->w[r][i & 3];
    t->m[i >> 2][i & 3] = m;
  } else if (i == 16) {
    double q = 0.0, p = 0.0;
    for (int r = 0; r < step; ++r) {
      const double f = (double)r / (double)step;
      q += (f + 1.0) * f * (f - 1.0) * (f - 2.0) * (1.0 / 24.0);
      p += f * (1.0 - f);
    }
    t->fourth = -2.0 * q / p;
  }
}

// Spindown polynomial of template i of the job (see TmplCoef).
__device__ __forceinline__ void tmpl_coef(const CoefJob& c, double j_ref, double dt, int64_t n, int i) {
  if (i >= c.count) return;
  const fstat_template tp = c.tmpl[c.order[c.first + i]];
  c.out[c.first + i] = spin_coef(j_ref, n, dt, tp.f1dot, tp.f2dot, c.spacing);
}
__global__ void __launch_bounds__(128)
k_tmpl_coef(const __grid_constant__ CoefJob job, double j_ref, double dt, int64_t n) {
  tmpl_coef(job, j_ref, dt, n, (int)blockIdx.x * 128 + (int)threadIdx.x);
}

// Timing nodes of the current sky position (FP64, every 2^node_log2 samples,
// from kNodeLead steps before sample 0 on): the Roemer delay at the detector time, and
// at the SSB epoch t_b^j the detector epoch T (T + t_m(T) = t_b^j: the
// fixed-point start T0 = t_b - t_m(t_b), for which a linear t_m is enough, then
// one Newton step; |dt_m/dT| ~ 1e-4 puts T0 within ~0.05 s of the root and
// |d2t_m/dT2| ~ 1e-10 /s the Newton step within ~1e-13 s of it, the root three
// fixed-point iterations reach), stored as v = (T - t0)/dt - j, and the antenna
// patterns at T (JKS 1998 eqs. 12-13).  The Newton step stays with the table
// cell of T0, whose cubic it leaves by 0.05 s in 30 s at most.
// Between nodes every per-sample quantity is the cubic interpolant through
// the four nearest nodes: t_m, T and a, b are smooth on the scale of the
// node spacing (rotation: (w_rot h)^4 R_E/c ~ 1e-14 s at h = 32 s), so for the
// times the interpolation error is below their FP64 rounding; a, b are within
// 6e-12 of the largest at 32 s (of which FP32 keeps 6e-8; FP64 plans' nodes lie
// closer, and A, B, C take in one more difference, see sum_abc).
//
// Bound by the FP64 pipe (~80 operations per node and detector), hence as few
// nodes as that accuracy allows (node_step_log2), no FP64 division, and the
// cubics above.  Two detectors, 10 days at 0.5 s: 10.6 us (63.7 with a node every
// 16 samples and Lagrange sums; 23.5 with the wider steps alone); 120 days at
// 1 s: 99 us (348, 251).
// Each block computes three nodes more than it stores, for the changes to the
// next node and the inner mark (NodeF32).
constexpr int kNodeThreads = 128, kNodeOut = kNodeThreads - 3;
// 1.5 2^20: added to a phase below 2^19 cycles it leaves the fraction in units of
// 2^-32 cycles, modulo a cycle, in the low word
constexpr double kTurns32 = 1572864.0;
__global__ void __launch_bounds__(kNodeThreads)
k_sky_nodes(const __grid_constant__ Geo g, const __grid_constant__ SkyPos s) {
  __shared__ double s_v[kNodeThreads], s_tm[kNodeThreads];
  __shared__ int s_vi[kNodeThreads];
  const int t = threadIdx.x;
  const int m = (int)blockIdx.x * kNodeOut + t - 1;  // stored by threads 1 .. kNodeOut
  const bool in = m >= 0 && m < g.n_nodes;
  const int step = 1 << g.node_log2;
  const int ji = (m - kNodeLead) * step;
  const double j = (double)ji;
  const double td = g.t0 + j * g.dt;
  const double tb = s.t_b0 + j * g.dt;
  const int X = blockIdx.y;
  const Cubic* tab = g.tm_tab + (int64_t)X * g.tab_n;
  SkyNode nd{};
  if (in) {
    TabPos p = tab_pos(g, tb);
    double T_ = tb - fma(p.f, tab[p.i].c1, tab[p.i].c0);
    p = tab_pos(g, T_);
    const Cubic c = tab[p.i];
    const double r = T_ + cubic_at(c, p.f) - tb;
    const double slope = fma(p.f, fma(p.f, 3.0 * c.c3, 2.0 * c.c2), c.c1);
    // r / (1 + dt_m/dT), the reciprocal by one Newton step from FP32
    const double den = fma(slope, g.tab_inv_h, 1.0);
    const double y = (double)__frcp_rn((float)den);
    const double dT = r * (y * fma(-den, y, 2.0));
    T_ -= dT;
    nd.v = fma(T_ - g.t0, g.inv_dt, -j);
    p.f = fma(-dT, g.tab_inv_h, p.f);
    const RotCell q = g.rot[p.i];
    const double cq = cubic_at(q.c, p.f), sq = cubic_at(q.s, p.f);
    const double cH = s.cx[X] * cq + s.sx[X] * sq, sH = s.sx[X] * cq - s.cx[X] * sq;
    nd.a = fma(cH, fma(s.ca[X][1], cH, fma(s.ca[X][2], sH, s.ca[X][3])), fma(s.ca[X][4], sH, s.ca[X][0]));
    nd.b = fma(cH, fma(s.cb[X][1], cH, fma(s.cb[X][2], sH, s.cb[X][3])), fma(s.cb[X][4], sH, s.cb[X][0]));
    p = tab_pos(g, td);
    nd.tm_det = cubic_at(tab[p.i], p.f);
  }
  // (a delay of 2^29 samples is far outside any data: every sample invalid)
  const int vi = max(-(1 << 29), min(1 << 29, __double2int_rn(nd.v)));
  s_vi[t] = vi;
  s_v[t] = nd.v;
  s_tm[t] = nd.tm_det;
  __syncthreads();
  if (!in || t < 1 || t > kNodeOut) return;
  const int64_t i = (int64_t)X * g.n_nodes + m;
  g.nodes[i] = nd;
  const bool next = m + 1 < g.n_nodes;
  NodeF32 f;
  f.a = (float)nd.a;
  f.b = (float)nd.b;
  f.vf = (float)(nd.v - (double)vi);
  f.dv = next ? (float)(s_v[t + 1] - nd.v) : 0.f;
  const double ph = g.f_het * nd.tm_det;
  const double d0 = next ? g.f_het * (s_tm[t + 1] - nd.tm_det) : 0.0;
  f.ph = (unsigned)__double2loint((ph - rint(ph)) + kTurns32);
  f.rate = (unsigned)__double2loint(fma(d0, __hiloint2double((1023 - g.node_log2) << 20, 0), kTurns32));  // d0 / step
  f.curv = m + 2 < g.n_nodes ? 2.f * (float)fma(g.f_het, s_tm[t + 2] - s_tm[t + 1], -d0) : 0.f;
  bool inner = false;
  if (m >= 1 && m + 2 < g.n_nodes) {
    const int lo = min(min(s_vi[t - 1], vi), min(s_vi[t + 1], s_vi[t + 2]));
    const int hi = max(max(s_vi[t - 1], vi), max(s_vi[t + 1], s_vi[t + 2]));
    // (a whole step of SSB samples, and all of their positions in the data)
    inner = hi - lo <= 4 && ji + step <= (int)g.n && ji + lo >= 3 && ji + (step - 1) + hi <= (int)g.n - 4;
  }
  f.vi_inner = 2 * vi + (inner ? 1 : 0);
  g.nodes32[i] = f;
}

// Steps (iii), (iv), (v), antenna weighting and detector sum, one SSB sample
// per thread and tile.  The sample positions u(j) of a tile's kSkyBlock
// consecutive SSB samples increase with j and span kSkyBlock samples give or
// take the delay's drift, so the block stages the detector samples its taps can
// touch, [rint(u_first) - D, rint(u_last) + D] of every detector, in shared
// memory (two barriers per tile), applying step (iii) on the way:
// z = x_h exp(-i 2 pi frac(f_h t_m(t_k))), divided by a common sigma_ref.  (Rescaling every detector's series by the same factor, with
// weights w_X = sigma_ref^2 / (2 sigma_X^2), scales G by sigma_ref and A, B, C by
// sigma_ref^2, which leaves eq. (Fstat) unchanged while every FP32 value stays
// O(1) whatever the units of x_h.)  Samples outside the data are staged as 0, the
// value that the taps there are to have.
//
// Taps.  FP32, full-series kernels: with x = d - m, |x| <= D + 1/2,
//   sin(pi x) / (N sin(pi x / N)) = (-1)^m sin(pi d)/pi (1/x + c2 x + c4 x^3 ..),
//   c2 = (pi/N)^2 / 6,
// one hardware reciprocal per tap; the c4 term is below 3e-9 where `series` is
// set (N above ~200 D; shorter series take the general form), and the taper's
// cosine by angle addition for +m and -m together.  Otherwise (short series, the
// periodic kernel, FP64) the denominator's sine by angle addition from per-tap
// constants.
//
// FP64 work per sample is kept to what needs it: the sample position u and
// a, b for the weighted sum G come from the FP32 image of the nodes in the
// mixed path (u's integer part exact, its fraction to ~6e-8 samples; G
// itself is FP32; the FP64 path keeps FP64 throughout);
// and A, B, C per node step: with a(r) = sum_q W_rq a_q the cubic
// interpolant of the step's four node values a_q, the step's
// sum_r a(r)^2 is the quadratic form a^T M a with M = sum_r W_r W_r^T
// (and likewise b^T M b, a^T M b), exact algebra in FP64, one thread per
// detector and step, in blocks of their own of the same launch, so that the
// FP64 work runs beside the others' FP32 work.  Callers read A to D as doubles, of
// which the cubic leaves 6e-12 at steps of 32 s: the node values take in the fourth
// difference (sum_abc), to 1e-14.  A launch of its own to add the
// sums and form the coefficients took 7 to 12 us; sums of the edges' samples by
// the sample blocks, 4 us more for a fence in every block.
//
// Bound by instruction issue (55 % of the slots; half of the warps resident) and the
// wait for a tile's samples.  Two detectors, D = 8, 10 days at 0.5 s: 70 us, where
// step (iii) as a pass of its own over memory and 25 instructions a tap took
// 17 + 17 + 122; 120 days at 1 s: 386 us (42 + 42 + 683).  D = 16, 400 001 samples:
// 24 us (45 with the constants of ResTab formed by every block).
constexpr int kWin = kSkyBlock + 2 * kMaxD + 8;  // staged window, samples (covers the drift)

template <typename T> struct C2;
template <> struct C2<float> { using type = float2; };
template <> struct C2<double> { using type = double2; };

struct XhArgs { const void* x[kMaxDet]; int c128[kMaxDet]; };

// z at detector sample k (0 <= k < n): step (iii) from the timing nodes
// (C128: some detector's series is in complex128)
template <typename T, bool C128>
__device__ __forceinline__ typename C2<T>::type z_sample(const Geo& g, int X, const void* xh, int c128, int k,
                                                         const double (*s_w)[4], const float (*s_wf)[4]) {
  const int r = k & ((1 << g.node_log2) - 1);
  const int m = X * g.n_nodes + (k >> g.node_log2) + kNodeLead;  // < 2^25
  double xr, xi;
  float xrf = 0.f, xif = 0.f;
  if (C128 && c128) {
    const double2 v = ((const double2*)xh)[k];
    xr = v.x * g.inv_sigma_ref;
    xi = v.y * g.inv_sigma_ref;
    xrf = (float)xr;
    xif = (float)xi;
  } else {
    const float2 v = ((const float2*)xh)[k];
    if constexpr (sizeof(T) == sizeof(float)) {
      xrf = v.x * g.isf;
      xif = v.y * g.isf;
    } else {
      xr = (double)v.x * g.inv_sigma_ref;
      xi = (double)v.y * g.inv_sigma_ref;
    }
  }
  if constexpr (sizeof(T) == sizeof(float) && !kNegCtrlFp32) {
    // The cubic through the four nodes written about the step's own one: with the
    // phase differences d of this step and of its neighbours, the weights sum to
    // ph + (r / step) d + w3 (d_next - d) - w0 (d_prev - d).  The first two terms in
    // integers modulo a cycle (exact but for rate's rounding, 63/2 units = 7e-9
    // cycles), the rest is ~1e-4 cycles.  In FP32 throughout d's rounding alone was
    // 3e-7 rad at 490 Hz and 64 samples a step, and grew with f_h.
    const float* wf = s_wf[r];
    const NodeF32* nf = g.nodes32 + m;
    const int4 q = *reinterpret_cast<const int4*>(&nf[0].vi_inner);  // vi_inner, ph, rate, curv
    const float p = fmaf((float)(int)((unsigned)q.y + (unsigned)r * (unsigned)q.z), (float)(1.0 / 2147483648.0),
                         fmaf(wf[3], __int_as_float(q.w), wf[0] * nf[-1].curv));  // half turns
    float sn, cs;
    sincospif(p, &sn, &cs);
    return make_float2(xrf * cs + xif * sn, xif * cs - xrf * sn);
  } else {
    const double* w = s_w[r];
    const SkyNode* nd = g.nodes + m;
    const double tm = w[0] * nd[-1].tm_det + w[1] * nd[0].tm_det + w[2] * nd[1].tm_det + w[3] * nd[2].tm_det;
    double ph = g.f_het * tm;
    if constexpr (kNegCtrlFp32) ph = (double)((float)g.f_het * (float)tm);
    ph -= floor(ph);
    if constexpr (sizeof(T) == sizeof(float)) {
      float sn, cs;
      sincospif(2.0f * (float)ph, &sn, &cs);
      return make_float2(xrf * cs + xif * sn, xif * cs - xrf * sn);
    } else {
      double sn, cs;
      sincospi(2.0 * ph, &sn, &cs);
      return make_double2(xr * cs + xi * sn, xi * cs - xr * sn);
    }
  }
}

__device__ __forceinline__ float rcp_approx(float x) {  // 1 ulp
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// taps -D..D by the series form: wp points at tap 0, tt[m] = taper's cos, sin
// (pi m / (D + 1)) times 0.46 (0 without taper), base 0.54 (1 without), both
// negated for odd m
template <int D_, typename TZ>
__device__ __forceinline__ void series_taps(int D, const TZ* wp, float d, float ct, float st, float c2,
                                            const float2* tt, float base, float* zr, float* zi) {
  const int n = D_ ? D_ : D;
  // m = 0
  float w = fmaf(ct, tt[0].x, base) * fmaf(c2, d, rcp_approx(d));
  TZ v = wp[0];
  float r = v.x * w, i = v.y * w;
#pragma unroll (D_ ? D_ : 4)
  for (int m = 1; m <= n; ++m) {
    const float2 t = tt[m];
    const float b0 = (m & 1) ? -base : base;
    const float e = fmaf(ct, t.x, b0);
    const float xp = d - (float)m, xm = d + (float)m;
    const float wp_ = fmaf(st, t.y, e) * fmaf(c2, xp, rcp_approx(xp));
    const float wm_ = fmaf(-st, t.y, e) * fmaf(c2, xm, rcp_approx(xm));
    const TZ a = wp[m], b = wp[-m];
    r = fmaf(a.x, wp_, r);
    i = fmaf(a.y, wp_, i);
    r = fmaf(b.x, wm_, r);
    i = fmaf(b.y, wm_, i);
  }
  *zr = r;
  *zi = i;
}

// Step (iv): the sample position u = k0 + dlt of SSB sample j at detector X,
// interpolated between the timing nodes (node: the step's, m its index within the
// detector).  FP32 path: u = j + v with v = vi + vf at the step's node plus the
// weighted node-to-node changes (the interpolating cubic written about that node),
// so the integer part is exact and only the fraction, |f| <~ 1/2, is rounded to
// FP32.  FP64 plans (and the FP32-timing negative control) form u in FP64.
// (k0 is held within 2^29: far outside the data, and invalid all the same.)
template <typename T> constexpr bool kWide = sizeof(T) == sizeof(double) || kNegCtrlFp32;
__device__ __forceinline__ int far_out(int k0) { return max(-(1 << 29), min(1 << 29, k0)); }
__device__ __forceinline__ int position(int j, float vf, float dvm, float dv, float dvp, int vi_inner, const float* wf, float* dlt) {
  // (explicit operations: sample blocks and sums decide alike which samples are valid)
  const float f = __fadd_rn(vf, __fmaf_rn(wf[2], dv, __fmaf_rn(wf[3], __fadd_rn(dv, dvp), __fmul_rn(-wf[0], dvm))));
  const float big = __fadd_rn(f, 12582912.f);  // 1.5 2^23 + rint(f)
  *dlt = __fsub_rn(f, __fsub_rn(big, 12582912.f));
  return far_out(j + (vi_inner >> 1) + (__float_as_int(big) - 0x4b400000));
}
template <typename T>
__device__ __forceinline__ int position(int j, const SkyNode* nd, const double* wn, T* dlt) {
  double u = (double)j + (wn[0] * nd[-1].v + wn[1] * nd[0].v + wn[2] * nd[1].v + wn[3] * nd[2].v);
  if constexpr (kNegCtrlFp32) u = (double)((float)j + (float)(u - (double)j));
  const int k0 = __double2int_rn(u);
  *dlt = (T)(u - (double)k0);
  return far_out(k0);
}

// Sums of the blocks that form A, B, C; done counts those that have left theirs.
struct Partials {
  unsigned* done;
  double* sum;  // [blocks][3]
};

// A, B, C over the node steps, block b of nb: a whole step of valid samples
// (inner) by its quadratic form, the samples of any other step one by one, a
// quarter of them per thread (a short series is mostly such steps: 3000 samples
// took 21 us with a step per thread).  The block that ends last adds the sums in
// a fixed order and forms D and eq. (Fstat)'s weights.
constexpr int kStepParts = 4;  // divides the shortest step
template <typename T>
__device__ __noinline__ void sum_abc(const Geo& g, int b, int nb, const Partials& left, SkyConst* sky, int* err) {
  __shared__ double red[3][kSkyBlock / 32];
  __shared__ bool last;
  const ResTab* tab = g.rtab;
  const int step = 1 << g.node_log2, t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int steps = (int)((g.n + step - 1) >> g.node_log2), total = steps * g.n_det;
  double v[3] = {0.0, 0.0, 0.0};
  for (int i = b * kSkyBlock + t; i < kStepParts * total; i += nb * kSkyBlock) {
    const int part = i / total, is = i - part * total;
    const int X = is / steps, sg = is - X * steps;
    const SkyNode* nd = g.nodes + X * g.n_nodes + sg + kNodeLead;
    const NodeF32* nf = g.nodes32 + X * g.n_nodes + sg + kNodeLead;
    const bool inner = nf[0].vi_inner & 1;
    if (inner && part > 0) continue;
    // the six nearest nodes: their mean fourth difference d adds d q(f) to the cubic,
    // q = (f+1) f (f-1) (f-2) / 24, which c f (1 - f) with the same sum over a step
    // stands for (to 2e-13 of a, b at a sample), a change of the outer nodes by -2 c d
    auto node_values = [&](double n0, double n1, double n2, double n3, double n4, double n5, double* v) {
      const double d = tab->fourth * (0.5 * ((n0 + n5) - 3.0 * (n1 + n4)) + (n2 + n3));
      v[0] = n1 + d;
      v[1] = n2;
      v[2] = n3;
      v[3] = n4 + d;
    };
    double av[4], bv[4];
    node_values(nd[-2].a, nd[-1].a, nd[0].a, nd[1].a, nd[2].a, nd[3].a, av);
    node_values(nd[-2].b, nd[-1].b, nd[0].b, nd[1].b, nd[2].b, nd[3].b, bv);
    double aa = 0.0, bb = 0.0, ab = 0.0;
    if (inner) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        double ma = 0.0, mb = 0.0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          ma += tab->m[q][r] * av[r];
          mb += tab->m[q][r] * bv[r];
        }
        aa += av[q] * ma;
        bb += bv[q] * mb;
        ab += av[q] * mb;
      }
    } else {
      const int per = step / kStepParts;
#pragma unroll 2
      for (int r = part * per; r < (part + 1) * per; ++r) {
        const int j = (sg << g.node_log2) + r;
        const double* wn = tab->w[r];
        int k0;
        T dlt;
        if constexpr (kWide<T>) k0 = position<T>(j, nd, wn, &dlt);
        else k0 = position(j, nf[0].vf, nf[-1].dv, nf[0].dv, nf[1].dv, nf[0].vi_inner, tab->wf[r], &dlt);
        if (j >= g.n || k0 < 0 || k0 > g.n - 1) continue;
        const double a = wn[0] * av[0] + wn[1] * av[1] + wn[2] * av[2] + wn[3] * av[3];
        const double c = wn[0] * bv[0] + wn[1] * bv[1] + wn[2] * bv[2] + wn[3] * bv[3];
        aa += a * a;
        bb += c * c;
        ab += a * c;
      }
    }
    const double w = g.w[X];
    v[0] += w * aa;
    v[1] += w * bb;
    v[2] += w * ab;
  }
  // over the block; result in thread 0
  auto reduce = [&] {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
      if (lane == 0) red[q][wid] = v[q];
    }
    __syncthreads();
    if (wid == 0)
      for (int q = 0; q < 3; ++q) {
        v[q] = lane < kSkyBlock / 32 ? red[q][lane] : 0.0;
        for (int o = kSkyBlock / 64; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
      }
  };
  reduce();
  if (nb > 1) {
    if (t == 0) {
      for (int q = 0; q < 3; ++q) left.sum[3 * b + q] = v[q];
      __threadfence();
      last = atomicAdd(left.done, 1u) == (unsigned)nb - 1;
      __threadfence();
    }
    __syncthreads();
    if (!last) return;
    for (int q = 0; q < 3; ++q) v[q] = t < nb ? __ldcg(left.sum + 3 * t + q) : 0.0;  // nb <= kSkyBlock
    reduce();
    if (t == 0) *left.done = 0;  // for the next launch
  }
  if (t > 0) return;
  double A = v[0], B = v[1], C = v[2];
  double D = A * B - C * C;
  sky->A = A;
  sky->B = B;
  sky->C = C;
  sky->D = D;
  const bool ok = isfinite(D) && D > 1e-12 * A * B && A > 0.0 && B > 0.0;
  if (!ok) {
    atomicCAS(err, 0, FSTAT_ERR_DEGENERATE);
    D = 1.0;
    A = B = C = 0.0;
  }
  const double inv = 1.0 / D;
  sky->kA = 2.0 * A * inv;
  sky->kB = 2.0 * B * inv;
  sky->kC = 4.0 * C * inv;
  sky->kAf = (float)sky->kA;
  sky->kBf = (float)sky->kB;
  sky->kCf = (float)sky->kC;
}

template <typename T, bool C128>
__global__ void __launch_bounds__(kSkyBlock, sizeof(T) == 4 ? 4 : 2)
k_resample(const __grid_constant__ Geo g, const __grid_constant__ XhArgs xh, typename PairMem<T>::type* __restrict__ G,
           int n1_log2, GCol gc, int tiles, int sample_blocks, const Partials part, int sum_blocks, SkyConst* __restrict__ sky,
           int* __restrict__ err, const __grid_constant__ CoefJob job, double j_ref) {
  using TZ = typename C2<T>::type;
  // the sums and the coefficients, by the launch's first blocks: both are chains of
  // FP64 operations that the others' time hides
  const int block = (int)blockIdx.x - ((int)gridDim.x - sample_blocks);
  if (block < 0) {
    if ((int)blockIdx.x < sum_blocks) sum_abc<T>(g, (int)blockIdx.x, sum_blocks, part, sky, err);
    else
      tmpl_coef(job, j_ref, g.dt, g.n, ((int)blockIdx.x - sum_blocks) * kSkyBlock + (int)threadIdx.x);
    return;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TZ* win_all = reinterpret_cast<TZ*>(smem_raw);  // [n_det][kWin]
  __shared__ TapK<T> tk[2 * kMaxD + 1];
  __shared__ float2 s_tt[kMaxD + 1];
  __shared__ int s_span[kMaxDet][2];
  __shared__ double s_w[kWide<T> ? kMaxStep : 1][4];  // node weights by j mod step
  __shared__ __align__(16) float s_wf[kMaxStep][4];
  const int step_log2 = g.node_log2, step = 1 << step_log2;
  const int D = g.dterms;
  const T len = kernel_len<T>(g);
  const bool taper = g.interp == FSTAT_INTERP_TAPERED;  // the Hamming taper only for the default kernel
  const T inv_taper = (T)1 / (T)(D + 1);
  // (pi (D + 1/2) / N)^4 7/360 < 3e-9
  const bool series = sizeof(T) == sizeof(float) && g.interp != FSTAT_INTERP_PERIODIC &&
                      3.14159265f * ((float)D + 0.5f) < 0.0198f * (float)g.n;
  const ResTab* tab = g.rtab;
  // (taps outside a staged window and short series take the general form)
  for (int m = threadIdx.x; m <= 2 * D; m += blockDim.x) tk[m] = taps_of(tab, T())[m];
  if (threadIdx.x >= 128 && threadIdx.x - 128 <= D) s_tt[threadIdx.x - 128] = tab->tt[threadIdx.x - 128];
  if (threadIdx.x < step) {
    *reinterpret_cast<float4*>(s_wf[threadIdx.x]) = *reinterpret_cast<const float4*>(tab->wf[threadIdx.x]);
    if (kWide<T>)
#pragma unroll
      for (int q = 0; q < 4; ++q) s_w[threadIdx.x][q] = tab->w[threadIdx.x][q];
  }
  __syncthreads();
  const double* wn = s_w[kWide<T> ? threadIdx.x & (step - 1) : 0];
  const float* wf = s_wf[threadIdx.x & (step - 1)];
  for (int tile = block; tile < tiles; tile += sample_blocks) {
    const int j0 = tile * kSkyBlock;
    const int j = j0 + (int)threadIdx.x;
    const int j_last = min(j0 + kSkyBlock, (int)g.n) - 1;
    const int node_j = (min(j, j_last) >> step_log2) + kNodeLead;
    int k0s[kMaxDet];
    T dlts[kMaxDet], was[kMaxDet], wbs[kMaxDet];
#pragma unroll
    for (int X = 0; X < kMaxDet; ++X) {
      if (X >= g.n_det) break;
      int k0;
      T dlt;
      if constexpr (!kWide<T>) {
        const NodeF32* nf = g.nodes32 + X * g.n_nodes + node_j;
        auto abvd = [&](int q) { return *reinterpret_cast<const float4*>(&nf[q]); };  // a, b, vf, dv
        const float4 m1 = abvd(-1), z0 = abvd(0), p1 = abvd(1), p2 = abvd(2);
        k0 = position(j, z0.z, m1.w, z0.w, p1.w, nf[0].vi_inner, wf, &dlt);
        // the antenna patterns at T, weighted
        const float wx = g.wf[X];
        was[X] = wx * (wf[0] * m1.x + wf[1] * z0.x + wf[2] * p1.x + wf[3] * p2.x);
        wbs[X] = wx * (wf[0] * m1.y + wf[1] * z0.y + wf[2] * p1.y + wf[3] * p2.y);
      } else {
        const SkyNode* nd = g.nodes + X * g.n_nodes + node_j;
        k0 = position<T>(j, nd, wn, &dlt);
        const double w = g.w[X];
        was[X] = (T)(w * (wn[0] * nd[-1].a + wn[1] * nd[0].a + wn[2] * nd[1].a + wn[3] * nd[2].a));
        wbs[X] = (T)(w * (wn[0] * nd[-1].b + wn[1] * nd[0].b + wn[2] * nd[1].b + wn[3] * nd[2].b));
      }
      if (j == j0) s_span[X][0] = k0;
      if (j == j_last) s_span[X][1] = k0;
      k0s[X] = k0;
      dlts[X] = dlt;
    }
    __syncthreads();  // the spans are in (and the previous tile's windows have been read)
    // the tile's windows of detector samples (u is monotonic in j)
    int los[kMaxDet], his[kMaxDet];
#pragma unroll
    for (int X = 0; X < kMaxDet; ++X) {
      if (X >= g.n_det) break;
      const int lo = s_span[X][0] - D;
      const int hi = min(s_span[X][1] + D, lo + kWin - 1);  // drift beyond the window: taps past it are formed alone
      los[X] = lo;
      his[X] = hi;
      TZ* win = win_all + X * kWin;
      // (the few samples past the block's width go to another warp for each detector)
      const int t = ((int)threadIdx.x - 64 * X) & (kSkyBlock - 1);
      for (int k = lo + t; k <= hi; k += kSkyBlock) {
        TZ v{};
        if (k >= 0 && k < g.n) v = z_sample<T, C128>(g, X, xh.x[X], xh.c128[X], k, s_w, s_wf);
        win[k - lo] = v;
      }
    }
    __syncthreads();
    Pair<T> acc = pzero<T>();
#pragma unroll
    for (int X = 0; X < kMaxDet; ++X) {
      if (X >= g.n_det) break;
      const TZ* win = win_all + X * kWin;
      const int k0 = k0s[X], lo = los[X], hi = his[X];
      const T dlt = dlts[X];
      const bool valid = j < g.n && k0 >= 0 && k0 <= g.n - 1;
      if (!valid) continue;
      T zr = 0, zi = 0;
      const int i0 = k0 - lo;  // window index of tap 0
      const bool inside = i0 >= D && i0 + D <= hi - lo;
      if (inside && dlt == (T)0) {
        zr = win[i0].x;
        zi = win[i0].y;
      } else {
        const T d = dlt;
        T sdt = 0, cdt = 0;
        const T sd = sinpi_t(d);
        if (taper) taper_sincospi(d * inv_taper, &sdt, &cdt);
        bool done = false;
        if constexpr (sizeof(T) == sizeof(float)) {
          if (series && inside) {
            const float base = taper ? 0.54f : 1.f;
            if (D == 8) series_taps<8>(D, win + i0, d, cdt, sdt, g.tap_c2, s_tt, base, &zr, &zi);
            else series_taps<0>(D, win + i0, d, cdt, sdt, g.tap_c2, s_tt, base, &zr, &zi);
            const float q = sd * 0.31830988618379067f;
            zr *= q;
            zi *= q;
            done = true;
          }
        }
        if (!done) {
          T sdl, cdl;
          sincospi_t(d / len, &sdl, &cdl);
          if (inside) {  // no bounds per tap (samples outside the data are staged as 0)
            const TZ* wp = win + i0;
#pragma unroll 4
            for (int m = -D; m <= D; ++m) {
              const TapK<T> q = tk[m + D];
              const T sx = sdl * q.c - cdl * q.s;
              T wgt = tap_div((m & 1) ? -sd : sd, len * sx);
              if (taper) wgt *= (T)0.54 + (T)0.46 * (cdt * q.tc + sdt * q.ts);
              zr += (T)wp[m].x * wgt;
              zi += (T)wp[m].y * wgt;
            }
          } else for (int m = -D; m <= D; ++m) {
            const int k = k0 + m;
            if (k < 0 || k >= g.n) continue;
            // sin(pi (d - m)) = (-1)^m sin(pi d); sin(pi (d - m)/len) by angle addition
            const TapK<T> q = tk[m + D];
            T wgt;
            if (d == (T)0) {
              wgt = m == 0 ? (T)1 : (T)0;
            } else {
              const T num = (m & 1) ? -sd : sd;
              const T sx = sdl * q.c - cdl * q.s;
              wgt = tap_div(num, len * sx);
              if (taper) wgt *= (T)0.54 + (T)0.46 * (cdt * q.tc + sdt * q.ts);
            }
            const int i = i0 + m;
            const TZ v = i >= 0 && i <= hi - lo ? win[i] : z_sample<T, C128>(g, X, xh.x[X], xh.c128[X], k, s_w, s_wf);
            zr += (T)v.x * wgt;
            zi += (T)v.y * wgt;
          }
        }
      }
      // the antenna-weighted detector sum G (FP32 a, b in the mixed path)
      const T wa = was[X], wb = wbs[X];
      acc.ar += wa * zr;
      acc.ai += wa * zi;
      acc.br += wb * zr;
      acc.bi += wb * zi;
    }
    if (j < g.n) {
      const int n2i = j >> n1_log2;
      pstore(G + (int64_t)(j - (n2i << n1_log2)) * gc.lc + gc.at(n2i), acc);
    }
  }
}

}  // namespace

int time_table_entries(double t_lo, double t_hi, double h) {
  return (int)std::ceil((t_hi - t_lo) / h) + 1;
}

cudaError_t launch_time_table(const Geo& g, TimeTab* tab, RotCell* rot, cudaStream_t st) {
  const int blocks = (g.tab_n + 255) / 256;
  k_time_table<<<blocks, 256, 0, st>>>(g, tab);
  k_rot_cells<<<blocks, 256, 0, st>>>(g, rot);
  return cudaGetLastError();
}

SkyPos sky_position(const Geo& g, double alpha, double delta) {
  SkyPos s{};
  const double ca = std::cos(alpha), sa = std::sin(alpha);
  const double sd = std::sin(delta), cd = std::cos(delta), s2d = 2.0 * sd * cd, c2d = cd * cd - sd * sd;
  const double nx = cd * ca, ny = cd * sa, nz = sd;  // unit vector to the source
  const double py = g.cos_obl * ny + g.sin_obl * nz;
  s.ox = g.au / g.c * nx;
  s.oy = g.au / g.c * py;
  // SSB grid start: t0 + orbital Roemer delay at the data midpoint
  const double ph = g.orb_ph0 + g.w_orb * (g.t0 + 0.5 * (double)g.n * g.dt);
  const double orb = g.au * (std::cos(ph) * nx + std::sin(ph) * py);
  s.t_b0 = g.t0 + orb / g.c;
  s.j_ref = (g.t_ref - s.t_b0) / g.dt;
  for (int X = 0; X < g.n_det; ++X) {
    const double s2g = g.s2g[X], c2g = g.c2g[X], sl = g.sl[X], cl = g.cl[X], s2l = g.s2l[X], c2l = g.c2l[X];
    s.rx[X] = g.rcl[X] / g.c * (g.clon[X] * nx + g.slon[X] * ny);
    s.ry[X] = g.rcl[X] / g.c * (g.clon[X] * ny - g.slon[X] * nx);
    s.rz[X] = g.rsl[X] / g.c * nz;
    s.cx[X] = ca * g.clon[X] + sa * g.slon[X];
    s.sx[X] = sa * g.clon[X] - ca * g.slon[X];
    // cos 2H = 2 cH^2 - 1, sin 2H = 2 sH cH
    const double a2 = s2g * (3.0 - c2l) * (3.0 - c2d) / 16.0, b2 = c2g * sl * sd;
    s.ca[X][0] = 0.75 * s2g * cl * cl * cd * cd - a2;
    s.ca[X][1] = 2.0 * a2;
    s.ca[X][2] = -0.5 * c2g * sl * (3.0 - c2d);
    s.ca[X][3] = 0.25 * s2g * s2l * s2d;
    s.ca[X][4] = -0.5 * c2g * cl * s2d;
    s.cb[X][0] = -b2;
    s.cb[X][1] = 2.0 * b2;
    s.cb[X][2] = 0.5 * s2g * (3.0 - c2l) * sd;
    s.cb[X][3] = c2g * cl * cd;
    s.cb[X][4] = 0.5 * s2g * s2l * cd;
  }
  return s;
}

// Up to eight tiles per resampling block, so that its tables are formed once
// for them, where that leaves six blocks per SM.
namespace {
int sample_blocks(int64_t n) {
  const int64_t tiles = (n + kSkyBlock - 1) / kSkyBlock, full = (int64_t)6 * device_sm_count();
  const int64_t per = std::min<int64_t>(8, std::max<int64_t>(1, tiles / full));
  return (int)((tiles + per - 1) / per);
}
// Blocks for the step sums, at most as many as the last one has threads to add: one
// per 256 samples, since an SM takes 16 cycles per FP64 warp instruction and a
// block's eight warps wait for one another (3001 samples, whole call: 52.8 us with a
// block per 1024 samples, 47.3 so).
int step_blocks(int64_t n) { return (int)std::min<int64_t>(std::min(device_sm_count(), kSkyBlock), n / 256 + 1); }
}  // namespace

size_t sky_partials_bytes(int64_t n) { return 16 + (size_t)step_blocks(n) * 3 * sizeof(double); }

size_t resample_table_bytes() { return sizeof(ResTab); }
cudaError_t launch_resample_table(const Geo& g, ResTab* t, cudaStream_t st) {
  k_resample_table<<<1, 2 * kMaxD + 1, 0, st>>>(g, t);
  return cudaGetLastError();
}

void launch_sky(const Geo& g, int precision, const SkyPos& pos, const void* const* xh, const int* xh_dtype, void* G,
                int n1, GCol gc, void* partials, SkyConst* sky, int* err, const CoefJob& job, cudaStream_t st) {
  k_sky_table<<<(g.tab_n + kTabOut - 1) / kTabOut, kTabThreads, 0, st>>>(g, pos);
  const dim3 nodes((unsigned)((g.n_nodes + kNodeOut - 1) / kNodeOut), (unsigned)g.n_det);
  k_sky_nodes<<<nodes, kNodeThreads, 0, st>>>(g, pos);
  XhArgs x{};
  bool c128 = false;
  for (int X = 0; X < g.n_det; ++X) {
    x.x[X] = xh[X];
    x.c128[X] = xh_dtype[X] == FSTAT_C128;
    c128 = c128 || x.c128[X];
  }
  const int samples = sample_blocks(g.n), sums = step_blocks(g.n), tiles = (int)((g.n + kSkyBlock - 1) / kSkyBlock);
  int l1 = 0;
  while ((1 << l1) < n1) ++l1;
  const int blocks = samples + sums + (job.count + kSkyBlock - 1) / kSkyBlock;
  const Partials part{(unsigned*)partials, (double*)((char*)partials + 16)};
  const size_t smem = (size_t)g.n_det * kWin * (precision == FSTAT_FP64 ? 16 : 8);  // at most 21 KB
  if (precision == FSTAT_FP64)
    k_resample<double, true><<<blocks, kSkyBlock, smem, st>>>(g, x, (PairMem<double>::type*)G, l1, gc, tiles, samples, part, sums, sky, err,
                                                              job, pos.j_ref);
  else if (c128)
    k_resample<float, true><<<blocks, kSkyBlock, smem, st>>>(g, x, (float4*)G, l1, gc, tiles, samples, part, sums, sky, err,
                                                              job, pos.j_ref);
  else
    k_resample<float, false><<<blocks, kSkyBlock, smem, st>>>(g, x, (float4*)G, l1, gc, tiles, samples, part, sums, sky, err,
                                                              job, pos.j_ref);
}

void launch_tmpl_coef(const SkyPos& pos, const Geo& g, const CoefJob& job, cudaStream_t st) {
  if (job.count == 0) return;
  k_tmpl_coef<<<(job.count + 127) / 128, 128, 0, st>>>(job, pos.j_ref, g.dt, g.n);
}

// Scan an input series for NaN/Inf.
template <typename TIn>
__global__ void k_check_finite(const TIn* __restrict__ x, int64_t n, int* err) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    TIn v = x[k];
    if (!isfinite((double)v.x) || !isfinite((double)v.y)) atomicCAS(err, 0, FSTAT_ERR_NONFINITE);
  }
}

void launch_check_finite(const void* x, int dtype, int64_t n, int* err, cudaStream_t st) {
  int blocks = (int)((n + 255) / 256);
  if (blocks > device_sm_count() * 32) blocks = device_sm_count() * 32;
  if (dtype == FSTAT_C128) k_check_finite<double2><<<blocks, 256, 0, st>>>((const double2*)x, n, err);
  else k_check_finite<float2><<<blocks, 256, 0, st>>>((const float2*)x, n, err);
}

}  // namespace fstat
