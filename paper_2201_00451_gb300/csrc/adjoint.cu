// 2F and its gradient in (f, f1dot, alpha, delta) at arbitrary parameters.
//
// The refined statistic is eq. (Fstat) with the demodulation integrals of
// eqs. (Fa_DET)/(Fb_DET) (Sec. 2) summed directly over detector samples at
// a single frequency:
//
//   Phi_k = (f - f_h) tau_k + f_h t_m(t_k) + f1dot tau_k^2/2 + f2dot tau_k^3/6   [cycles]
//   tau_k = t_k - t_ref + t_m(t_k),   t_m = (r(t_k) / c) . n(alpha, delta)
//   Fa = sum_X w_X sum_k x_X[k] a_X(t_k) e^{-i 2 pi Phi_k},  Fb with b,
//   a = d(t_k) : e+(alpha, delta),  b = d(t_k) : ex(alpha, delta)
//
// Over a block of S consecutive samples (a few tens of seconds) everything in
// these sums except x and the phase factor is a polynomial: the Earth turns
// by ~1e-3 rad.  So per candidate and block the phase is evaluated once in
// double-float (FP32 pairs, ~48 bits) at the block's middle sample together
// with its derivatives, per sample only
//
//   e_u = x_u exp(-i 2 pi (Phi(u) - Phi(0))),  E_q = sum_u e_u u^q,  q = 0, 1, 2
//
// is formed (a cubic in u, one sine/cosine, three complex sums), and Fa, Fb
// and their derivatives are combinations of E_0, E_1, E_2 with the local
// expansions of a, b, tau and dPhi/dtheta.  A, B, C need no sum at all: a and
// b are harmonics 0-2 of the sidereal angle, whose products sum over the
// sample grid in closed form.
//
// Bound by FP32 issue: ~22 instructions per candidate and sample plus ~480
// per block.  256 candidates of the 10-day two-detector data: 11.7 ms with the
// phase, the patterns and 29 sums evaluated at every sample (~300
// instructions), 1.19 ms here; one candidate 5.2 ms -> 0.08 ms (items of 2^14
// samples instead of 2^17 fill the GPU).

#include <math.h>

#include <algorithm>
#include <type_traits>

#include "fstat_internal.cuh"

namespace fstat {
namespace adj {

constexpr int kWarps = 8;               // (candidate, chunk) items per CTA, one warp each
constexpr int kChunkSamples = 1 << 14;  // samples per item: the unit of every sum, whatever the candidate count
constexpr int kAcc = 20;                // accumulated quantities per candidate
constexpr int kInner = 64;              // per-sample path: terms per first-level sum

// ------------------------------------------------------------ double-float
struct df {
  float h, l;
};
__device__ __forceinline__ df df_from(double x) {
  float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ df two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ df df_add(df a, df b) {
  df s = two_sum(a.h, b.h);
  float e = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
  float h = __fadd_rn(s.h, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s.h))};
}
__device__ __forceinline__ df df_mul(df a, df b) {
  float p = __fmul_rn(a.h, b.h);
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  float h = __fadd_rn(p, e);
  return {h, __fsub_rn(e, __fsub_rn(h, p))};
}
__device__ __forceinline__ df df_mulf(df a, float b) { return df_mul(a, {b, 0.f}); }
// fractional part of a double-float in [-1/2, 1/2]
__device__ __forceinline__ float df_frac(df a) {
  float k = rintf(a.h);
  return __fadd_rn(__fsub_rn(a.h, k), a.l);
}

// ------------------------------------------------------------ blocks
// Samples per block: the largest S whose half-span h = S dt / 2 keeps
// (2 w h)^3 / 6 <= 2e-8 for the sidereal and orbital rates w, the first
// neglected term of the patterns' expansion (FP32 rounding is 6e-8; the
// phase's, f R_E/c (w h)^4 / 24, is then below 1e-10 cycles).  For the
// sidereal rate that is dt <= 2.1 s (S = 32), 4.2 s (16), 8.4 s (8); beyond,
// S = 1 evaluates every sample by itself.  And short enough against the data: the
// third-order terms of the derivatives' sums, a' times the square of the time
// across a block, are 2 w h (S / n)^2 of them, kept to 1e-7 (100 samples at 2 s with
// S = 32: d/df1dot off by 4e-5; 511: 7.5e-6, with S = 1 3e-7).  At dt = 0.5 s that is
// S = 32 from 3457 samples on, 16 from 1223, 8 from 433.
int block_samples(const Geo& g) {
  const double w = std::max(fabs(g.w_rot), fabs(g.w_orb)) * g.dt;
  for (int S : {32, 16, 8}) {
    const double x = w * S;  // 2 w h
    if (x * x * x <= 1.2e-7 && x * S * S <= 1e-7 * (double)g.n * (double)g.n) return S;
  }
  return 1;
}

// Block tables, 32 blocks (one tile) at a time, field by field: at a block's
// middle sample the time since t_ref (double-float), r/c (double-float) and
// its first three derivatives per sample, and the sidereal angle's
// harmonics.  S = 1 keeps no derivatives.
enum Field { fTau = 0, fR = 2, fCos = 8, fR1 = 12, fR2 = 15, fR3 = 18, fAll = 21 };
constexpr int fields(int S) { return S == 1 ? (int)fR1 : (int)fAll; }

struct Layout {
  int S;
  int64_t tiles;        // tiles of 32 blocks per detector
  size_t x_bytes, node_bytes;
};
Layout layout(const Geo& g) {
  Layout l;
  l.S = block_samples(g);
  l.tiles = (g.n + 32 * l.S - 1) / (32 * l.S);
  l.x_bytes = (size_t)g.n_det * l.tiles * 32 * l.S * sizeof(float2);
  l.node_bytes = (size_t)g.n_det * l.tiles * 32 * fields(l.S) * sizeof(float);
  return l;
}

struct Series { const void* x[kMaxDet]; int dtype[kMaxDet]; };

// w x_h / sigma_ref, tile by tile as [i][lane] (sample i of the lane's
// block; pairs of samples side by side for S > 1), zero past the data: every
// later read is coalesced.
__global__ void k_series_table(Geo g, Series src, int S, int64_t tiles, float2* __restrict__ out) {
  const int X = blockIdx.y;
  const double scale = g.inv_sigma_ref * g.w[X];
  const int64_t total = tiles * 32 * S;
  for (int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
    const int64_t tile = o / (32 * S);
    const int q = (int)(o - tile * (32 * S));
    const int lane = S > 1 ? (q >> 1) & 31 : q;
    const int i = S > 1 ? 2 * (q >> 6) + (q & 1) : 0;
    const int64_t k = (tile * 32 + lane) * S + i;
    float2 v = make_float2(0.f, 0.f);
    if (k < g.n) {
      if (src.dtype[X] == FSTAT_C128) {
        const double2 d = ((const double2*)src.x[X])[k];
        v = make_float2((float)(d.x * scale), (float)(d.y * scale));
      } else {
        const float2 d = ((const float2*)src.x[X])[k];
        v = make_float2((float)(d.x * scale), (float)(d.y * scale));
      }
    }
    out[X * total + o] = v;
  }
}

__global__ void k_block_table(Geo g, int S, int64_t tiles, float* __restrict__ out) {
  const int X = blockIdx.y, nf = S == 1 ? fields(1) : fields(2);
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < tiles * 32;
       b += (int64_t)gridDim.x * blockDim.x) {
    const double k = (double)(b * S + S / 2), t = g.t0 + k * g.dt;
    double so, co, sp, cp;
    sincos(g.orb_ph0 + g.w_orb * t, &so, &co);
    sincos(g.lon[X] + g.sid_ph0 + g.w_rot * t, &sp, &cp);
    float* f = out + ((X * tiles + b / 32) * nf) * 32 + (b & 31);
    auto put = [&](int q, double v) { f[32 * q] = (float)v; };
    auto put2 = [&](int q, double v) {
      const float h = (float)v;
      f[32 * q] = h;
      f[32 * (q + 1)] = (float)(v - (double)h);
    };
    const double ox = g.au / g.c, oy = g.au * g.cos_obl / g.c, oz = g.au * g.sin_obl / g.c;
    const double rr = g.rcl[X] / g.c, wo = g.w_orb * g.dt, wr = g.w_rot * g.dt;
    put2(fTau, (g.t0 - g.t_ref) + k * g.dt);
    put2(fR, ox * co + rr * cp);
    put2(fR + 2, oy * so + rr * sp);
    put2(fR + 4, oz * so + g.rsl[X] / g.c);
    put(fCos, cp);
    put(fCos + 1, sp);
    put(fCos + 2, cp * cp - sp * sp);
    put(fCos + 3, 2.0 * sp * cp);
    if (S == 1) continue;
    put(fR1, -wo * ox * so - wr * rr * sp);
    put(fR1 + 1, wo * oy * co + wr * rr * cp);
    put(fR1 + 2, wo * oz * co);
    put(fR2, -wo * wo * ox * co - wr * wr * rr * cp);
    put(fR2 + 1, -wo * wo * oy * so - wr * wr * rr * sp);
    put(fR2 + 2, -wo * wo * oz * so);
    put(fR3, wo * wo * wo * ox * so + wr * wr * wr * rr * sp);
    put(fR3 + 1, -wo * wo * wo * oy * co - wr * wr * wr * rr * cp);
    put(fR3 + 2, -wo * wo * wo * oz * co);
  }
}

// ------------------------------------------------------------ candidates
constexpr int kPat = 6;  // a, b, da/dalpha, db/dalpha, da/ddelta, db/ddelta
// harmonics of the sidereal angle phi: 1, cos 2phi, sin 2phi, cos phi, sin phi
struct CandConst {
  df nx, ny, nz;           // sky vector
  float dna[3], dnd[3];    // d n / d alpha, d n / d delta
  df fmh;                  // f - f_h
  df fh;                   // f_h
  df f1h;                  // f1dot / 2
  df f2s;                  // f2dot / 6
  df step;                 // (f - f_h) dt, mod 1
  df dt;
  float f, f1, f2, pad_;   // for dPhi/dt_m = f + f1dot tau + f2dot tau^2 / 2
  float pat[kMaxDet][kPat][5];
  double abc[9];           // A, B, C, then d/dalpha, d/ddelta (read by k_finalize)
};

// Antenna patterns (JKS 1998 eqs. 12-13) as harmonics of phi for one
// detector: with H = alpha - phi and u = (1, cos 2H, sin 2H, cos H, sin H),
// a = sum ka_i u_i, b = sum kb_i u_i, and their sky derivatives.
__device__ void patterns(const Geo& g, int X, double sa, double ca, double sd, double cd, double (*p)[5]) {
  const double sl = g.sl[X], cl = g.cl[X], sg = g.s2g[X], cg = g.c2g[X], s2l = g.s2l[X], c2l = g.c2l[X];
  const double s2d = 2.0 * sd * cd, c2d = cd * cd - sd * sd;
  // value and d/ddelta of the coefficients
  const double k[4][5] = {
      {0.75 * sg * cl * cl * cd * cd, sg * (3.0 - c2l) * (3.0 - c2d) / 16.0, -0.25 * cg * sl * (3.0 - c2d),
       0.25 * sg * s2l * s2d, -0.5 * cg * cl * s2d},
      {0.0, cg * sl * sd, 0.25 * sg * (3.0 - c2l) * sd, cg * cl * cd, 0.5 * sg * s2l * cd},
      {-1.5 * sg * cl * cl * cd * sd, sg * (3.0 - c2l) * s2d / 8.0, -0.5 * cg * sl * s2d, 0.5 * sg * s2l * c2d,
       -cg * cl * c2d},
      {0.0, cg * sl * cd, 0.25 * sg * (3.0 - c2l) * cd, -cg * cl * sd, -0.5 * sg * s2l * sd}};
  const double s2a = 2.0 * sa * ca, c2a = ca * ca - sa * sa;
  auto turn = [&](const double* u, double* o) {
    o[0] = u[0];
    o[1] = u[1] * c2a + u[2] * s2a;
    o[2] = u[1] * s2a - u[2] * c2a;
    o[3] = u[3] * ca + u[4] * sa;
    o[4] = u[3] * sa - u[4] * ca;
  };
  for (int q = 0; q < 2; ++q) {
    const double da[5] = {0.0, 2.0 * k[q][2], -2.0 * k[q][1], k[q][4], -k[q][3]};  // d/dalpha of u
    turn(k[q], p[q]);
    turn(da, p[2 + q]);
    turn(k[2 + q], p[4 + q]);
  }
}

// sums over the sample grid of the products of two harmonics 1, cos 2phi, sin 2phi,
// cos phi, sin phi, per detector
struct Harmonics { double m[kMaxDet][5][5]; };

// sum_k w u(phi_k) v(phi_k) for two patterns u, v over the grid
__device__ __forceinline__ double pat_sum(const double* u, const double* v, const double (*m)[5]) {
  double t = 0.0;
  for (int i = 0; i < 5; ++i)
    for (int j = 0; j < 5; ++j) t += u[i] * m[i][j] * v[j];
  return t;
}

// A warp per candidate.  The chain of FP64 operations is what this kernel lasts (64 us
// with a thread per candidate, whatever their number), so the eleven sums of each
// detector go to lanes of their own.  With k_finalize's CTA per candidate a call for
// one candidate over 10 days takes 82 us instead of 137, for 256 of them 63 us less.
constexpr int kSums = 11;
__global__ void __launch_bounds__(32)
k_cand_consts(const __grid_constant__ Geo g, const __grid_constant__ Harmonics h, const fstat_candidate* __restrict__ cand,
              CandConst* __restrict__ out) {
  __shared__ double s_sum[kMaxDet * kSums];
  const int lane = threadIdx.x;
  const fstat_candidate c = cand[blockIdx.x];
  CandConst& k = out[blockIdx.x];
  double sa, ca, sd, cd;
  sincos(c.alpha, &sa, &ca);
  sincos(c.delta, &sd, &cd);
  for (int i = lane; i < g.n_det * kSums; i += 32) {
    const int X = i / kSums, q = i - X * kSums;
    double p[kPat][5];
    patterns(g, X, sa, ca, sd, cd, p);
    if (q < kPat)
      for (int m = 0; m < 5; ++m) k.pat[X][q][m] = (float)p[q][m];
    // 0-2: aa, bb, ab; then a da, b db, da b, a db by alpha and by delta
    const int d = q < 3 ? 0 : q < 7 ? 1 : 2, e = q < 3 ? q : (q - 3) & 3;
    const double *da = p[2 * d], *db = p[2 * d + 1];
    const double* u = e == 1 ? p[1] : d && e == 2 ? da : p[0];
    const double* v = e == 0 ? da : d && e == 2 ? p[1] : db;
    s_sum[i] = pat_sum(u, v, h.m[X]);
  }
  __syncwarp();
  if (lane < 9) {
    const int d = lane / 3, e = lane - 3 * d;
    double t = 0.0;
    for (int X = 0; X < g.n_det; ++X) {
      const double* r = s_sum + X * kSums + (d ? 4 * d - 1 : 0);
      const double w = d ? 2.0 * g.w[X] : g.w[X];
      t += d && e == 2 ? g.w[X] * (r[2] + r[3]) : w * r[e];
    }
    k.abc[lane] = t;
  }
  if (lane > 0) return;
  k.nx = df_from(cd * ca);
  k.ny = df_from(cd * sa);
  k.nz = df_from(sd);
  k.dna[0] = (float)(-cd * sa);
  k.dna[1] = (float)(cd * ca);
  k.dna[2] = 0.f;
  k.dnd[0] = (float)(-sd * ca);
  k.dnd[1] = (float)(-sd * sa);
  k.dnd[2] = (float)cd;
  k.fmh = df_from(c.f - g.f_het);
  k.fh = df_from(g.f_het);
  k.f1h = df_from(c.f1dot / 2.0);
  k.f2s = df_from(c.f2dot / 6.0);
  const double st = (c.f - g.f_het) * g.dt;
  k.step = df_from(st - rint(st));
  k.f = (float)c.f;
  k.f1 = (float)c.f1dot;
  k.f2 = (float)c.f2dot;
  k.dt = df_from(g.dt);
  k.pad_ = 0.f;
}

// ------------------------------------------------------------ the sums
// value, first and second derivative per sample (at a block's middle) of a
// pattern; w = the sidereal angle per sample
struct Local { float v, d1, d2; };
template <bool DERIV>
__device__ __forceinline__ Local local(const float* p, float c1, float s1, float c2, float s2, float w) {
  const float h2 = p[1] * c2 + p[2] * s2, h1 = p[3] * c1 + p[4] * s1;
  Local r{p[0] + h2 + h1, 0.f, 0.f};
  if constexpr (DERIV) {
    const float q2 = p[2] * c2 - p[1] * s2, q1 = p[4] * c1 - p[3] * s1;
    r.d1 = w * (2.f * q2 + q1);
    r.d2 = -w * w * (4.f * h2 + h1);
  }
  return r;
}

struct cpx { float r, i; };

// a - rint(a) for |a| < 2^22
__device__ __forceinline__ float less_rint(float a) {
  return __fsub_rn(a, __fsub_rn(__fadd_rn(a, 12582912.f), 12582912.f));
}

// One warp per (candidate, chunk of kChunkSamples samples): lane l of a tile
// takes the tile's block l.  Neighbouring warps take neighbouring candidates
// of one chunk, so the tables are read from L1.
// accumulated quantities (kAcc): 0-1 Fa, 2-3 Fb, 4-7 dFa,dFb/df, 8-11 d/df1dot,
// 12-15 d/dalpha, 16-19 d/ddelta
template <int S>
__global__ void __launch_bounds__(kWarps * 32, 2)
k_moments(int n_det, int64_t tiles, const float2* __restrict__ xt, const float* __restrict__ nodes, float w_step,
          const CandConst* __restrict__ cc, int n_cand, int n_chunks, double* __restrict__ partial) {
  constexpr int NF = fields(S);
  constexpr int kTiles = kChunkSamples / (32 * S);
  __shared__ CandConst sc[kWarps];
  __shared__ float s_red[kWarps][kAcc][33];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t item = (int64_t)blockIdx.x * kWarps + warp;
  if (item >= (int64_t)n_cand * n_chunks) return;
  const int chunk = (int)(item / n_cand), cand = (int)(item - (int64_t)chunk * n_cand);
  {
    const int* src = reinterpret_cast<const int*>(cc + cand);
    int* dst = reinterpret_cast<int*>(&sc[warp]);
    for (int q = lane; q < (int)(sizeof(CandConst) / 4); q += 32) dst[q] = src[q];
  }
  __syncwarp();
  const CandConst& K = sc[warp];
  const float two_pi = 6.28318530717958647692f;
  const int64_t beg = (int64_t)chunk * kTiles, end = min(beg + kTiles, (int64_t)n_det * tiles);
  float acc[kAcc], outer[S == 1 ? kAcc : 1];
#pragma unroll
  for (int q = 0; q < kAcc; ++q) acc[q] = 0.f;
  if constexpr (S == 1)
#pragma unroll
    for (int q = 0; q < kAcc; ++q) outer[q] = 0.f;
  for (int64_t tile = beg; tile < end; ++tile) {
    const int X = (int)(tile / tiles);
    const float* nd = nodes + (tile * NF) * 32 + lane;
    auto fld = [&](int q) { return __ldg(nd + 32 * q); };
    const float rx = fld(fR), ry = fld(fR + 2), rz = fld(fR + 4);
    // t_m = (r/c) . n, tau and Phi at the block's middle sample, in double-float
    const df tm = df_add(df_add(df_mul({rx, fld(fR + 1)}, K.nx), df_mul({ry, fld(fR + 3)}, K.ny)),
                         df_mul({rz, fld(fR + 5)}, K.nz));
    const df tau = df_add({fld(fTau), fld(fTau + 1)}, tm);
    const df tau2 = df_mul(tau, tau);
    const df ph = df_add(df_add(df_mul(K.fmh, tau), df_mul(K.fh, tm)),
                         df_add(df_mul(K.f1h, tau2), df_mul(K.f2s, df_mul(tau2, tau))));
    const float t = tau.h;
    const float rate = K.f + K.f1 * t + 0.5f * K.f2 * t * t;  // dPhi/dt_m
    bool wide = false;
    float p1h = 0.f, p1l = 0.f, p2h = 0.f, p2 = 0.f, p3 = 0.f, dtau = 0.f, r1x = 0.f, r1y = 0.f, r1z = 0.f, r2x = 0.f, r2y = 0.f,
          r2z = 0.f;
    if constexpr (S > 1) {
      r1x = fld(fR1); r1y = fld(fR1 + 1); r1z = fld(fR1 + 2);
      r2x = fld(fR2); r2y = fld(fR2 + 1); r2z = fld(fR2 + 2);
      const float d1 = r1x * K.nx.h + r1y * K.ny.h + r1z * K.nz.h;
      const float d2 = r2x * K.nx.h + r2y * K.ny.h + r2z * K.nz.h;
      const float d3 = fld(fR3) * K.nx.h + fld(fR3 + 1) * K.ny.h + fld(fR3 + 2) * K.nz.h;
      dtau = K.dt.h + d1;
      const float spin = K.f1 + K.f2 * t, rate1 = (K.f1 * t + 0.5f * K.f2 * t * t) * dtau;
      // dPhi per sample = (f - f_h) dt + f dt_m + (f1dot tau + f2dot tau^2/2) dtau,
      // mod 1 (u is an integer), split so that u p1h is exact
      df s = two_sum(K.step.h, K.f * d1);
      s.l += K.step.l;
      p2 = 0.5f * (rate * d2 + spin * dtau * dtau);
      p3 = (1.f / 6.f) * (rate * d3 + 3.f * spin * dtau * d2 + K.f2 * dtau * dtau * dtau);
      // a continuous-wave source's spindown moves the frequency by far less
      // than a bin of 1/dt over the data; a short series admits larger ones
      constexpr float h = 0.5f * S;
      wide = __any_sync(0xffffffffu, fabsf(rate1) + h * h * (fabsf(p2) + h * fabsf(p3)) > 0.0625f);
      if (wide) {  // the spindown's part of the slope and curvature in double-float, both mod 1
        df dt1 = two_sum(K.dt.h, d1);
        dt1.l += K.dt.l;
        const df a = df_mulf(df_mul(K.f1h, tau), 2.f), b = df_mulf(df_mul(K.f2s, tau2), 3.f);
        const df q = df_mul(df_add(a, b), dt1);
        s = df_add(s, {__fsub_rn(q.h, rintf(q.h)), q.l});
        const df c = df_mul(df_mul(df_add(K.f1h, df_mulf(df_mul(K.f2s, tau), 3.f)), dt1), dt1);
        const float hi = __fsub_rn(c.h, rintf(c.h));
        p2h = rintf(hi * 16384.f) * (1.f / 16384.f);
        p2 = __fadd_rn(__fsub_rn(hi, p2h), __fadd_rn(c.l, 0.5f * rate * d2));
      } else {
        const float e = s.l;
        s = two_sum(s.h, rate1);
        s.l += e;
      }
      const float hi = __fsub_rn(s.h, rintf(s.h));
      p1h = rintf(hi * 131072.f) * (1.f / 131072.f);
      p1l = __fadd_rn(__fsub_rn(hi, p1h), s.l);
    }
    // the block's moments
    cpx E0{0.f, 0.f}, E1{0.f, 0.f}, E2{0.f, 0.f};
    if constexpr (S > 1) {
      const float4* x = reinterpret_cast<const float4*>(xt + tile * (32 * S)) + lane;
      auto moments = [&](auto far) {
#pragma unroll
        for (int i = 0; i < S; i += 2) {
          const float4 v = __ldg(x + 16 * i);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float u = (float)(i + e - S / 2);
            const float xr = e ? v.z : v.x, xi = e ? v.w : v.y;
            float f = fmaf(u, fmaf(u, fmaf(u, p3, p2), p1l), less_rint(__fmul_rn(u, p1h)));
            if constexpr (decltype(far)::value) f = less_rint(f + less_rint(__fmul_rn(u * u, p2h)));
            float sn, cs;
            __sincosf(two_pi * f, &sn, &cs);
            const float er = xr * cs + xi * sn, ei = xi * cs - xr * sn;
            E0.r += er;
            E0.i += ei;
            E1.r = fmaf(u, er, E1.r);
            E1.i = fmaf(u, ei, E1.i);
            E2.r = fmaf(u * u, er, E2.r);
            E2.i = fmaf(u * u, ei, E2.i);
          }
        }
      };
      if (wide) moments(std::true_type());
      else moments(std::false_type());
    } else {
      const float2 v = __ldg(xt + tile * 32 + lane);
      E0 = {v.x, v.y};
    }
    {
      // (its error is common to the block: the accurate function)
      float sn, cs;
      sincospif(2.f * df_frac(ph), &sn, &cs);
      auto rot = [&](cpx& e) { e = {e.r * cs + e.i * sn, e.i * cs - e.r * sn}; };
      rot(E0);
      if constexpr (S > 1) {
        rot(E1);
        rot(E2);
      }
    }
    const float c1 = fld(fCos), s1 = fld(fCos + 1), c2 = fld(fCos + 2), s2 = fld(fCos + 3);
    // dPhi/dalpha, dPhi/ddelta (over 2 pi) and their expansions
    const float ra = rx * K.dna[0] + ry * K.dna[1], rd = rx * K.dnd[0] + ry * K.dnd[1] + rz * K.dnd[2];
    float ga[3] = {rate * ra, 0.f, 0.f}, gd[3] = {rate * rd, 0.f, 0.f};
    if constexpr (S > 1) {
      const float drate = (K.f1 + K.f2 * t) * dtau;
      const float ra1 = r1x * K.dna[0] + r1y * K.dna[1], rd1 = r1x * K.dnd[0] + r1y * K.dnd[1] + r1z * K.dnd[2];
      ga[1] = rate * ra1 + drate * ra;
      gd[1] = rate * rd1 + drate * rd;
      // the frequency's own curvature, for large second spindowns (read here: kept
      // over the loop, f2dot costs a spilled register and 1.7 % of the kernel)
      const float drate2 = 0.5f * *(const volatile float*)&K.f2 * dtau * dtau;
      ga[2] = 0.5f * rate * (r2x * K.dna[0] + r2y * K.dna[1]) + drate * ra1 + drate2 * ra;
      gd[2] = 0.5f * rate * (r2x * K.dnd[0] + r2y * K.dnd[1] + r2z * K.dnd[2]) + drate * rd1 + drate2 * rd;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {  // a, b
      const Local p = local<(S > 1)>(K.pat[X][q], c1, s1, c2, s2, w_step);
      // sum e p u^m over the block
      cpx m0{p.v * E0.r, p.v * E0.i}, m1{0.f, 0.f}, m2{0.f, 0.f};
      if constexpr (S > 1) {
        const float h2 = 0.5f * p.d2;
        m0.r = fmaf(p.d1, E1.r, fmaf(h2, E2.r, m0.r));
        m0.i = fmaf(p.d1, E1.i, fmaf(h2, E2.i, m0.i));
        m1 = {fmaf(p.d1, E2.r, p.v * E1.r), fmaf(p.d1, E2.i, p.v * E1.i)};
        m2 = {p.v * E2.r, p.v * E2.i};
      }
      // sum e p g for a function g = g0 + g1 u + g2 u^2
      auto times = [&](float g0, float g1, float g2) -> cpx {
        if constexpr (S > 1) return {fmaf(g2, m2.r, fmaf(g1, m1.r, g0 * m0.r)), fmaf(g2, m2.i, fmaf(g1, m1.i, g0 * m0.i))};
        else return {g0 * m0.r, g0 * m0.i};
      };
      acc[2 * q] += m0.r;
      acc[2 * q + 1] += m0.i;
      // d/dtheta of e p = e (p_theta - i 2 pi Phi_theta p)
      const cpx vf = times(two_pi * t, two_pi * dtau, 0.f);
      const cpx v1 = times(two_pi * 0.5f * t * t, two_pi * t * dtau, two_pi * 0.5f * dtau * dtau);
      acc[4 + 2 * q] += vf.i;
      acc[5 + 2 * q] -= vf.r;
      acc[8 + 2 * q] += v1.i;
      acc[9 + 2 * q] -= v1.r;
#pragma unroll
      for (int d = 0; d < 2; ++d) {  // alpha, delta
        const float* gg = d ? gd : ga;
        const cpx vg = times(two_pi * gg[0], two_pi * gg[1], two_pi * gg[2]);
        const Local y = local<(S > 1)>(K.pat[X][2 + 2 * d + q], c1, s1, c2, s2, w_step);
        cpx z{y.v * E0.r, y.v * E0.i};
        if constexpr (S > 1) {
          const float h2 = 0.5f * y.d2;
          z.r = fmaf(y.d1, E1.r, fmaf(h2, E2.r, z.r));
          z.i = fmaf(y.d1, E1.i, fmaf(h2, E2.i, z.i));
        }
        acc[12 + 4 * d + 2 * q] += z.r + vg.i;
        acc[13 + 4 * d + 2 * q] += z.i - vg.r;
      }
    }
    if constexpr (S == 1) {
      if (((tile - beg) & (kInner - 1)) == kInner - 1) {
#pragma unroll
        for (int q = 0; q < kAcc; ++q) { outer[q] += acc[q]; acc[q] = 0.f; }
      }
    }
  }
  // the lanes' sums through shared memory: lane q adds quantity q's 32 values
  // in double-float, which costs a tenth of FP64 adds on this GPU
#pragma unroll
  for (int q = 0; q < kAcc; ++q) {
    if constexpr (S == 1) acc[q] += outer[q];
    s_red[warp][q][lane] = acc[q];
  }
  __syncwarp();
  if (lane < kAcc) {
    df s{0.f, 0.f};
    for (int l = 0; l < 32; ++l) {
      const df a = two_sum(s.h, s_red[warp][lane][l]);
      s = {a.h, __fadd_rn(s.l, a.l)};
    }
    partial[item * kAcc + lane] = (double)s.h + (double)s.l;
  }
}

// sum the chunk partials (fixed order) and apply the chain rule in FP64, one
// CTA per candidate (a warp alone took 30 us for the 211 chunks of 10 days);
// partial[chunk][cand][kAcc]
__global__ void __launch_bounds__(kWarps * 32)
k_finalize(const double* __restrict__ partial, const CandConst* __restrict__ cc, int n_cand, int n_chunks,
           float* __restrict__ twoF, float* __restrict__ grad) {
  __shared__ double s_sum[kWarps][kAcc];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x;
  if (lane < kAcc) {
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    int c = warp;
    for (; c + 3 * kWarps < n_chunks; c += 4 * kWarps)
#pragma unroll
      for (int q = 0; q < 4; ++q) t[q] += partial[((int64_t)(c + q * kWarps) * n_cand + i) * kAcc + lane];
    for (; c < n_chunks; c += kWarps) t[0] += partial[((int64_t)c * n_cand + i) * kAcc + lane];
    s_sum[warp][lane] = (t[0] + t[1]) + (t[2] + t[3]);
  }
  __syncthreads();
  if (warp > 0) return;
  if (lane < kAcc) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += s_sum[w][lane];
    s_sum[0][lane] = t;
  }
  __syncwarp();
  if (lane >= 4) return;
  const double* s = s_sum[0];
  const double* m = cc[i].abc;
  const double A = m[0], B = m[1], C = m[2];
  const double D = A * B - C * C;
  const double far = s[0], fai = s[1], fbr = s[2], fbi = s[3];
  const double fa2 = far * far + fai * fai, fb2 = fbr * fbr + fbi * fbi, re = far * fbr + fai * fbi;
  const double N = B * fa2 + A * fb2 - 2.0 * C * re;
  const int j = lane;  // d/d(f, f1dot, alpha, delta)
  if (j == 0) twoF[i] = (float)(2.0 * N / D);
  const double dar = s[4 + 4 * j], dai = s[5 + 4 * j], dbr = s[6 + 4 * j], dbi = s[7 + 4 * j];
  const double dfa2 = 2.0 * (far * dar + fai * dai);
  const double dfb2 = 2.0 * (fbr * dbr + fbi * dbi);
  const double dre = dar * fbr + dai * fbi + far * dbr + fai * dbi;
  double dA = 0.0, dB = 0.0, dC = 0.0;
  if (j >= 2) {
    dA = m[3 * (j - 1)];
    dB = m[3 * (j - 1) + 1];
    dC = m[3 * (j - 1) + 2];
  }
  const double dN = dB * fa2 + B * dfa2 + dA * fb2 + A * dfb2 - 2.0 * (dC * re + C * dre);
  const double dD = dA * B + A * dB - 2.0 * C * dC;
  grad[4 * i + j] = (float)(2.0 * (dN * D - N * dD) / (D * D));
}

// sum_{k < n} exp(i m phi_k), phi_k = phi_0 + k step: the geometric sum
// exp(i m (phi_0 + (n-1) step / 2)) sin(n x) / sin(x), x = m step / 2
Harmonics harmonics(const Geo& g) {
  Harmonics h{};
  for (int X = 0; X < g.n_det; ++X) {
    double C[5], S[5];
    for (int m = 0; m <= 4; ++m) {
      const double step = g.w_rot * g.dt, x = 0.5 * m * step, n = (double)g.n, sx = sin(x);
      // at a multiple of pi the quotient's limit, n cos(n x) / cos(x)
      const double amp = fabs(sx) < 1e-14 ? n * cos(n * x) / cos(x) : sin(n * x) / sx;
      const double mid = m * (g.lon[X] + g.sid_ph0 + g.w_rot * g.t0 + 0.5 * (n - 1.0) * step);
      C[m] = amp * cos(mid);
      S[m] = amp * sin(mid);
    }
    const double m[5][5] = {{C[0], C[2], S[2], C[1], S[1]},
                            {C[2], 0.5 * (C[0] + C[4]), 0.5 * S[4], 0.5 * (C[3] + C[1]), 0.5 * (S[3] - S[1])},
                            {S[2], 0.5 * S[4], 0.5 * (C[0] - C[4]), 0.5 * (S[3] + S[1]), 0.5 * (C[1] - C[3])},
                            {C[1], 0.5 * (C[3] + C[1]), 0.5 * (S[3] + S[1]), 0.5 * (C[0] + C[2]), 0.5 * S[2]},
                            {S[1], 0.5 * (S[3] - S[1]), 0.5 * (C[1] - C[3]), 0.5 * S[2], 0.5 * (C[0] - C[2])}};
    for (int i = 0; i < 25; ++i) h.m[X][i / 5][i % 5] = m[i / 5][i % 5];
  }
  return h;
}

int chunk_count(const Geo& g, const Layout& l) {
  const int64_t per = kChunkSamples / (32 * l.S);
  return (int)((g.n_det * l.tiles + per - 1) / per);
}

// Candidates per launch: at most 4096, and the partial sums (160 B per
// candidate and chunk) stay within 64 MB; the fewest that this gives, 100 for
// the longest data of four detectors, still fill the GPU.
int batch_size(int n_cand, const Geo& g, const Layout& l) {
  const int64_t per = (int64_t)chunk_count(g, l) * kAcc * sizeof(double);
  return (int)std::min<int64_t>(std::min(n_cand, 4096), std::max<int64_t>(64, ((int64_t)64 << 20) / per));
}

size_t consts_bytes(int n_cand) { return ((size_t)n_cand * sizeof(CandConst) + 255) & ~(size_t)255; }

}  // namespace adj

size_t grad_table_bytes(const Geo& g) {
  const adj::Layout l = adj::layout(g);
  return l.x_bytes + l.node_bytes + 256;
}

cudaError_t launch_grad_tables(const Geo& g, const void* const* xh, const int* dtype, void* base, cudaStream_t st) {
  const adj::Layout l = adj::layout(g);
  adj::Series src{};
  for (int X = 0; X < g.n_det; ++X) { src.x[X] = xh[X]; src.dtype[X] = dtype[X]; }
  const int64_t blocks = l.tiles * 32, cap = (int64_t)device_sm_count() * 16;
  adj::k_series_table<<<dim3((unsigned)std::min(cap, (blocks * l.S + 255) / 256), g.n_det), 256, 0, st>>>(
      g, src, l.S, l.tiles, (float2*)base);
  adj::k_block_table<<<dim3((unsigned)std::min(cap, (blocks + 127) / 128), g.n_det), 128, 0, st>>>(
      g, l.S, l.tiles, (float*)((char*)base + l.x_bytes));
  return cudaGetLastError();
}

size_t grad_scratch_bytes(int n_cand, const Geo& g) {
  const adj::Layout l = adj::layout(g);
  const int b = adj::batch_size(n_cand, g, l);
  return adj::consts_bytes(b) + (size_t)b * adj::chunk_count(g, l) * adj::kAcc * sizeof(double) + 256;
}

int grad_launches(int n_cand, const Geo& g) {
  const int b = adj::batch_size(n_cand, g, adj::layout(g));
  return 3 * ((n_cand + b - 1) / b);
}

cudaError_t launch_grad(const Geo& g, const void* tables, const fstat_candidate* cand_dev, int n_cand,
                        void* scratch, float* twoF, float* grad, cudaStream_t st) {
  using namespace adj;
  const Layout l = layout(g);
  const int chunks = chunk_count(g, l), batch = batch_size(n_cand, g, l);
  const Harmonics h = harmonics(g);
  const float2* x = (const float2*)tables;
  const float* nodes = (const float*)((const char*)tables + l.x_bytes);
  CandConst* cc = (CandConst*)scratch;
  double* partial = (double*)((char*)scratch + consts_bytes(batch));
  const float w_step = (float)(g.w_rot * g.dt);
  for (int c0 = 0; c0 < n_cand; c0 += batch) {
    const int n = std::min(batch, n_cand - c0);
    k_cand_consts<<<n, 32, 0, st>>>(g, h, cand_dev + c0, cc);
    const unsigned grid = (unsigned)(((int64_t)n * chunks + kWarps - 1) / kWarps);
    auto run = [&](auto kernel) {
      kernel<<<grid, kWarps * 32, 0, st>>>(g.n_det, l.tiles, x, nodes, w_step, cc, n, chunks, partial);
    };
    switch (l.S) {
      case 32: run(k_moments<32>); break;
      case 16: run(k_moments<16>); break;
      case 8: run(k_moments<8>); break;
      default: run(k_moments<1>); break;
    }
    k_finalize<<<n, kWarps * 32, 0, st>>>(partial, cc, n, chunks, twoF + c0, grad + 4 * (int64_t)c0);
  }
  return cudaGetLastError();
}

}  // namespace fstat
