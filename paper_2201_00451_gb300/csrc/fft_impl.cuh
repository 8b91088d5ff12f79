// Batched Stockham FFT for the template loop: Sec. 3 steps (vi) and (vii).
//
// For one template, Fa and Fb are forward DFTs of length N = n_fft of the
// zero-padded, spindown-corrected series y[j] = G[j] exp(-i 2 pi phi(j)),
// j < n (eqs. Fa, Fb).  N = N1 * N2 is split four-step style:
//
//   pass A (column n1 < N1):  Y[n1][k2] = sum_{n2} y[n1 + N1 n2] W_N2^{n2 k2}
//   pass B (row k2 < N2):     X[k2 + N2 k1] = sum_{n1} Y[n1][k2] W_N1^{n1 (k1 + k2 / N2)}
//
// The four-step twiddle W_N^{n1 k2} is the row's fraction of a bin k2 / N2:
// pass B evaluates its DFT at the shifted frequencies k1 + k2 / N2, which
// only moves the angle of twiddles it applies anyway.
//
// Each column / row FFT runs in shared memory as Stockham radix-16/8/4
// passes (out-of-place index map, in-place buffer, butterflies in
// registers).  Pass A computes the spindown phase on the fly, pass B
// evaluates eq. (Fstat) on the final butterfly outputs and stores 2F in
// ascending frequency (fftshift folded into the index).  Fa and Fb travel
// together as one 16-byte (FP32) / 32-byte (FP64) element, so every index,
// twiddle and phase is computed once for both.
//
// Twiddles are folded into the butterflies: a radix-2 step a +- w b is six
// multiply-adds per complex value, so a twiddled radix-16 butterfly on a pair
// is 384 instructions instead of 120 (twiddles) + 336 (butterfly) and its
// eight distinct factors replace fifteen powers.  FP32 takes each level's
// factor from the hardware sine/cosine of its own exact angle, FP64 from
// tables.  CA / CB, the columns / rows per CTA, are template parameters chosen
// per FFT length by the autotuner.
#pragma once

#include <cuda.h>  // CUtensorMap (encoded through the runtime's driver entry point)
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "fstat_internal.cuh"

namespace fstat {
namespace fft {

template <typename T> struct TwT;
template <> struct TwT<float> { using type = float2; };
template <> struct TwT<double> { using type = double2; };

// ------------------------------------------------------------ radix schedule
// Radix-16 first: the fewest exchanges at 16 points per thread.  V: 0 = a pass
// with two shared buffers where they fit; bits 1 and 2 (the persistent launch,
// fft_fused.cuh) = one buffer that bulk copies fill densely.  The first radix
// is the largest.
__host__ __device__ constexpr int np_of(int L, int) { return L <= 256 ? 2 : (L <= 4096 ? 3 : 4); }
__host__ __device__ constexpr int r_of(int L, int p, int) {
  return L == 32      ? (p == 0 ? 8 : 4)
         : L == 64    ? 8
         : L == 128   ? (p == 0 ? 16 : 8)
         : L == 256   ? 16
         : L == 512   ? 8
         : L == 1024  ? (p == 0 ? 16 : 8)
         : L == 2048  ? (p == 1 ? 8 : 16)
         : L == 8192  ? (p == 2 ? 2 : 16)  // pass A of FP32 plans only
                      : 16;                // 4096
}
__host__ __device__ constexpr int ns_of(int L, int p, int V) {
  return p == 0 ? 1 : ns_of(L, p - 1, V) * r_of(L, p - 1, V);
}
__host__ __device__ constexpr int log2c(int x) { return x <= 1 ? 0 : 1 + log2c(x / 2); }

// product of the schedule's radices (must be L)
__host__ __device__ constexpr int radix_product(int L, int V, int p = 0) {
  return p == np_of(L, V) ? 1 : r_of(L, p, V) * radix_product(L, V, p + 1);
}

template <typename T, int L, int V = 0> struct Shape {
  static constexpr int NP = np_of(L, V);
  static constexpr int R0 = r_of(L, 0, V);        // largest radix, points per thread
  static constexpr int TPC = L / R0;              // threads per column
  static constexpr int PS = log2c(R0);            // shared-memory padding shift
  static constexpr int LP = L + (L >> PS);        // padded column length
  static constexpr int RL = r_of(L, NP - 1, V);   // last radix
  static constexpr int NSL = L / RL;              // span of the last pass
  static constexpr int CA_DEF = TPC >= 128 ? 1 : 128 / TPC;
  static constexpr int CB_MIN = sizeof(T) == 4 ? 2 : 1;
  static constexpr int CB_DEF = TPC >= 128 ? CB_MIN : (128 / TPC > CB_MIN ? 128 / TPC : CB_MIN);
  using PM = typename PairMem<T>::type;
  using TW = typename TwT<T>::type;
  // every pass's radix divides the points per thread (each thread owns whole
  // butterflies of every pass, the last one included) and the radices
  // multiply to L
  static_assert(radix_product(L, V) == L, "radix schedule does not multiply to the length");
  static_assert(R0 % RL == 0 && R0 >= RL, "the last pass's butterflies do not cover the points of a thread");
};

// Shared memory of a persistent pass kernel: NBUF padded buffers of C
// columns; two (prefetch the next tile while transforming this one) when
// they fit, else one.
constexpr size_t kSmemCap = (size_t)220 * 1024;
template <typename T, int L, int C, int V = 0> struct Buf {
  static constexpr size_t ONE = (size_t)C * Shape<T, L, V>::LP * sizeof(typename Shape<T, L, V>::PM);
  static constexpr int NBUF = !(V & 2) && 2 * ONE <= kSmemCap ? 2 : 1;
  static constexpr size_t BYTES = NBUF * ONE;
};

// Peaks mode: a persistent pass-B CTA keeps the band keys of up to
// kPeakBands bands in shared memory across its tiles and flushes them to
// global memory once, when every band spans whole output rows (then each
// band's bins in a tile sit in the same threads in every tile).
constexpr int kPeakBands = 1024;
// pass-B epilogues: store 2F, reduce it (peaks), add it to a shifted row
constexpr int kStore = 0, kPeaks = 1, kAccumulate = 2;
// With one buffer the tile's 2F goes to a region of its own (SEP, when it
// fits) instead of the buffer, so that the next tile's copies can start
// early as in the other epilogues.  Layout: buffers, band keys, 2F tile.
template <typename T, int L, int C, int V> struct PeakSmem {
  static constexpr size_t EXTRA = (size_t)kPeakBands * sizeof(unsigned long long);
  static constexpr bool ACC = Buf<T, L, C, V>::BYTES + EXTRA <= 227 * 1024;
  static constexpr size_t KEYS_END = Buf<T, L, C, V>::BYTES + (ACC ? EXTRA : 0);
  static constexpr size_t SF = (size_t)L * C * sizeof(float);
  static constexpr bool SEP = Buf<T, L, C, V>::NBUF == 1 && KEYS_END + SF <= 227 * 1024;
  static constexpr size_t BYTES = KEYS_END + (SEP ? SF : 0);
};

// 16-byte asynchronous global -> shared copies (completion tracked by
// commit groups; cp.async.wait_group is a hardware wait, not a spin loop).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
template <typename PM> __device__ __forceinline__ void cp_pair(PM* dst, const PM* src) {
  cp_async16(dst, src);
  if constexpr (sizeof(PM) == 32) cp_async16((char*)dst + 16, (const char*)src + 16);
}

// Bulk copies: pass A's staged columns and pass B's tiles (fft_warp.cuh) as
// contiguous blocks, the persistent launch's pass-B tiles as 2D boxes through a
// tensor map (TMA).  One thread issues them, completion is counted in bytes on an
// mbarrier, and every thread waits on the barrier's phase.
// Each wait gives up after kWaitLimit polls (a GPU that stopped delivering
// copies must not hang the kernel): it then records FSTAT_ERR_TIMEOUT and
// the kernel returns.
constexpr int kWaitLimit = 1 << 22;
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, int limit = kWaitLimit) {
  for (int i = 0; i < limit; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
// order this thread's earlier shared-memory accesses before async-proxy writes
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::
          "r"(smem_u32(dst)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// rows per box of a pass-B tile load (the box height limit is 256)
constexpr int kTmaRows = 256;
// contiguous bulk copy global -> shared (16-byte aligned addresses, size a
// multiple of 16), completion counted in bytes on the mbarrier
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// load with acquire semantics at GPU scope (a counter another CTA releases)
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// order this thread's earlier generic-proxy accesses to global memory (and
// what it acquired) before its later async-proxy (bulk copy) accesses
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;\n" ::: "memory");
}

__device__ __forceinline__ int pad_idx(int pos, int ps) { return pos + (pos >> ps); }

template <typename TW> __device__ __forceinline__ TW tw_ld(const TW* p) { return __ldg(p); }

// (cos, sin) of 2 pi x for x in turns, |x| <= 1/2: the hardware sine/cosine
// (accurate to ~4e-7 absolute on [-pi, pi]) brought to unit length.  The
// hardware's pair is short by ~7e-8 on average, which a transform's nine factors
// per sample add up: 2F came out 1.3e-6 low throughout at 2^22 points.
__device__ __forceinline__ void turn_sincos(float x, float* s, float* c) {
  float sv, cv;
  __sincosf(6.28318530717958647692f * x, &sv, &cv);
  const float h = 0.5f * __fmaf_rn(-sv, sv, __fmaf_rn(-cv, cv, 1.f));
  *s = __fmaf_rn(sv, h, sv);
  *c = __fmaf_rn(cv, h, cv);
}

// ------------------------------------------------------------- small DFTs
// Decimation in time, radix-2 steps: level M = 2, 4 .. R combines the two
// transforms of length M/2 of a residue class of inputs, E and O, into
// y_m = E_m + w_M^m O_m and y_{m + M/2} = E_m - w_M^m O_m with
// w_M^m = exp(-2 pi i R theta / M) exp(-2 pi i m / M), theta being the
// butterfly's twiddle angle in turns (input s carries exp(-2 pi i s theta)).
// The second half of m is the first times -i, so level M has max(M / 4, 1)
// distinct factors.
__host__ __device__ constexpr int tw_off(int M) { return M / 4; }  // 2: 0, 4: 1, 8: 2, 16: 4
// cos, sin of 2 pi j / 16, j = 0..3
__host__ __device__ constexpr double cos16(int j) {
  return j == 0 ? 1.0 : j == 1 ? 0.92387953251128675613 : j == 2 ? 0.70710678118654752440 : 0.38268343236508977173;
}
__host__ __device__ constexpr double sin16(int j) { return j == 0 ? 0.0 : cos16(4 - j); }

template <typename T, int R> struct Twiddles {
  static constexpr int N = R / 2;  // factors over all levels
  T c[N], s[N];
  // the level's other factors from its first one
  template <int M> __device__ __forceinline__ void spread() {
    constexpr int o = tw_off(M);
#pragma unroll
    for (int m = 1; m < M / 4; ++m) {
      const T cm = (T)cos16(m * 16 / M), sm = (T)-sin16(m * 16 / M);
      c[o + m] = fmadd(c[o], cm, -(s[o] * sm));
      s[o + m] = fmadd(c[o], sm, s[o] * cm);
    }
  }
  template <int M> __device__ __forceinline__ void square() {  // level M from level 2M
    const T x = c[tw_off(2 * M)], y = s[tw_off(2 * M)];
    c[tw_off(M)] = fmadd(x, x, -(y * y));
    s[tw_off(M)] = (x + x) * y;
    spread<M>();
  }
  template <int M> __device__ __forceinline__ void squares() {
    square<M>();
    if constexpr (M > 2) squares<M / 2>();
  }
  // every other level by its angle, the one below it by squaring: the rounding
  // of a factor doubles once only
  template <int M> __device__ __forceinline__ void level(float theta) {
    turn_sincos(-theta * (float)(R / M), &s[tw_off(M)], &c[tw_off(M)]);
    spread<M>();
    if constexpr (M > 2) square<M / 2>();
    if constexpr (M > 4) level<M / 4>(theta);
  }
  // theta in [0, 1/R)
  __device__ __forceinline__ explicit Twiddles(float theta) { level<R>(theta); }
  // from the angle's own factor exp(-2 pi i theta)
  __device__ __forceinline__ Twiddles(T cw, T sw) {
    c[tw_off(R)] = cw;
    s[tw_off(R)] = sw;
    spread<R>();
    if constexpr (R > 2) squares<R / 2>();
  }
};

// (a, b) <- (a + w b, a - w b), the difference as 2 a - (a + w b)
template <typename T> __device__ __forceinline__ void bfly(Pair<T>& a, Pair<T>& b, T c, T s) {
  const Pair<T> t{fmadd(-s, b.ai, fmadd(c, b.ar, a.ar)), fmadd(s, b.ar, fmadd(c, b.ai, a.ai)),
                  fmadd(-s, b.bi, fmadd(c, b.br, a.br)), fmadd(s, b.br, fmadd(c, b.bi, a.bi))};
  b = {fmadd((T)2, a.ar, -t.ar), fmadd((T)2, a.ai, -t.ai), fmadd((T)2, a.br, -t.br), fmadd((T)2, a.bi, -t.bi)};
  a = t;
}
template <typename T> __device__ __forceinline__ void bfly_1(Pair<T>& a, Pair<T>& b) {
  const Pair<T> t = padd(a, b);
  b = psub(a, b);
  a = t;
}

// Level M of a radix-R butterfly in place: residue r of the inputs mod R/M
// holds its length-M/2 transforms at r and r + R/M; transform output m sits
// at (m bit-reversed) R/M.  PLAIN: theta = 0, constant factors; HALF (PLAIN
// only): inputs R/2 .. R-1 are zero.
__host__ __device__ constexpr int bit_rev(int m, int bits) {
  int r = 0;
  for (int i = 0; i < bits; ++i) r |= ((m >> i) & 1) << (bits - 1 - i);
  return r;
}
template <typename T, int R, int M, bool PLAIN, bool HALF>
__device__ __forceinline__ void dit_level(Pair<T>* x, const Twiddles<T, R>* w) {
  constexpr int G = R / M, H = M / 2;  // residues, half length
#pragma unroll
  for (int m = 0; m < H; ++m) {
    const int base = bit_rev(m, log2c(H)) * (2 * G);
#pragma unroll
    for (int r = 0; r < G; ++r) {
      Pair<T>&a = x[base + r], &b = x[base + r + G];
      if constexpr (HALF && M == 2) {
        b = a;
      } else {
        // the second quarter of the circle: times -i
        const bool q = M >= 4 && m >= M / 4;
        const int k = q ? m - M / 4 : m;
        if constexpr (PLAIN) {
          if (k == 0) {
            if (q) b = pmul_mi(b);
            bfly_1(a, b);
          } else {
            const T c = (T)cos16(k * 16 / M), s = (T)-sin16(k * 16 / M);
            if (q) bfly(a, b, s, -c);
            else bfly(a, b, c, s);
          }
        } else {
          const T c = w->c[tw_off(M) + k], s = w->s[tw_off(M) + k];
          if (q) bfly(a, b, s, -c);
          else bfly(a, b, c, s);
        }
      }
    }
  }
  if constexpr (M < R) dit_level<T, R, 2 * M, PLAIN, HALF>(x, w);
}
template <typename T, int R, bool PLAIN, bool HALF>
__device__ __forceinline__ void dit(Pair<T>* x, const Twiddles<T, R>* w) {
  dit_level<T, R, 2, PLAIN, HALF>(x, w);
  Pair<T> t[R];
#pragma unroll
  for (int m = 0; m < R; ++m) t[m] = x[bit_rev(m, log2c(R))];
#pragma unroll
  for (int m = 0; m < R; ++m) x[m] = t[m];
}
// y_m = sum_s x_s exp(-2 pi i m s / R) in place
template <typename T, int R> __device__ __forceinline__ void dft(Pair<T>* x) { dit<T, R, true, false>(x, nullptr); }
// the same when x[R/2 .. R) is zero (and unread): the first pass of pass A
// when zero padding leaves every column at most L/2 samples
template <typename T, int R> __device__ __forceinline__ void dft_half(Pair<T>* x) { dit<T, R, true, true>(x, nullptr); }
// y_m = sum_s x_s exp(-2 pi i s (theta + m / R))
template <typename T, int R> __device__ __forceinline__ void dft_tw(Pair<T>* x, const Twiddles<T, R>& w) {
  dit<T, R, false, false>(x, &w);
}

// A row's fraction of a bin, k2 / N2, added to every output frequency of
// pass B (see the top).  FP32: the fraction itself (exact).  FP64: its
// factor for each Stockham pass, exp(-2 pi i (k2 / N2) / (NS R)), from the
// tables behind the length's roots (tables.cu).
template <typename T> struct Twist;
template <> struct Twist<float> {
  float frac;
  __device__ __forceinline__ Twist(const float2*, int, int k2, int n2) : frac((float)k2 / (float)n2) {}  // exact
  __device__ __forceinline__ explicit Twist(float f = 0.f) : frac(f) {}
};
template <> struct Twist<double> {
  const double2* row;
  int n2;
  __device__ __forceinline__ Twist(const double2* twL, int L, int k2, int n2_) : row(twL + L + k2), n2(n2_) {}
  __device__ __forceinline__ Twist() : row(nullptr), n2(0) {}
};

// Twiddles of butterfly b of Stockham pass P: angle ((b mod NS) + twist) / (NS R)
template <int L, int P, int V, bool TWIST>
__device__ __forceinline__ Twiddles<float, r_of(L, P, V)> pass_twiddles(int b, const float2*, const Twist<float>& tw) {
  constexpr int R = r_of(L, P, V), NS = ns_of(L, P, V);
  // at most 9 + 13 bits: exact
  return Twiddles<float, R>(((float)(b & (NS - 1)) + (TWIST ? tw.frac : 0.f)) * (1.f / (float)(NS * R)));
}
template <int L, int P, int V, bool TWIST>
__device__ __forceinline__ Twiddles<double, r_of(L, P, V)> pass_twiddles(int b, const double2* __restrict__ twL,
                                                                         const Twist<double>& tw) {
  constexpr int R = r_of(L, P, V), NS = ns_of(L, P, V);
  double2 w = {1.0, 0.0};
  if constexpr (NS > 1) w = tw_ld(twL + (b & (NS - 1)) * (L / (NS * R)));
  if constexpr (TWIST) {
    const double2 t = tw_ld(tw.row + P * tw.n2);
    w = NS > 1 ? double2{w.x * t.x - w.y * t.y, w.x * t.y + w.y * t.x} : t;
  }
  return Twiddles<double, R>(w.x, w.y);
}

// --------------------------------------------------------- Stockham passes
// After pass 0 (done by the caller, in registers), store it and run passes
// 1..NP-1.  On return v holds the last pass's outputs: butterfly
// b = t + q * TPC, output index b + s * NSL in v[q * RL + s].
// Shared-memory address of logical position pos is pad(pos) * STRIDE.
// at_free() runs once the last pass has read the buffer into registers (all
// threads past the barrier that follows): the buffer is free from there on.
struct NoOp {
  __device__ __forceinline__ void operator()() const {}
};
template <typename T, int L, int V, int STRIDE, int P, bool TWIST, typename F = NoOp>
__device__ __forceinline__ void passes(Pair<T>* v, typename PairMem<T>::type* buf, int t,
                                       const typename TwT<T>::type* __restrict__ twL, const Twist<T>& twist,
                                       const F& at_free = F()) {
  using S = Shape<T, L, V>;
  constexpr int R = r_of(L, P, V);
  constexpr int NS = ns_of(L, P, V);
  constexpr int NB = S::R0 / R;  // butterflies per thread
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int b = t + q * S::TPC;
#pragma unroll
    for (int s = 0; s < R; ++s) v[q * R + s] = pload(buf + pad_idx(b + s * (L / R), S::PS) * STRIDE);
  }
  __syncthreads();
  if constexpr (P + 1 == S::NP) at_free();
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int b = t + q * S::TPC;
    dft_tw<T, R>(v + q * R, pass_twiddles<L, P, V, TWIST>(b, twL, twist));
  }
  if constexpr (P + 1 < S::NP) {
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int b = t + q * S::TPC;
      const int base = (b / NS) * NS * R + (b & (NS - 1));
#pragma unroll
      for (int s = 0; s < R; ++s) pstore(buf + pad_idx(base + s * NS, S::PS) * STRIDE, v[q * R + s]);
    }
    __syncthreads();
    passes<T, L, V, STRIDE, P + 1, TWIST, F>(v, buf, t, twL, twist, at_free);
  }
}

// store pass-0 outputs (one radix-R0 butterfly per thread, Ns = 1)
template <typename T, int L, int V, int STRIDE>
__device__ __forceinline__ void store_pass0(const Pair<T>* v, typename PairMem<T>::type* buf, int t) {
  using S = Shape<T, L, V>;
#pragma unroll
  for (int s = 0; s < S::R0; ++s) pstore(buf + pad_idx(t * S::R0 + s, S::PS) * STRIDE, v[s]);
  __syncthreads();
}

// ----------------------------------------------------- spindown phase
// e^{-i 2 pi phi} at the samples of one first-pass butterfly, x_s = x0 + s D
// (TmplCoef).
//
// FP32: the polynomial and its first two differences are evaluated once per
// butterfly, the samples follow by differences: three integer adds, a conversion
// and a sine/cosine each instead of a double-float cubic.  Double-float Horner with error-free products and sums (explicitly
// rounded, so the compiler cannot contract them), then phases modulo a cycle
// in units of 2^-32, whose adds are exact.  The units' rounding grows with the
// distance from the sample that the differences start at: at most 1.2e-8
// cycles within 8 samples of it, so they start at s = 0 when only the lower
// half holds data (HALF) and in the middle otherwise (inside the data, where
// the excursion limit of spin_in_range holds).
template <int N> __device__ __forceinline__ int poly_turns(const float (*c)[2], float x) {
  float h = c[N][0], l = c[N][1];
#pragma unroll
  for (int q = N - 1; q >= 0; --q) {
    const float p = __fmul_rn(h, x);
    float e = fmaf(h, x, -p);
    e = fmaf(l, x, e);
    const float S = __fadd_rn(p, c[q][0]);
    const float bb = __fsub_rn(S, p);
    float err = __fadd_rn(__fsub_rn(p, __fsub_rn(S, bb)), __fsub_rn(c[q][0], bb));
    err = __fadd_rn(err, __fadd_rn(e, c[q][1]));
    h = __fadd_rn(S, err);
    l = __fsub_rn(err, __fsub_rn(h, S));
  }
  const float f = __fsub_rn(h, rintf(h));  // exact
  // (f = 1/2 saturates one unit short)
  return (int)((unsigned)__float2int_rn(__fmul_rn(f, 4294967296.f)) + (unsigned)__float2int_rn(__fmul_rn(l, 4294967296.f)));
}
template <typename T, int R, bool HALF> struct Spin;
template <int R, bool HALF> struct Spin<float, R, HALF> {
  static constexpr int S0 = HALF ? 0 : R / 2;
  unsigned ph[R];
  // x0: sample offset of s = 0 from J; D: spacing
  __device__ __forceinline__ Spin(const TmplCoef& c, int x0, int D) {
    const float x = (float)(x0 + S0 * D);
    const unsigned p = poly_turns<3>(c.phi, x), d1 = poly_turns<2>(c.d1, x), d2 = poly_turns<1>(c.d2, x), d3 = c.d3;
    unsigned f = p, a = d1, b = d2;
#pragma unroll
    for (int s = S0; s < (HALF ? R / 2 : R); ++s) {
      ph[s] = f;
      f += a;
      a += b;
      b += d3;
    }
    f = p; a = d1; b = d2;
#pragma unroll
    for (int s = S0 - 1; s >= 0; --s) {
      b -= d3;
      a -= b;
      f -= a;
      ph[s] = f;
    }
  }
  __device__ __forceinline__ void rot(int s, float* cs, float* sn) {
    float sv, cv;
    __sincosf((float)(int)ph[s] * (float)(6.28318530717958647692 / 4294967296.0), &sv, &cv);
    *cs = cv;
    *sn = -sv;
  }
};
// FP64: the polynomial at every sample, and for columns of 256 points or more its
// factor as a 256th root of unity (of the column's own table tw) times a turn of at
// most 1/512, whose Taylor series are cut at 1e-17.  Like sincospi at every sample it
// leaves 4e-17 to 4e-15 (excursions of 0.005 to 17 cycles); the differences as
// factors, r <- r m, m <- m k, .., leave 1e-15 to 4e-14.  Eight templates, us, with
// those, with sincospi and so: 200 001 samples at 2^18 577, 602, 550; 500 001 at 2^20
// 2274, 2380, 2254; 4 000 001 at 2^22 10749, 11940, 10890.
template <int R, bool HALF> struct Spin<double, R, HALF> {
  const TmplCoef& c;
  int x0, D;
  __device__ __forceinline__ Spin(const TmplCoef& c_, int x0_, int D_) : c(c_), x0(x0_), D(D_) {}
  template <int L> __device__ __forceinline__ void rot(int s, const double2* __restrict__ tw, double* cs, double* sn) {
    const double x = (double)(x0 + s * D);
    const double ph = ((c.p[3] * x + c.p[2]) * x + c.p[1]) * x + c.p[0];
    if constexpr (L < 256) {
      sincospi(-2.0 * (ph - rint(ph)), sn, cs);
    } else {
      constexpr double kRint = 6755399441055744.0;  // 1.5 2^52: adds an integer to the low word
      constexpr double p = 6.283185307179586, p2 = p * p;
      const double t = fma(ph, 256.0, kRint);
      const double r = fma(t - kRint, -1.0 / 256.0, ph), r2 = r * r;  // exact
      const double2 w = __ldg(tw + (__double2loint(t) & 255) * (L / 256));
      const double sr = r * fma(r2, fma(r2, p * p2 * p2 / 120.0, -p * p2 / 6.0), p);
      const double e = r2 * fma(r2, fma(r2, -p2 * p2 * p2 / 720.0, p2 * p2 / 24.0), -p2 / 2.0);  // cosine - 1
      *cs = fma(w.x, e, fma(w.y, sr, w.x));
      *sn = fma(w.y, e, fma(-w.x, sr, w.y));
    }
  }
};

// ------------------------------------------------------------- pass A
// One tile = CA columns, whose samples were copied to `buf`: at padded natural
// positions by cp.async, or (V bit 2) in G's order by bulk copies.
template <typename T, int L, int CA, int V, typename F = NoOp>
__device__ __forceinline__ void pass_a_tile(int tile, typename PairMem<T>::type* buf, int c, int t,
                                            const typename PairMem<T>::type* __restrict__ G, GCol gc,
                                            int n, int n1, const typename TwT<T>::type* __restrict__ twL,
                                            const TmplCoef& tc, typename PairMem<T>::type* __restrict__ Z,
                                            const F& at_free = F()) {
  using S = Shape<T, L, V>;
  using PM = typename PairMem<T>::type;
  constexpr bool kDense = (V & 4) != 0;
  const int col = tile * CA + c;
  Pair<T> v[S::R0];
  const int x0 = col + n1 * t - tc.J, D = n1 * S::TPC;
  // zero padding to at least twice the data (n <= n1 L / 2): no column has
  // a sample at n2 >= L/2, the upper half of every first butterfly is zero
  auto load = [&](auto half) {
    constexpr bool HALF = decltype(half)::value;
    Spin<T, S::R0, HALF> spin(tc, x0, D);
#pragma unroll
    for (int s = 0; s < (HALF ? S::R0 / 2 : S::R0); ++s) {
      const int n2 = t + s * S::TPC;
      if (col + n1 * n2 < n) {
        T cs, sn;
        if constexpr (sizeof(T) == 8) spin.template rot<L>(s, twL, &cs, &sn);
        else spin.rot(s, &cs, &sn);
        v[s] = pmul(pload(buf + (kDense ? gc.at(n2) : pad_idx(n2, S::PS))), cs, sn);
      } else {
        v[s] = pzero<T>();
      }
    }
  };
  const bool half = (int64_t)n1 * (L / 2) >= (int64_t)n;
  if (half) load(std::true_type());
  else load(std::false_type());
  __syncthreads();  // the staged column is overwritten below
  if (half) dft_half<T, S::R0>(v);
  else dft<T, S::R0>(v);
  store_pass0<T, L, V, 1>(v, buf, t);
  passes<T, L, V, 1, 1, false, F>(v, buf, t, twL, Twist<T>(), at_free);

  PM* zrow = Z + (int64_t)col * L;
  constexpr int NB = S::R0 / S::RL;
#pragma unroll
  for (int q = 0; q < NB; ++q)
#pragma unroll
    for (int s = 0; s < S::RL; ++s) pstore(zrow + t + q * S::TPC + s * S::NSL, v[q * S::RL + s]);
}

// The CTA transforms tiles b, b + grid, ...; the next tile's samples are
// copied asynchronously into the other buffer while the current one is
// transformed in place, or, with one buffer, into that buffer as soon as the
// last Stockham pass has read it (under that pass and the epilogue).
template <typename T, int L, int CA, int V>
__global__ void __launch_bounds__(CA * Shape<T, L, V>::TPC)
k_pass_a(const typename PairMem<T>::type* __restrict__ G, GCol gc, int n, int n1,
         const typename TwT<T>::type* __restrict__ twL, const TmplCoef* __restrict__ coefp,
         typename PairMem<T>::type* __restrict__ Z) {
  using S = Shape<T, L, V>;
  using B = Buf<T, L, CA, V>;
  using PM = typename PairMem<T>::type;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  PM* smem = reinterpret_cast<PM*>(smem_raw);
  const int c = threadIdx.x / S::TPC;
  const int t = threadIdx.x % S::TPC;
  const TmplCoef tc = *coefp;
  {
    const int n_tiles = n1 / CA;
    auto stage = [&](int it) { return smem + (B::NBUF == 2 ? (it & 1) : 0) * (CA * S::LP) + c * S::LP; };
    auto prefetch = [&](int tile, PM* dst) {
      const int col = tile * CA + c;
      const PM* gcol = G + (int64_t)col * gc.lc;
#pragma unroll
      for (int s = 0; s < S::R0; ++s) {
        const int n2 = t + s * S::TPC;
        if (col + n1 * n2 < n) cp_pair(dst + pad_idx(n2, S::PS), gcol + gc.at(n2));
      }
    };
    int tile = blockIdx.x;
    if (tile < n_tiles) prefetch(tile, stage(0));
    cp_async_commit();
    for (int it = 0; tile < n_tiles; ++it, tile += gridDim.x) {
      PM* buf = stage(it);
      const int next = tile + gridDim.x;
      if constexpr (B::NBUF == 2) {
        if (next < n_tiles) prefetch(next, stage(it + 1));
        cp_async_commit();
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncthreads();
      if constexpr (B::NBUF == 2) {
        pass_a_tile<T, L, CA, V>(tile, buf, c, t, G, gc, n, n1, twL, tc, Z);
        __syncthreads();  // this buffer is the prefetch target two tiles on
      } else {
        // no barrier after the tile: it stopped reading the buffer before
        // the barrier at which the next tile's copies were issued
        pass_a_tile<T, L, CA, V>(tile, buf, c, t, G, gc, n, n1, twL, tc, Z, [&] {
          if (next < n_tiles) prefetch(next, buf);
          cp_async_commit();
        });
      }
    }
  }
}

// ------------------------------------------------------------- pass B
// Peaks epilogue.  sf holds the tile's 2F as [r][c] (r = ascending row of
// the output, c = column of the CTA), so bin m = k2_0 + c + n2 r increases
// with the flat index f = r CB + c.  Each thread takes E consecutive
// values.  Band boundaries fall on multiples of a power of two in f (every
// band is 2^log2_band consecutive bins and k2_0 is a multiple of CB), so
// when no thread's run straddles one, the lanes of one band form an
// aligned power-of-two group: a masked butterfly gives the group maximum
// and the group's first lane alone updates the band key.
template <int CB, int E>
__device__ __forceinline__ void peak_epilogue(const float* sf, int k2_0, int n2, const PeakArgs& pk,
                                              unsigned long long* ks) {
  constexpr unsigned FULL = 0xffffffffu;
  const int f0 = threadIdx.x * E;
  float v[E];
  if constexpr (E % 4 == 0) {
#pragma unroll
    for (int j = 0; j < E; j += 4) {
      const float4 q = *reinterpret_cast<const float4*>(sf + f0 + j);
      v[j] = q.x; v[j + 1] = q.y; v[j + 2] = q.z; v[j + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < E; ++j) v[j] = sf[f0 + j];
  }
  auto bin = [&](int f) { return (unsigned)(k2_0 + (f & (CB - 1)) + n2 * (f / CB)); };
  float best = v[0];
  int jb = 0;
#pragma unroll
  for (int j = 1; j < E; ++j)
    if (v[j] > best) { best = v[j]; jb = j; }
  const int lane = threadIdx.x & 31;
  if (pk.count && __any_sync(FULL, best > pk.thr)) {
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const bool hit = v[j] > pk.thr;
      const unsigned bal = __ballot_sync(FULL, hit);
      if (!bal) continue;
      const int leader = __ffs(bal) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(pk.count, (unsigned long long)__popc(bal));
      base = __shfl_sync(FULL, base, leader);
      if (hit) {
        const unsigned long long idx = base + __popc(bal & ((1u << lane) - 1u));
        if (idx < (unsigned long long)pk.cap) {
          fstat_peak e;
          e.tmpl = pk.tmpl;
          e.bin = (int32_t)bin(f0 + j);
          e.twoF = v[j];
          pk.peaks[idx] = e;
        }
      }
    }
  }
  if (pk.band_key) {
    // shared keys of this CTA when it accumulates, else the global row
    unsigned long long* keys = ks ? ks : pk.band_key;
    const int lb = pk.log2_band;
    // a band is a run of 2^lp consecutive f: CB W / n2 when it spans whole
    // rows, else the CTA's part of one row (at most CB values)
    constexpr int LCB = log2c(CB), LE = log2c(E);
    const int ln2 = 31 - __clz(n2);
    const int lp = lb >= ln2 ? LCB + lb - ln2 : (lb < LCB ? lb : LCB);
    // In shared keys, a band within one warp's values has a single writer
    // (the same lane in every tile), so a plain update suffices.
    const bool excl = ks != nullptr && lp <= LE + 5;
    auto update = [&](unsigned b, unsigned long long key) {
      if (excl) {
        if (key > keys[b]) keys[b] = key;
      } else {
        atomicMax(keys + b, key);
      }
    };
    if (lp >= LE) {
      // the run lies in one band; lanes of a band form an aligned group
      const unsigned band = bin(f0) >> lb;
      unsigned long long key = band_key(best, bin(f0 + jb));
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long ok = __shfl_xor_sync(FULL, key, o);
        if (o < (1 << (lp - LE)) && ok > key) key = ok;
      }
      if ((lane & ((1 << (lp - LE < 5 ? lp - LE : 5)) - 1)) == 0) update(band, key);
    } else {
      // runs of P values, each one band, inside this thread's values
      const int pm = (1 << lp) - 1;
      float bv = v[0];
      int bj = 0;
#pragma unroll
      for (int j = 1; j < E; ++j) {
        if ((j & pm) == 0) {
          update(bin(f0 + bj) >> lb, band_key(bv, bin(f0 + bj)));
          bv = v[j]; bj = j;
        } else if (v[j] > bv) {
          bv = v[j]; bj = j;
        }
      }
      update(bin(f0 + bj) >> lb, band_key(bv, bin(f0 + bj)));
    }
  }
}

template <typename T, int L, int CB, int V, int MODE, typename F = NoOp>
__device__ __forceinline__ void pass_b_tile(int tile, typename PairMem<T>::type* buf, int c, int t,
                                            int n2, const typename TwT<T>::type* __restrict__ twL, T kA, T kB, T kC,
                                            float* __restrict__ out, const PeakArgs& pk,
                                            unsigned long long* ks, float* sf_sep, const F& at_free = F()) {
  using S = Shape<T, L, V>;
  const int k2 = tile * CB + c;
  constexpr int NB = S::R0 / S::RL;
  // accumulate mode: the running sums this thread adds to, loaded before
  // the transform so their latency hides under it
  float acc[MODE == kAccumulate ? S::R0 : 1];
  if (MODE == kAccumulate && !pk.first) {
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int s = 0; s < S::RL; ++s) {
        const int r = (t + q * S::TPC + s * S::NSL + L / 2) & (L - 1);
        const int mg = k2 + n2 * r - pk.shift;
        acc[q * S::RL + s] = (unsigned)mg < (unsigned)(n2 * L) ? out[mg] : 0.f;
      }
  }
  Pair<T> v[S::R0];
  // staged rows: padded positions (per-thread copies) or dense rows (TMA boxes)
  constexpr bool kDense = (V & 4) != 0;
#pragma unroll
  for (int s = 0; s < S::R0; ++s)
    v[s] = pload(buf + (kDense ? t + s * S::TPC : pad_idx(t + s * S::TPC, S::PS)) * CB);
  __syncthreads();  // the staged rows are overwritten below
  const Twist<T> twist(twL, L, k2, n2);
  dft_tw<T, S::R0>(v, pass_twiddles<L, 0, V, true>(0, twL, twist));
  store_pass0<T, L, V, CB>(v, buf, t);
  passes<T, L, V, CB, 1, true, F>(v, buf, t, twL, twist, at_free);

  // peaks epilogue: the tile's 2F in its own region, or in the CTA's stage
  // once every thread is done with it as the exchange buffer
  float* sf = sf_sep ? sf_sep : reinterpret_cast<float*>(buf - c);
  if constexpr (MODE == kPeaks) {
    if (!sf_sep) __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int b = t + q * S::TPC;
#pragma unroll
    for (int s = 0; s < S::RL; ++s) {
      const Pair<T>& x = v[q * S::RL + s];
      const int k1 = b + s * S::NSL;
      const T tf = two_f(x, kA, kB, kC);
      const int r = (k1 + L / 2) & (L - 1);
      if constexpr (MODE == kPeaks) {
        sf[r * CB + c] = (float)tf;
      } else if constexpr (MODE == kAccumulate) {
        // semi-coherent sum: this segment's bin m adds to global bin m - shift
        const int mg = k2 + n2 * r - pk.shift;
        const bool in = (unsigned)mg < (unsigned)(n2 * L);
        if (pk.first) out[mg & (n2 * L - 1)] = in ? (float)tf : 0.f;  // the bins that wrap are the ones no bin reaches
        else if (in) out[mg] = acc[q * S::RL + s] + (float)tf;
      } else {
        __stcs(out + k2 + n2 * r, (float)tf);  // streaming store: keep G and Z in L2
      }
    }
  }
  if constexpr (MODE == kPeaks) {
    __syncthreads();
    peak_epilogue<CB, L * CB / (CB * S::TPC)>(sf, tile * CB, n2, pk, ks);
  }
}

template <typename T, int L, int CB, int V, int MODE>
__global__ void __launch_bounds__(CB * Shape<T, L, V>::TPC)
k_pass_b(const typename PairMem<T>::type* __restrict__ Z, int n2,
         const typename TwT<T>::type* __restrict__ twL, const SkyConst* __restrict__ sky,
         float* __restrict__ out, const PeakArgs pk) {
  using S = Shape<T, L, V>;
  using B = Buf<T, L, CB, V>;
  using PM = typename PairMem<T>::type;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  PM* smem = reinterpret_cast<PM*>(smem_raw);
  const int c = threadIdx.x % CB;
  const int t = threadIdx.x / CB;
  T kA, kB, kC;
  if constexpr (sizeof(T) == 4) { kA = sky->kAf; kB = sky->kBf; kC = sky->kCf; }
  else { kA = sky->kA; kB = sky->kB; kC = sky->kC; }
  // peaks mode with whole-row bands: this CTA's band keys in shared memory
  unsigned long long* ks = nullptr;
  float* sf_sep = nullptr;
  if constexpr (MODE == kPeaks && PeakSmem<T, L, CB, V>::SEP)
    sf_sep = reinterpret_cast<float*>(smem_raw + PeakSmem<T, L, CB, V>::KEYS_END);
  int n_bands = 0;
  if constexpr (MODE == kPeaks && PeakSmem<T, L, CB, V>::ACC) {
    if (pk.band_key && pk.log2_band >= 31 - __clz(n2)) {
      n_bands = (L * n2) >> pk.log2_band;
      if (n_bands <= kPeakBands) {
        ks = reinterpret_cast<unsigned long long*>(smem_raw + Buf<T, L, CB, V>::BYTES);
        for (int b = threadIdx.x; b < n_bands; b += blockDim.x) ks[b] = 0ull;
        // visible to the epilogue after the tile loop's first barrier
      }
    }
  }
  const int n_tiles = n2 / CB;
  auto stage = [&](int it) { return smem + (B::NBUF == 2 ? (it & 1) : 0) * (CB * S::LP) + c; };
  auto prefetch = [&](int tile, PM* dst) {
    const int k2 = tile * CB + c;
#pragma unroll
    for (int s = 0; s < S::R0; ++s) {
      const int n1 = t + s * S::TPC;
      cp_pair(dst + pad_idx(n1, S::PS) * CB, Z + (int64_t)n1 * n2 + k2);
    }
  };
  // with one buffer (and no peaks epilogue that reuses it) the next
  // tile's copies start as soon as the last Stockham pass has read it
  constexpr bool kEarly = B::NBUF == 1 && (MODE != kPeaks || PeakSmem<T, L, CB, V>::SEP);
  int tile = blockIdx.x;
  if constexpr (B::NBUF == 2 || kEarly) {
    if (tile < n_tiles) prefetch(tile, stage(0));
    cp_async_commit();
  }
  for (int it = 0; tile < n_tiles; ++it, tile += gridDim.x) {
    PM* buf = stage(it);
    const int next = tile + gridDim.x;
    if constexpr (B::NBUF == 2) {
      if (next < n_tiles) prefetch(next, stage(it + 1));
      cp_async_commit();
      cp_async_wait<1>();
    } else if constexpr (kEarly) {
      cp_async_wait<0>();
    } else {
      prefetch(tile, buf);
      cp_async_commit();
      cp_async_wait<0>();
    }
    __syncthreads();
    if constexpr (kEarly) {
      // no barrier after the tile: it stopped reading the buffer before
      // the barrier at which the next tile's copies were issued
      pass_b_tile<T, L, CB, V, MODE>(tile, buf, c, t, n2, twL, kA, kB, kC, out, pk, ks, sf_sep, [&] {
        if (next < n_tiles) prefetch(next, buf);
        cp_async_commit();
      });
    } else {
      pass_b_tile<T, L, CB, V, MODE>(tile, buf, c, t, n2, twL, kA, kB, kC, out, pk, ks, sf_sep);
      __syncthreads();  // this buffer is the prefetch target two tiles on
    }
  }
  if constexpr (MODE == kPeaks) {
    if (ks) {
      if constexpr (kEarly) __syncthreads();  // else the loop ended on one
      // every tile's keys are in
      for (int b = threadIdx.x; b < n_bands; b += blockDim.x)
        if (ks[b]) atomicMax(pk.band_key + b, ks[b]);
    }
  }
}

// ------------------------------------------------------------- launchers
// Resident CTAs of a persistent kernel: SM count x CTAs per SM, asked of the
// runtime once per kernel, device and shared-memory size.  (One kernel type
// may stand for several instantiations: the key is the function itself.)
cudaError_t resident_ctas(const void* kernel, int threads, size_t smem, int* out, int* out_per_sm);
template <typename K>
cudaError_t resident_ctas(K* kernel, int threads, size_t smem, int* out, int* out_per_sm) {
  return resident_ctas(reinterpret_cast<const void*>(kernel), threads, smem, out, out_per_sm);
}

// Persistent grid: every resident CTA, or at most `res` per SM (res > 0),
// which leaves room on each SM for a CTA of the other pass of a
// neighbouring template running on another stream.
inline int persistent_grid(int tiles, int ctas, int per_sm, int res) {
  int g = ctas;
  if (res > 0 && res < per_sm) g = ctas / per_sm * res;
  return tiles < g ? tiles : g;
}

// Dynamic shared memory a CTA may opt into (227 KB on sm_100 / sm_103).
constexpr size_t kSmemOptIn = (size_t)227 * 1024;

template <typename T, int L, int CA, int V>
cudaError_t run_a(const void* G, GCol gc, int64_t n, int n1, const void* twA, const TmplCoef* coef, void* Z,
                  cudaStream_t st, int res) {
  using S = Shape<T, L, V>;
  using PM = typename S::PM;
  constexpr size_t smem = Buf<T, L, CA, V>::BYTES;
  constexpr int threads = CA * S::TPC;
  int ctas = 0, per_sm = 0;
  const cudaError_t e = resident_ctas(k_pass_a<T, L, CA, V>, threads, smem, &ctas, &per_sm);
  if (e != cudaSuccess) return e;
  if (n1 % CA) return cudaErrorInvalidConfiguration;
  k_pass_a<T, L, CA, V><<<persistent_grid(n1 / CA, ctas, per_sm, res), threads, smem, st>>>(
      (const PM*)G, gc, (int)n, n1, (const typename S::TW*)twA, coef, (PM*)Z);
  return cudaGetLastError();
}

// cuTensorMapEncodeTiled, through the runtime's driver entry point (the
// library does not link the driver API).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(f);
  }
  return fn;
}

// Tensor map of pass B's input (FP32 pairs): L rows of n2 pairs, i.e. rows
// of 4 n2 floats at a pitch of 16 n2 bytes; a box is CB pairs (16 CB bytes,
// a multiple of 16) by min(L, kTmaRows) rows.  Box x coordinates are
// multiples of 4 CB floats, so every copy starts on a 16-byte boundary.
inline cudaError_t z_tensor_map(CUtensorMap* map, const void* Z, int L, int n2, int CB) {
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  if (((uintptr_t)Z & 15) || CB * 4 > 256) return cudaErrorInvalidValue;
  const cuuint64_t dims[2] = {(cuuint64_t)n2 * 4, (cuuint64_t)L};
  const cuuint64_t strides[1] = {(cuuint64_t)n2 * 16};
  const cuuint32_t box[2] = {(cuuint32_t)(CB * 4), (cuuint32_t)(L < kTmaRows ? L : kTmaRows)};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(Z), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <typename T, int L, int CB, int V, int MODE>
cudaError_t run_b(const void* Z, int n2, const void* twB, const SkyConst* sky, float* out, const PeakArgs& pk,
                  cudaStream_t st, int res) {
  using S = Shape<T, L, V>;
  constexpr size_t smem = MODE == kPeaks ? PeakSmem<T, L, CB, V>::BYTES : Buf<T, L, CB, V>::BYTES;
  constexpr int threads = CB * S::TPC;
  static_assert(MODE != kPeaks || (L * CB * sizeof(float) <= Buf<T, L, CB, V>::ONE), "peaks epilogue reuses the stage");
  static_assert(MODE != kPeaks || threads % 32 == 0, "peaks epilogue works on whole warps");
  int ctas = 0, per_sm = 0;
  const cudaError_t e = resident_ctas(k_pass_b<T, L, CB, V, MODE>, threads, smem, &ctas, &per_sm);
  if (e != cudaSuccess) return e;
  if (n2 % CB) return cudaErrorInvalidConfiguration;
  k_pass_b<T, L, CB, V, MODE><<<persistent_grid(n2 / CB, ctas, per_sm, res), threads, smem, st>>>(
      (const typename S::PM*)Z, n2, (const typename S::TW*)twB, sky, out, pk);
  return cudaGetLastError();
}

// shape code: c = columns (A) / rows (B) per CTA, 0 = default; v = schedule.
// One shape is compiled per length.
template <typename T, int L>
cudaError_t pick_a(int ca, int v, const void* G, GCol gc, int64_t n, int n1, const void* twA, const TmplCoef* coef,
                   void* Z, cudaStream_t st, int res) {
  using S = Shape<T, L, 0>;
  if (v != 0 || (ca > 0 && ca != S::CA_DEF)) return cudaErrorInvalidConfiguration;
  return run_a<T, L, S::CA_DEF, 0>(G, gc, n, n1, twA, coef, Z, st, res);
}
template <typename T, int L, int MODE>
cudaError_t pick_b(int cb, int v, const void* Z, int n2, const void* twB, const SkyConst* sky, float* out,
                   const PeakArgs& pk, cudaStream_t st, int res) {
  using S = Shape<T, L, 0>;
  if (MODE == kPeaks && v == 8) v = 0;
  if (v != 0 || (cb > 0 && cb != S::CB_DEF)) return cudaErrorInvalidConfiguration;
  return run_b<T, L, S::CB_DEF, 0, MODE>(Z, n2, twB, sky, out, pk, st, res);
}

#define FSTAT_LEN_CASES(F, ...)            \
  case 5: return F<T, 32 __VA_ARGS__;    \
  case 6: return F<T, 64 __VA_ARGS__;    \
  case 7: return F<T, 128 __VA_ARGS__;   \
  case 8: return F<T, 256 __VA_ARGS__;   \
  case 9: return F<T, 512 __VA_ARGS__;   \
  case 10: return F<T, 1024 __VA_ARGS__; \
  case 11: return F<T, 2048 __VA_ARGS__; \
  case 12: return F<T, 4096 __VA_ARGS__;

template <typename T>
cudaError_t dispatch_a(int log2_n2, int ca, int v, const void* G, GCol gc, int64_t n, int n1, const void* twA,
                       const TmplCoef* coef, void* Z, cudaStream_t st, int res) {
  switch (log2_n2) {
    FSTAT_LEN_CASES(pick_a, >(ca, v, G, gc, n, n1, twA, coef, Z, st, res))
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, int MODE>
cudaError_t dispatch_b(int log2_n1, int cb, int v, const void* Z, int n2, const void* twB, const SkyConst* sky,
                       float* out, const PeakArgs& pk, cudaStream_t st, int res) {
  switch (log2_n1) {
    FSTAT_LEN_CASES(pick_b, , MODE>(cb, v, Z, n2, twB, sky, out, pk, st, res))
    default: return cudaErrorInvalidValue;
  }
}

#undef FSTAT_LEN_CASES

}  // namespace fft
}  // namespace fstat
