// Step (ii) of Sec. 3 from short Fourier transforms (fstat_set_sfts): per
// SFT s the band of B bins around f_h is inverse-transformed to B samples
// at dt = T_sft / B, rotated by exp(-2 pi i f_h t_s) and scaled by 1/M:
//
//   x_h[s B + m] = exp(-2 pi i f_h t_s) / M * sum_{i=0}^{B-1} X_s[i] exp(2 pi i (i - B/2) m / B)
//
// (column i of the band holds SFT bin q_h - B/2 + i).  B need not be a
// power of two (1800 s and 2 Hz give 3600 bins), so the transform is a
// Stockham pipeline over B's own factors, one SFT per CTA in two
// shared-memory buffers: factors up to 16 as register butterflies, larger
// primes as direct sums of that length.  Every root of unity is taken from
// one table of B entries at an exactly reduced integer index.  FP32 for
// mixed plans, FP64 for FP64 plans.
//
// The direct sum over all B bins is issue-bound at B terms per sample;
// 3600 = 16 x 15 x 15 needs about 46.  Two detectors x 480 SFTs of 3600 bins
// from pinned memory to 2F of two templates: 9436 us with the direct sums
// (4205 us of kernel per detector), 508 us here.  A band of prime length
// keeps the direct sum (480 SFTs of 4001 bins from device memory: 4.3 ms).

#include <math.h>

#include <algorithm>

#include "fstat_internal.cuh"
#include "sft.cuh"

namespace fstat {

namespace {

constexpr int kSftThreads = 256;
constexpr int kSftOut = 4;           // outputs per thread of a direct pass
constexpr int kSftMaxPasses = 16;    // B < 2^16 has at most 15 prime factors
constexpr size_t kSftSmemMax = (size_t)220 * 1024;

template <typename T> struct C2;
template <> struct C2<float> { using type = float2; };
template <> struct C2<double> { using type = double2; };

// Largest factor done as one register butterfly: a radix-R thread holds 2R
// values and R roots, so FP64 stops at 8 (16 would spill).
template <typename T> constexpr int max_radix() { return sizeof(T) == 4 ? 16 : 8; }

struct SftPlan {
  int np;
  int r[kSftMaxPasses];
};

// B as a product of radices: primes above max_radix stand alone (direct
// passes), the rest is packed greedily into the largest radices that divide
// what is left (few passes; a radix-R butterfly costs ~R multiply-adds per
// point, a pass one exchange through shared memory).  Direct passes come first,
// where a warp's lanes read the same roots, or (direct_last) last, the longest at the
// end: its outputs can go to several CTAs, and it has a shared-memory buffer to spare
// for the roots.
SftPlan sft_factors(int B, int max_r) {
  SftPlan p{};
  int rest = B;
  for (int q = max_r + 1; (int64_t)q * q <= rest;) {
    bool prime = true;
    for (int d = 2; d * d <= q && prime; ++d) prime = q % d != 0;
    if (prime && rest % q == 0) {
      p.r[p.np++] = q;
      rest /= q;
    } else {
      ++q;
    }
  }
  while (rest > 1) {
    int r = 0;
    for (int q = max_r; q >= 2 && !r; --q)
      if (rest % q == 0) r = q;
    if (!r) {  // no divisor up to max_r: a smaller-than-max_r^2 remainder splits into one large prime and its cofactor
      r = rest;
      for (int d = 2; d * d <= rest; ++d)
        if (rest % d == 0) { r = rest / d; break; }
    }
    p.r[p.np++] = r;
    rest /= r;
  }
  if (p.np == 0) p.r[p.np++] = 1;
  return p;
}
void direct_last(SftPlan& p, int max_r) {
  std::sort(std::stable_partition(p.r, p.r + p.np, [&](int r) { return r <= max_r; }), p.r + p.np);
}

// exp(2 pi i j / B), j < B, computed in FP64
template <typename T>
__global__ void k_sft_roots(int64_t B, typename C2<T>::type* __restrict__ w) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < B; j += (int64_t)gridDim.x * blockDim.x) {
    double s, c;
    sincospi(2.0 * (double)j / (double)B, &s, &c);
    w[j] = {(T)c, (T)s};
  }
}

// y_q = sum_s x_s exp(2 pi i q s / R), in place.  wr[j] = exp(2 pi i j / R).
// The inputs s and R - s meet the same cosine and opposite sines, as do the
// outputs q and R - q, so folding both ways leaves R^2 real multiply-adds.
template <typename T, int R>
__device__ __forceinline__ void dft_odd_even(typename C2<T>::type* x, const typename C2<T>::type* wr) {
  using V = typename C2<T>::type;
  constexpr int H = (R - 1) / 2;  // folded pairs
  V a[H + 1], d[H + 1];
#pragma unroll
  for (int s = 1; s <= H; ++s) {
    a[s] = {x[s].x + x[R - s].x, x[s].y + x[R - s].y};
    d[s] = {x[s].x - x[R - s].x, x[s].y - x[R - s].y};
  }
  const V x0 = x[0];
  V xm = {(T)0, (T)0};
  if constexpr (R % 2 == 0) xm = x[R / 2];
  V y0 = x0;
#pragma unroll
  for (int s = 1; s <= H; ++s) { y0.x += a[s].x; y0.y += a[s].y; }
  x[0] = {y0.x + xm.x, y0.y + xm.y};
  if constexpr (R % 2 == 0) {
    V yh = x0;
#pragma unroll
    for (int s = 1; s <= H; ++s) {
      if (s & 1) { yh.x -= a[s].x; yh.y -= a[s].y; }
      else { yh.x += a[s].x; yh.y += a[s].y; }
    }
    x[R / 2] = (R / 2) & 1 ? V{yh.x - xm.x, yh.y - xm.y} : V{yh.x + xm.x, yh.y + xm.y};
  }
#pragma unroll
  for (int q = 1; q <= H; ++q) {
    V e = x0, o = {(T)0, (T)0};
    if constexpr (R % 2 == 0) {
      if (q & 1) { e.x -= xm.x; e.y -= xm.y; }
      else { e.x += xm.x; e.y += xm.y; }
    }
#pragma unroll
    for (int s = 1; s <= H; ++s) {
      const int k = (q * s) % R;
      const T c = k <= R / 2 ? wr[k].x : wr[R - k].x;
      const T sn = k <= R / 2 ? wr[k].y : -wr[R - k].y;
      e.x += a[s].x * c;
      e.y += a[s].y * c;
      o.x += d[s].x * sn;
      o.y += d[s].y * sn;
    }
    // y_q = e + i o, y_{R-q} = e - i o
    x[q] = {e.x - o.y, e.y + o.x};
    x[R - q] = {e.x + o.y, e.y - o.x};
  }
}

template <typename T> struct Out {
  typename C2<T>::type* p;  // shared-memory buffer, or the series
  const typename C2<T>::type* roots;
  T rc, rs;     // the last pass's common factor
  int B;
  bool last;
  int* err;
  // value of transform output m: stored, or finished (the shift of the band
  // centre, the SFT's phase and 1/M) and checked in the last pass
  __device__ __forceinline__ void put(int m, typename C2<T>::type v) const {
    if (last) {
      const typename C2<T>::type w = roots[(unsigned)((B - B / 2) * m) % (unsigned)B];
      const T fr = w.x * rc - w.y * rs, fi = w.x * rs + w.y * rc;
      v = {v.x * fr - v.y * fi, v.x * fi + v.y * fr};
      if (!isfinite(v.x) || !isfinite(v.y)) atomicCAS(err, 0, FSTAT_ERR_NONFINITE);
    }
    p[m] = v;
  }
};

template <typename T, int R>
__device__ __forceinline__ void pass_r(const typename C2<T>::type* src, const Out<T>& out, int B, int ns) {
  using V = typename C2<T>::type;
  const int nb = B / R, step = B / (ns * R);
  V wr[R / 2 + 1];
#pragma unroll
  for (int j = 0; j <= R / 2; ++j) wr[j] = out.roots[j * nb];
  for (int b = threadIdx.x; b < nb; b += kSftThreads) {
    const int hi = b / ns, k = b - hi * ns;
    V x[R];
#pragma unroll
    for (int s = 0; s < R; ++s) {
      x[s] = src[b + s * nb];
      if (s > 0) {
        const V w = out.roots[k * step * s];  // k step s < B / ns * (ns - 1) / R * (R - 1) < B
        x[s] = {x[s].x * w.x - x[s].y * w.y, x[s].x * w.y + x[s].y * w.x};
      }
    }
    dft_odd_even<T, R>(x, wr);
    const int base = hi * ns * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) out.put(base + q * ns, x[q]);
  }
}

// one pass of any length r by its defining sum: kSftOut outputs q of one
// butterfly per thread share each input; the root index (k step + q B/r) s
// advances by an exactly reduced step per term.  The last pass's outputs spread
// over the grid's y, whose CTAs have all formed the passes before it
template <typename T>
__device__ __forceinline__ void pass_direct(const typename C2<T>::type* src, const Out<T>& out, int B, int ns, int r) {
  using V = typename C2<T>::type;
  const int nb = B / r, step = B / (ns * r), groups = (r + kSftOut - 1) / kSftOut;
  const int y = out.last ? blockIdx.y : 0, ny = out.last ? gridDim.y : 1;
  for (int u = y * kSftThreads + threadIdx.x; u < nb * groups; u += kSftThreads * ny) {
    const int g = u / nb, b = u - g * nb, hi = b / ns, k = b - hi * ns;
    int e[kSftOut], j[kSftOut];
    V y[kSftOut];
#pragma unroll
    for (int t = 0; t < kSftOut; ++t) {
      const int q = g + t * groups;
      e[t] = q < r ? k * step + q * nb : 0;  // < B
      j[t] = 0;
      y[t] = {(T)0, (T)0};
    }
    for (int s = 0; s < r; ++s) {
      const V x = src[b + s * nb];
#pragma unroll
      for (int t = 0; t < kSftOut; ++t) {
        const V w = out.roots[j[t]];
        y[t].x += x.x * w.x - x.y * w.y;
        y[t].y += x.x * w.y + x.y * w.x;
        j[t] += e[t];
        if (j[t] >= B) j[t] -= B;
      }
    }
    const int base = hi * ns * r + k;
#pragma unroll
    for (int t = 0; t < kSftOut; ++t) {
      const int q = g + t * groups;
      if (q < r) out.put(base + q * ns, y[t]);
    }
  }
}

// SPARE: the roots do not fit beside the data and the last pass is a direct one, which
// takes them into the buffer that it does not write (a kernel of its own: the others'
// pointer to the roots stays fixed, 3 % of 480 SFTs of 3600 bins)
template <typename T, typename TIn, bool SPARE>
__global__ void __launch_bounds__(kSftThreads)
k_sft_to_xh(const TIn* __restrict__ bins, const typename C2<T>::type* __restrict__ roots, int B, SftPlan plan,
            int roots_in_smem, double f_het, double t_start, double t_sft, double inv_m,
            typename C2<T>::type* __restrict__ xh, int* err) {
  using V = typename C2<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* cur = reinterpret_cast<V*>(smem_raw);
  V* nxt = cur + B;  // unused (and not there) with a single pass
  const int s = blockIdx.x;
  const TIn* src = bins + (int64_t)s * B;
  Out<T> out;
  out.roots = roots;
  if (roots_in_smem) {
    V* sw = cur + (size_t)(plan.np > 1 ? 2 : 1) * B;
    for (int i = threadIdx.x; i < B; i += kSftThreads) sw[i] = roots[i];
    out.roots = sw;
  }
  for (int i = threadIdx.x; i < B; i += kSftThreads) {
    const TIn v = src[i];
    cur[i] = {(T)v.x, (T)v.y};
  }
  // exp(-2 pi i f_h t_s) / M with f_h t_s reduced mod 1 in FP64
  const double t_s = t_start + (double)s * t_sft;
  double ph = f_het * t_s;
  ph -= floor(ph);
  double sn, cs;
  sincospi(2.0 * ph, &sn, &cs);
  out.rc = (T)(cs * inv_m);
  out.rs = (T)(-sn * inv_m);
  out.B = B;
  out.err = err;
  int ns = 1;
  for (int p = 0; p < plan.np; ++p) {
    __syncthreads();
    const int r = plan.r[p];
    out.last = p + 1 == plan.np;
    out.p = out.last ? xh + (int64_t)s * B : nxt;
    if constexpr (SPARE)
      if (out.last) {
        for (int i = threadIdx.x; i < B; i += kSftThreads) nxt[i] = roots[i];
        out.roots = nxt;
        __syncthreads();
      }
    switch (r) {
#define FSTAT_SFT_R(R) \
  case R: if constexpr (R <= max_radix<T>()) { pass_r<T, R>(cur, out, B, ns); break; }
      FSTAT_SFT_R(2) FSTAT_SFT_R(3) FSTAT_SFT_R(4) FSTAT_SFT_R(5) FSTAT_SFT_R(6) FSTAT_SFT_R(7) FSTAT_SFT_R(8)
      FSTAT_SFT_R(9) FSTAT_SFT_R(10) FSTAT_SFT_R(11) FSTAT_SFT_R(12) FSTAT_SFT_R(13) FSTAT_SFT_R(14)
      FSTAT_SFT_R(15) FSTAT_SFT_R(16)
#undef FSTAT_SFT_R
      default: pass_direct<T>(cur, out, B, ns, r); break;
    }
    ns *= r;
    V* t = cur;
    cur = nxt;
    nxt = t;
  }
}

template <typename T, typename TIn>
cudaError_t run_sft(const void* bins, int64_t n_sft, int B, double f_het, double t_start, double t_sft,
                    int64_t m_raw, void* roots, void* xh, int* err, cudaStream_t st) {
  using V = typename C2<T>::type;
  SftPlan plan = sft_factors(B, max_radix<T>());
  // data buffers, and the roots beside them where they fit (else from L1)
  size_t smem = (size_t)(plan.np > 1 ? 2 : 1) * B * sizeof(V);
  const bool in_smem = smem + (size_t)B * sizeof(V) <= kSftSmemMax;
  if (in_smem) smem += (size_t)B * sizeof(V);
  // The longest direct pass over as many CTAs per SFT as have threads for it and, behind
  // other passes (formed by each of them), as the GPU holds.  us per call, one CTA per
  // SFT with roots that do not fit read from L1 -> so: 1 SFT of 3998 = 2 x 1999 bins
  // 818 -> 236, of 4193 = 7 x 599 314 -> 99; 1 of 12003 = 3 x 4001 18400 -> 414, 480 of
  // them 100900 -> 17600 (one direct sum over the whole band: 449, 405, 1217, 38400).
  // With one CTA and its roots at hand direct passes stay first (182 SFTs of 938 = 14 x
  // 67 bins to 2F: 139 us, 143 with the direct one last).
  const int longest = *std::max_element(plan.r, plan.r + plan.np);
  unsigned split = 1;
  bool spare = false;
  if (longest > max_radix<T>()) {
    const int groups = (longest + kSftOut - 1) / kSftOut;
    split = (unsigned)(((int64_t)(B / longest) * groups + kSftThreads - 1) / kSftThreads);
    const int64_t room = (int64_t)device_sm_count() * std::max<int64_t>(1, (228 * 1024) / (int64_t)(smem + 1024));
    if (plan.np > 1) split = (unsigned)std::min<int64_t>(split, std::max<int64_t>(1, room / n_sft));
    spare = !in_smem;
    if (split > 1 || spare) direct_last(plan, max_radix<T>());
  }
  const auto kernel = spare ? k_sft_to_xh<T, TIn, true> : k_sft_to_xh<T, TIn, false>;
  // (the limit belongs to the kernel, not to this call: every call sets the same
  // value, so that none lowers it between another thread's setting and launch)
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSftSmemMax);
  if (e != cudaSuccess) return e;
  k_sft_roots<T><<<(B + 255) / 256, 256, 0, st>>>(B, (V*)roots);
  const dim3 grid((unsigned)n_sft, split);
  kernel<<<grid, kSftThreads, smem, st>>>((const TIn*)bins, (const V*)roots, B, plan, in_smem, f_het, t_start, t_sft,
                                          1.0 / (double)m_raw, (V*)xh, err);
  return cudaGetLastError();
}

}  // namespace

size_t sft_smem_bytes(int B, int precision) {
  return (size_t)2 * B * (precision == FSTAT_FP64 ? sizeof(double2) : sizeof(float2));
}

cudaError_t launch_sft_to_xh(int precision, int in_dtype, const void* bins, int64_t n_sft, int B, double f_het,
                             double t_start, double t_sft, int64_t m_raw, void* roots, void* xh, int* err,
                             cudaStream_t st) {
  const bool in64 = in_dtype == FSTAT_C128;
  if (precision == FSTAT_FP64)
    return in64 ? run_sft<double, double2>(bins, n_sft, B, f_het, t_start, t_sft, m_raw, roots, xh, err, st)
                : run_sft<double, float2>(bins, n_sft, B, f_het, t_start, t_sft, m_raw, roots, xh, err, st);
  return in64 ? run_sft<float, double2>(bins, n_sft, B, f_het, t_start, t_sft, m_raw, roots, xh, err, st)
              : run_sft<float, float2>(bins, n_sft, B, f_het, t_start, t_sft, m_raw, roots, xh, err, st);
}

}  // namespace fstat
