// FP32 FFT passes whose exchanges stay inside a warp.
//
// The passes of fft_impl.cuh exchange data between every two Stockham steps
// across the whole CTA, so its warps load, compute and store in step and
// neither the FMA pipe nor shared memory is busy for more than half the time.
// Here a transform of length L = RL * SUB is split by decimation in time:
//
//   X[k' + SUB m] = sum_{r < RL} W_L^{r k'} W_RL^{r m} X_r[k'],
//   X_r[k'] = sum_{j < SUB} x[r + RL j] W_SUB^{j k'}
//
// Each X_r is computed by SUB / 16 threads of one warp, 16 points per thread,
// with exchanges that only __syncwarp() orders; one exchange across the CTA
// feeds the last radix-RL step.  That leaves two CTA barriers per tile
// instead of five, and between them the warps run freely.  Elements r + RL j
// of a residue r lie together in shared memory, in G and in the intermediate,
// so every access is conflict-free or coalesced without padding.
//
// What bounds it: issue slots and shared-memory wavefronts, which at 16 warps
// per SM (64 data registers a thread) add up rather than overlap: at 2^24 the
// two passes issue 104 us and move 99 us of shared-memory wavefronts per
// template, and took 203 us.  So instructions and exchanges are what counts.
// Per template, two streams (GB300): 2^22 42.8 -> 40.7 us, 2^24 211 -> 190 us
// against the CTA-wide FP32 passes with separate twiddles and a double-float
// phase per sample; pass B alone at 2^24 105 -> 92 us.  Measured and not kept:
// two groups of a CTA taking turns at shared memory through named barriers
// (101.7 -> 107 us for pass A at 4096 points), the intermediate as [n1][k2] rows
// (below).
//
// Intermediate (ZLayout): tile by tile of pass B, [k2 / CB][r][j][k2 mod CB]
// for n1 = r + RL j, so that a tile is one contiguous block.  Pass A's stores
// then go out in pieces of CB pairs, which cost it nothing measurable, and pass
// B at 2^24 reads its 268 MB in 60 us with no arithmetic in the way, against 99
// us from [n1][k2] rows through a tensor map.
#pragma once

#include "fft_impl.cuh"

namespace fstat {
namespace fft {

// SUB: the whole transform where CB interleaved ones of SUBMAX points or fewer
// fit a warp (16 points per thread), else all but the last radix of the
// schedule (r_of, shared with the CTA-wide passes, so that both compute the
// same bits).
template <int L, int CB, int SUBMAX> struct WShape {
  static constexpr int NP = np_of(L, 0);
  static constexpr bool WHOLE = L * CB <= 512 && L <= SUBMAX;
  static constexpr int RL = WHOLE ? 1 : r_of(L, NP - 1, 0);
  static constexpr int SUB = L / RL;
  static constexpr int NS = WHOLE ? NP : NP - 1;  // stages of a sub-transform
  static constexpr int GW = SUB / 16;             // threads of one sub-transform
  static constexpr int TPC = L / 16;              // threads of one transform
  static constexpr int NT = CB * TPC < 32 ? 32 : CB * TPC;
  static constexpr int COLS = NT / (CB * TPC);    // groups of CB transforms per CTA
  static constexpr int R0 = r_of(L, 0, 0);
  static constexpr int RE = r_of(L, NS - 1, 0);   // radix of the sub-transform's last stage
  static constexpr bool WARP = SUB * CB <= 512;   // a sub-transform's threads share a warp
  static constexpr int MINB = NT <= 512 ? 512 / NT : 1;  // 128 registers a thread, 16 warps per SM
  static constexpr bool OK = SUB <= SUBMAX && SUB >= 16 && NT <= 1024;
};
template <int L, int CB, int SUBMAX> __device__ __forceinline__ void sub_sync() {
  if constexpr (WShape<L, CB, SUBMAX>::WARP) __syncwarp();
  else __syncthreads();
}

// Stages P.. of a sub-transform: v holds stage P - 1's outputs (v[w R + q] =
// output q of butterfly u + w GW).  reg: the sub-transform's region (element
// stride CB); xb: the sub-transform's first thread among its warp's (any value
// common to its threads).  The
// first exchange is a transpose of R0-element rows, swizzled by the row.
template <int L, int CB, int SUBMAX, int P, bool TWIST>
__device__ __forceinline__ void sub_stages(Pair<float>* v, float4* reg, int u, int xb, float frac) {
  using S = WShape<L, CB, SUBMAX>;
  if constexpr (P < S::NS) {
    constexpr int RP = r_of(L, P - 1, 0), NSP = ns_of(L, P - 1, 0);
    constexpr int R = r_of(L, P, 0), NSR = ns_of(L, P, 0);
    auto phys = [&](int pos) {
      if constexpr (P > 1) return pos * CB;
      const int row = pos / S::R0;
      return (row * S::R0 + ((pos % S::R0) ^ ((row + xb) & (S::R0 - 1)))) * CB;
    };
#pragma unroll
    for (int w = 0; w < 16 / RP; ++w)
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        const int b = u + w * S::GW;
        pstore(reg + phys((b / NSP) * NSP * RP + b % NSP + q * NSP), v[w * RP + q]);
      }
    sub_sync<L, CB, SUBMAX>();
#pragma unroll
    for (int w = 0; w < 16 / R; ++w)
#pragma unroll
      for (int s = 0; s < R; ++s) v[w * R + s] = pload(reg + phys(u + w * S::GW + s * (S::SUB / R)));
    sub_sync<L, CB, SUBMAX>();
#pragma unroll
    for (int w = 0; w < 16 / R; ++w) {
      const int b = u + w * S::GW;
      dft_tw<float, R>(v + w * R, pass_twiddles<L, P, 0, TWIST>(b, nullptr, Twist<float>(frac)));
    }
    sub_stages<L, CB, SUBMAX, P + 1, TWIST>(v, reg, u, xb, frac);
  }
}

// The radix-RL step across the CTA.  buf(r): the region of residue r.
// at_mid(): has the CTA's barrier after every thread's stores of its
// sub-transform's outputs; at_free(): every thread has read them (the regions
// are free).
template <int L, int CB, int SUBMAX, bool TWIST, typename B, typename M, typename F>
__device__ __forceinline__ void last_step(Pair<float>* v, float4* reg, const B& buf, int u, int tt, float frac,
                                          const M& at_mid, const F& at_free) {
  using S = WShape<L, CB, SUBMAX>;
  if constexpr (S::RL > 1) {
    constexpr int R = S::RE, RL = S::RL;
#pragma unroll
    for (int q = 0; q < 16 / R; ++q)
#pragma unroll
      for (int s = 0; s < R; ++s) pstore(reg + (u + q * S::GW + s * (S::SUB / R)) * CB, v[q * R + s]);
    at_mid();
#pragma unroll
    for (int q = 0; q < 16 / RL; ++q)
#pragma unroll
      for (int r = 0; r < RL; ++r) v[q * RL + r] = pload(buf(r) + (tt + q * S::TPC) * CB);
    __syncthreads();
    at_free();
#pragma unroll
    for (int q = 0; q < 16 / RL; ++q)
      dft_tw<float, RL>(v + q * RL,
                        pass_twiddles<L, S::NP - 1, 0, TWIST>(tt + q * S::TPC, nullptr, Twist<float>(frac)));
  } else {
    at_mid();
    at_free();
  }
}
// output index of v[e] after last_step
template <int L, int CB, int SUBMAX> __device__ __forceinline__ int out_index(int e, int u, int tt) {
  using S = WShape<L, CB, SUBMAX>;
  if constexpr (S::RL > 1) return tt + (e / S::RL) * S::TPC + (e % S::RL) * S::SUB;
  return u + (e / S::RE) * S::GW + (e % S::RE) * (S::SUB / S::RE);
}

__device__ __forceinline__ Pair<float> nan_pair() {
  const float q = __int_as_float(0x7fffffff);
  return {q, q, q, q};
}

// ------------------------------------------------------------- pass A
// G holds column n1's samples residue by residue: sample n2 = r + RL j at
// [(n1 RL + r) lcs + j].  STAGED: the next column (RL lcs pairs) is copied by
// one bulk copy behind the buffer while this one is transformed; otherwise the
// samples are loaded straight into registers.
constexpr int kSubA = 512;  // longest sub-transform of pass A
template <int L> using WA = WShape<L, 1, kSubA>;

template <int L, bool STAGED>
__global__ void __launch_bounds__(WA<L>::NT, WA<L>::MINB)
k_wpass_a(const float4* __restrict__ G, int lcs, int n, int n1, const TmplCoef* __restrict__ coef,
          float4* __restrict__ z0, ZLayout zy, int n_tmpl, int* __restrict__ err, int wait_limit) {
  using S = WA<L>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float4* smem = reinterpret_cast<float4*>(smem_raw);
  // slot: residue (one column per CTA) or column (whole columns per warp)
  const int slot = threadIdx.x / S::GW, u = threadIdx.x % S::GW;
  const int r = S::RL > 1 ? slot : 0, cc = S::RL > 1 ? 0 : slot;
  float4* reg = smem + slot * S::SUB;
  const int tpt = n1 / S::COLS, n_tiles = tpt * n_tmpl;  // tiles per template, in the launch
  const int stride = S::RL * lcs;                        // pairs per column
  float4* stg = smem + S::NT * 16;
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(stg + S::COLS * stride);
  unsigned issued = 0, waited = 0;
  // one bulk copy per tile (neighbouring columns are contiguous); copy u
  // completes phase u of the mbarrier
  auto issue = [&](int tile) {
    const unsigned bytes = (unsigned)(S::COLS * stride * sizeof(float4));
    fence_proxy_async();  // the staging area's earlier reads precede the copy
    mbar_expect_tx(bar, bytes);
    bulk_load(stg, G + (int64_t)(tile % tpt) * S::COLS * stride, bytes, bar);
    ++issued;
  };
  int tile = blockIdx.x;
  if constexpr (STAGED) {
    if (threadIdx.x == 0) {
      mbar_init(bar, 1);
      mbar_fence_init();
      if (tile < n_tiles) issue(tile);
    }
    __syncthreads();
  }
  auto z_col = [&](int col) { return (col & ((1 << zy.rl) - 1)) * zy.sub + (col >> zy.rl); };  // [r][j]
  auto z_at = [&](int zp, int k2) {
    return (((int64_t)(k2 >> zy.cb) * n1 + zp) << zy.cb) + (k2 & ((1 << zy.cb) - 1));
  };
  bool all_ok = true;
  for (; tile < n_tiles; tile += gridDim.x) {
    const int k = tile / tpt, col = (tile - k * tpt) * S::COLS + cc;
    const TmplCoef tc = coef[k];
    if constexpr (STAGED) {
      // the plan may shorten this wait (tests of the timeout path); the
      // drain below always keeps the full limit
      const bool ok = mbar_wait(bar, waited & 1u, wait_limit >= 0 ? wait_limit : kWaitLimit);
      if (ok) ++waited;
      if constexpr (S::NT == 32) all_ok = __all_sync(0xffffffffu, ok) != 0;
      else all_ok = __syncthreads_and(ok) != 0;
      if (!all_ok) break;
    }
    const float4* src = STAGED ? stg + cc * stride + r * lcs : G + ((int64_t)col * S::RL + r) * lcs;
    Pair<float> v[16];
    // no sample at n2 >= L/2: the upper half of every first butterfly is zero
    const bool half = (int64_t)n1 * (L / 2) >= (int64_t)n;
    auto load = [&](auto hf) {  // v[w R0 + s] = input s of butterfly u + w GW
      constexpr bool HALF = decltype(hf)::value;
#pragma unroll
      for (int w = 0; w < 16 / S::R0; ++w) {
        const int j0 = col + n1 * (r + S::RL * (u + w * S::GW)), D = n1 * (L / S::R0);
        Spin<float, S::R0, HALF> spin(tc, j0 - tc.J, D);
#pragma unroll
        for (int s = 0; s < (HALF ? S::R0 / 2 : S::R0); ++s) {
          Pair<float>& x = v[w * S::R0 + s];
          if (j0 + s * D < n) {
            const float4* p = src + u + w * S::GW + s * (S::SUB / S::R0);
            const Pair<float> g = STAGED ? pload(p) : pload_g(p);
            float cs, sn;
            spin.rot(s, &cs, &sn);
            x = pmul(g, cs, sn);
          } else {
            x = pzero<float>();
          }
        }
        if (HALF) dft_half<float, S::R0>(v + w * S::R0);
        else dft<float, S::R0>(v + w * S::R0);
      }
    };
    if (half) load(std::true_type());
    else load(std::false_type());
    sub_stages<L, 1, kSubA, 1, false>(v, reg, u, (threadIdx.x & 31) - u, 0.f);
    last_step<L, 1, kSubA, false>(
        v, reg, [&](int q) { return smem + q * S::SUB; }, u, threadIdx.x, 0.f,
        [&] {
          if constexpr (S::RL > 1) __syncthreads();
          if constexpr (STAGED)
            if (threadIdx.x == 0 && tile + (int)gridDim.x < n_tiles) issue(tile + gridDim.x);
        },
        [] {});
    float4* z = z0 + (int64_t)k * L * n1;
    const int zp = z_col(col);
    auto zat = [&](int k2) { return z_at(zp, k2); };
    if constexpr (L >= 512) {  // the outputs' spacing is a multiple of any CB
      float4* z0 = z + zat(out_index<L, 1, kSubA>(0, u, threadIdx.x));
#pragma unroll
      for (int e = 0; e < 16; ++e) pstore(z0 + (int64_t)out_index<L, 1, kSubA>(e, 0, 0) * n1, v[e]);
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) pstore(z + zat(out_index<L, 1, kSubA>(e, u, threadIdx.x)), v[e]);
    }
  }
  if (STAGED && !all_ok) {
    // a wait ran out: the columns not formed become NaN (which pass B carries to
    // every bin), so that nobody takes what was there before for a result;
    // record it, then give the copy still in flight a bounded chance to land
    // before the CTA's shared memory goes away
    for (; tile < n_tiles; tile += gridDim.x) {
      const int k = tile / tpt, c0 = (tile - k * tpt) * S::COLS;
      for (int i = threadIdx.x; i < S::COLS * L; i += S::NT)
        pstore(z0 + (int64_t)k * L * n1 + z_at(z_col(c0 + i / L), i & (L - 1)), nan_pair());
    }
    if (threadIdx.x == 0) {
      if (err) atomicCAS(err, 0, FSTAT_ERR_TIMEOUT);
      for (unsigned q = waited; q < issued; ++q) mbar_wait(bar, q & 1u);
    }
  }
}

// ------------------------------------------------------------- pass B
constexpr int kSubB = 256;  // longest sub-transform of pass B
template <int L, int CB> using WB = WShape<L, CB, kSubB>;

// A tile = CB neighbouring rows k2 = one contiguous block of the intermediate,
// which arrives in NQ parts of RL / NQ residues by bulk copies into a ring of
// NSLOT part-sized slots (NSLOT > NQ as far as the CTAs that the registers
// allow leave room): the next tile's first parts are on their way during the
// whole of this one, the rest from the moment every thread has read this tile
// for its last step.
template <int L, int CB, int MODE> struct WSmemB {
  using S = WB<L, CB>;
  static constexpr size_t TILE = (size_t)L * CB * sizeof(float4);
  static constexpr int NQ = S::RL >= 4 ? 4 : 1;
  static constexpr size_t PART = TILE / NQ;
  static constexpr size_t KEYS = (size_t)kPeakBands * sizeof(unsigned long long);
  static constexpr size_t SF = (size_t)L * CB * sizeof(float);  // the tile's 2F (peaks mode)
  static constexpr size_t EXTRA = (MODE == kPeaks ? SF + KEYS : 0) + 128;  // and the mbarriers
  // a CTA's shared memory is its own plus 1 KB, of 228 KB per SM
  static constexpr size_t ROOM = (size_t)228 * 1024 / S::MINB - 1024;
  static constexpr int FIT = ROOM > EXTRA ? (int)((ROOM - EXTRA) / PART) : 0;
  static constexpr int CAP = 2 * NQ - (NQ > 1);  // 7 parts of a quarter, 2 whole tiles
  static constexpr int NSLOT = FIT > CAP ? CAP : FIT < NQ ? NQ : FIT;  // (fewer CTAs where not even one tile fits)
  static constexpr size_t SF_AT = NSLOT * PART, KEYS_AT = SF_AT + (MODE == kPeaks ? SF : 0);
  static constexpr size_t BAR_AT = KEYS_AT + (MODE == kPeaks ? KEYS : 0);
  static constexpr size_t BYTES = BAR_AT + 128;
  static constexpr bool OK = BYTES <= kSmemOptIn;
};

template <int L, int CB, int MODE>
__global__ void __launch_bounds__(WB<L, CB>::NT, WB<L, CB>::MINB)
k_wpass_b(int n2, const SkyConst* __restrict__ sky, float* __restrict__ out, const int* __restrict__ ord,
          int64_t out_rows, int n_tmpl, int n_bands, const PeakArgs pk0, const float4* __restrict__ z0) {
  using S = WB<L, CB>;
  using M = WSmemB<L, CB, MODE>;
  static_assert(S::COLS == 1, "pass B tiles fill at least a warp");
  static_assert(M::NSLOT <= 16, "mbarriers");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  constexpr int RQ = S::RL / M::NQ;              // residues per part
  constexpr int PP = (int)(M::PART / sizeof(float4));
  const int c = threadIdx.x % CB, tt = threadIdx.x / CB;
  const int r = tt / S::GW, u = tt % S::GW;
  const float kA = sky->kAf, kB = sky->kBf, kC = sky->kCf;
  float* sf = reinterpret_cast<float*>(smem_raw + M::SF_AT);
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem_raw + M::BAR_AT);
  // peaks mode with whole-row bands: this CTA's band keys of the current template
  unsigned long long* ks = nullptr;
  if constexpr (MODE == kPeaks) {
    if (pk0.band_key && pk0.log2_band >= 31 - __clz(n2) && n_bands <= kPeakBands)
      ks = reinterpret_cast<unsigned long long*>(smem_raw + M::KEYS_AT);
  }
  const int tpt = n2 / CB, n_tiles = tpt * n_tmpl;
  // part g = NQ it + q of this CTA's tiles it = 0, 1, ..: slot g mod NSLOT,
  // phase g / NSLOT of the slot's mbarrier.  Thread 0 issues them in order.
  int issued = 0;
  auto issue_below = [&](int end) {
    for (; issued < end; ++issued) {
      const int it = issued / M::NQ, q = issued % M::NQ, slot = issued % M::NSLOT;
      const int64_t tile = blockIdx.x + (int64_t)it * gridDim.x;
      if (tile >= n_tiles) break;
      mbar_expect_tx(&bar[slot], (unsigned)M::PART);
      bulk_load(smem_raw + slot * M::PART, z0 + tile * (L * CB) + q * PP,
                (unsigned)M::PART, &bar[slot]);
    }
  };
  if (threadIdx.x == 0) {
    for (int q = 0; q < M::NSLOT; ++q) mbar_init(&bar[q], 1);
    mbar_fence_init();
    issue_below(M::NSLOT);
  }
  if constexpr (MODE == kPeaks)
    if (ks)
      for (int b = threadIdx.x; b < n_bands; b += S::NT) ks[b] = 0ull;
  __syncthreads();
  bool all_ok = true;
  int cur = -1;  // template whose keys ks holds
  PeakArgs pk = pk0;
  float* row = out;
  auto flush = [&] {  // the keys of template `cur` to global memory
    __syncthreads();
    for (int b = threadIdx.x; b < n_bands; b += S::NT) {
      if (ks[b]) atomicMax(pk.band_key + b, ks[b]);
      ks[b] = 0ull;
    }
    __syncthreads();
  };
  int it = 0, g0 = 0;         // tile of this CTA, slot of its first part
  unsigned par0 = 0;          // phase parity of that slot
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
    const int k = tile / tpt, k2 = (tile - k * tpt) * CB + c;
    if (k != cur) {
      if constexpr (MODE == kPeaks)
        if (ks && cur >= 0) flush();
      cur = k;
      if (ord) {
        const int i = ord[k];
        if constexpr (MODE == kPeaks) {
          if (pk0.band_key) pk.band_key = pk0.band_key + (int64_t)i * n_bands;
          pk.tmpl = pk0.tmpl + i;
        } else {
          row = out + (int64_t)(i % out_rows) * ((int64_t)n2 * L);
        }
      }
    }
    // accumulate mode: the running sums this thread adds to, loaded before
    // the transform so their latency hides under it
    float acc[MODE == kAccumulate ? 16 : 1];
    if (MODE == kAccumulate && !pk.first) {
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const int mg = k2 + n2 * ((out_index<L, CB, kSubB>(e, u, tt) + L / 2) & (L - 1)) - pk.shift;
        acc[e] = (unsigned)mg < (unsigned)(n2 * L) ? row[mg] : 0.f;
      }
    }
    auto region = [&](int rr) {  // of residue rr
      const int q = g0 + rr / RQ;
      return reinterpret_cast<float4*>(smem_raw) + (q < M::NSLOT ? q : q - M::NSLOT) * PP + (rr % RQ) * (S::SUB * CB) + c;
    };
    float4* reg = region(r);
    // this thread's part only.  The plan may shorten this first wait (tests of
    // the timeout path); the drain below always keeps the full limit.
    const int mq = g0 + r / RQ;
    const bool wrap = mq >= M::NSLOT;
    const bool ok = mbar_wait(&bar[wrap ? mq - M::NSLOT : mq], par0 ^ (wrap ? 1u : 0u),
                              pk.wait_set ? pk.wait_limit : kWaitLimit);
    if constexpr (S::RL == 1) all_ok = __all_sync(0xffffffffu, ok) != 0;
    if constexpr (S::RL == 1)
      if (!all_ok) break;
    const float frac = (float)k2 / (float)n2;
    Pair<float> v[16];
#pragma unroll
    for (int w = 0; w < 16 / S::R0; ++w)
#pragma unroll
      for (int s = 0; s < S::R0; ++s)
        v[w * S::R0 + s] = pload(reg + (u + w * S::GW + s * (S::SUB / S::R0)) * CB);
    sub_sync<L, CB, kSubB>();
    {
      const Twiddles<float, S::R0> w0 = pass_twiddles<L, 0, 0, true>(0, nullptr, Twist<float>(frac));
#pragma unroll
      for (int w = 0; w < 16 / S::R0; ++w) dft_tw<float, S::R0>(v + w * S::R0, w0);
    }
    sub_stages<L, CB, kSubB, 1, true>(v, reg, u, S::WARP ? (int)(threadIdx.x & 31) / CB - u : 0, frac);
    auto next = [&] {
      if (threadIdx.x == 0) {
        fence_proxy_async();  // this tile's reads and writes of its slots precede the copies into them
        issue_below(M::NQ * (it + 1) + M::NSLOT);
      }
      g0 += M::NQ;
      if (g0 >= M::NSLOT) { g0 -= M::NSLOT; par0 ^= 1u; }
      if (g0 >= M::NSLOT) { g0 -= M::NSLOT; par0 ^= 1u; }
    };
    last_step<L, CB, kSubB, true>(v, reg, region, u, tt, frac, [&] {
      if constexpr (S::RL > 1) all_ok = __syncthreads_and(ok) != 0;
    }, [&] {
      if constexpr (S::RL > 1)
        if (all_ok) next();
    });
    if constexpr (S::RL > 1) {
      if (!all_ok) break;
    } else {  // one warp: its last reads were ordered by __syncwarp
      __syncwarp();
      next();
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const Pair<float>& x = v[e];
      const float tf = two_f(x, kA, kB, kC);
      const int rr = (out_index<L, CB, kSubB>(e, u, tt) + L / 2) & (L - 1);
      if constexpr (MODE == kPeaks) {
        sf[rr * CB + c] = tf;
      } else if constexpr (MODE == kAccumulate) {
        // semi-coherent sum: this segment's bin m adds to global bin m - shift
        const int mg = k2 + n2 * rr - pk.shift;
        const bool in = (unsigned)mg < (unsigned)(n2 * L);
        if (pk.first) row[mg & (n2 * L - 1)] = in ? tf : 0.f;  // the bins that wrap around are the ones no bin reaches
        else if (in) row[mg] = acc[e] + tf;
      } else {
        __stcs(row + k2 + n2 * rr, tf);  // streaming store: keep G and Z in L2
      }
    }
    if constexpr (MODE == kPeaks) {
      __syncthreads();
      peak_epilogue<CB, 16>(sf, k2 - c, n2, pk, ks);
      if constexpr (S::RL == 1) __syncthreads();  // else the next tile's barriers precede its writes to sf
    }
  }
  if (!all_ok) {
    // a wait ran out: 2F of the rows not formed becomes NaN (as in pass A);
    // record it, then give the loads still in flight a bounded chance to land
    // before the CTA's shared memory goes away
    if constexpr (MODE != kPeaks) {
      for (int tile = blockIdx.x + it * gridDim.x; tile < n_tiles; tile += gridDim.x) {
        const int k = tile / tpt, m0 = (tile - k * tpt) * CB;
        if (ord) row = out + (int64_t)(ord[k] % out_rows) * ((int64_t)n2 * L);
        for (int i = threadIdx.x; i < L * CB; i += S::NT) {
          const int mg = m0 + (i & (CB - 1)) + n2 * (i / CB) - (MODE == kAccumulate ? pk.shift : 0);
          const bool in = MODE == kStore || (unsigned)mg < (unsigned)(n2 * L);
          if (in) row[mg] = nan_pair().ar;
          else if (pk.first) row[mg & (n2 * L - 1)] = 0.f;
        }
      }
    }
    if (threadIdx.x == 0) {
      if (pk.err) atomicCAS(pk.err, 0, FSTAT_ERR_TIMEOUT);
      for (int g = M::NQ * it; g < issued; ++g) mbar_wait(&bar[g % M::NSLOT], (unsigned)(g / M::NSLOT) & 1u);
    }
    return;
  }
  if constexpr (MODE == kPeaks)
    if (ks && cur >= 0) flush();
}

// ------------------------------------------------------------- launchers
// Pass A.  staging: 0 = where the staged columns leave room for as many CTAs
// as registers allow, 1 = required, 2 = none.
template <int L>
cudaError_t run_wa(const float4* G, int lcs, int64_t n, int n1, const TmplCoef* coef, float4* z, ZLayout zy, int n_tmpl,
                   int staging, int* err, int wait_limit, cudaStream_t st, int res) {
  using S = WA<L>;
  if (n1 % S::COLS) return cudaErrorInvalidConfiguration;
  constexpr size_t buf = (size_t)S::NT * 16 * sizeof(float4);
  const size_t with = buf + (size_t)S::COLS * S::RL * lcs * sizeof(float4) + 16;
  // (a CTA's shared memory is its own plus 1 KB, of 228 KB per SM)
  const bool fits = with <= kSmemOptIn, room = (with + 1024) * S::MINB <= (size_t)228 * 1024;
  if (staging == 1 && !fits) return cudaErrorInvalidConfiguration;
  const bool staged = staging == 1 || (staging == 0 && fits && room);
  auto launch = [&](auto kernel, size_t smem) {
    int ctas = 0, per_sm = 0;
    const cudaError_t e = resident_ctas(kernel, S::NT, smem, &ctas, &per_sm);
    if (e != cudaSuccess) return e;
    kernel<<<persistent_grid(n1 / S::COLS * n_tmpl, ctas, per_sm, res), S::NT, smem, st>>>(
        G, lcs, (int)n, n1, coef, z, zy, n_tmpl, err, wait_limit);
    return cudaGetLastError();
  };
  if (staged) return launch(k_wpass_a<L, true>, with);
  return launch(k_wpass_a<L, false>, buf);
}

struct WBArgs {
  const SkyConst* sky;
  float* out;
  const int* ord;
  int64_t out_rows;
  int n_tmpl, n_bands;
  PeakArgs pk;
};

template <int L, int CB> constexpr bool wb_ok() {
  return WB<L, CB>::OK && WB<L, CB>::COLS == 1 && WSmemB<L, CB, kPeaks>::OK;
}

template <int L, int CB, int MODE>
cudaError_t run_wb(float4* z, int n2, const WBArgs& a, cudaStream_t st, int res) {
  using S = WB<L, CB>;
  if constexpr (!wb_ok<L, CB>()) {
    return cudaErrorInvalidConfiguration;
  } else {
    constexpr size_t smem = WSmemB<L, CB, MODE>::BYTES;
    static_assert(smem <= kSmemOptIn, "shared memory of a CTA");
    if (n2 % CB) return cudaErrorInvalidConfiguration;
    int ctas = 0, per_sm = 0;
    const cudaError_t e = resident_ctas(k_wpass_b<L, CB, MODE>, S::NT, smem, &ctas, &per_sm);
    if (e != cudaSuccess) return e;
    k_wpass_b<L, CB, MODE><<<persistent_grid(n2 / CB * a.n_tmpl, ctas, per_sm, res), S::NT, smem, st>>>(
        n2, a.sky, a.out, a.ord, a.out_rows, a.n_tmpl, a.n_bands, a.pk, z);
    return cudaGetLastError();
  }
}

// rows per tile unless the caller asks for others: 64 bytes of a row where two
// CTAs of such tiles fit an SM's registers, and at least a warp
template <int L> constexpr int default_wcb() { return L >= 2048 ? 2 : L >= 128 ? 4 : 512 / L; }

// rows per tile of length L that a shape code stands for: itself, or the default
template <int L> constexpr int wb_rows(int cb) {
  return (cb == 1 && wb_ok<L, 1>()) || (cb == 2 && wb_ok<L, 2>()) || (cb == 4 && wb_ok<L, 4>()) ||
                 (cb == 8 && wb_ok<L, 8>())
             ? cb
             : default_wcb<L>();
}

template <int L, int MODE>
cudaError_t pick_wb(int cb, float4* z, int n2, const WBArgs& a, cudaStream_t st, int res) {
  switch (wb_rows<L>(cb)) {
    case 1: return run_wb<L, 1, MODE>(z, n2, a, st, res);
    case 2: return run_wb<L, 2, MODE>(z, n2, a, st, res);
    case 4: return run_wb<L, 4, MODE>(z, n2, a, st, res);
    case 8: return run_wb<L, 8, MODE>(z, n2, a, st, res);
    default: return run_wb<L, default_wcb<L>(), MODE>(z, n2, a, st, res);
  }
}
template <int MODE>
cudaError_t dispatch_wb(int log2_n1, int cb, float4* z, int n2, const WBArgs& a, cudaStream_t st, int res) {
  switch (log2_n1) {
    case 5: return pick_wb<32, MODE>(cb, z, n2, a, st, res);
    case 6: return pick_wb<64, MODE>(cb, z, n2, a, st, res);
    case 7: return pick_wb<128, MODE>(cb, z, n2, a, st, res);
    case 8: return pick_wb<256, MODE>(cb, z, n2, a, st, res);
    case 9: return pick_wb<512, MODE>(cb, z, n2, a, st, res);
    case 10: return pick_wb<1024, MODE>(cb, z, n2, a, st, res);
    case 11: return pick_wb<2048, MODE>(cb, z, n2, a, st, res);
    case 12: return pick_wb<4096, MODE>(cb, z, n2, a, st, res);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fft
}  // namespace fstat
