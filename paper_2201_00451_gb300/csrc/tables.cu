// Twiddle tables of the FP64 passes (the FP32 passes use the hardware
// sine/cosine): roots of unity exp(-2 pi i m / M), evaluated by sincospi.
//
// Layout of one table block for n_fft = N1 * N2 = 2^(l1 + l2):
//   [ N2 entries, M = N2 ]          Stockham roots of pass A
//   [ N1 entries, M = N1 ]          Stockham roots of pass B
//   [ 4 x N2 entries ]              pass B's twist: for its Stockham pass p
//                                   of span NS and radix R, and row k2,
//                                   exp(-2 pi i (k2 / N2) / (NS R))
#include "fft_impl.cuh"

#include <algorithm>
#include <mutex>
#include <vector>

namespace fstat {
namespace {

// exp(-2 pi i / M * i), M = 2^log2m
__global__ void k_roots(double2* out, int count, int log2m) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  double s, c;
  sincospi(-2.0 * (double)i / (double)((int64_t)1 << log2m), &s, &c);
  out[i] = {c, s};
}

// log2(NS R) after pass p of a length-L transform's schedule 0
template <int L> int span_log2(int p) {
  int r = 0;
  for (int q = 0; q <= p && q < fft::np_of(L, 0); ++q) r += fft::log2c(fft::r_of(L, q, 0));
  return r;
}
int pass_span_log2(int log2l, int p) {
  switch (log2l) {
    case 5: return span_log2<32>(p);
    case 6: return span_log2<64>(p);
    case 7: return span_log2<128>(p);
    case 8: return span_log2<256>(p);
    case 9: return span_log2<512>(p);
    case 10: return span_log2<1024>(p);
    case 11: return span_log2<2048>(p);
    default: return span_log2<4096>(p);
  }
}

void roots(double2* out, int count, int log2m, cudaStream_t st) {
  k_roots<<<(count + 255) / 256, 256, 0, st>>>(out, count, log2m);
}

}  // namespace

namespace fft {
cudaError_t resident_ctas(const void* kernel, int threads, size_t smem, int* out, int* out_per_sm) {
  // a kernel of this library takes at most a few shared-memory sizes per plan
  struct Entry { const void* k; int dev; size_t smem; int ctas, per_sm; };
  static std::mutex mu;
  static std::vector<Entry> known;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  for (const Entry& x : known)
    if (x.k == kernel && x.dev == dev && x.smem == smem) {
      *out = x.ctas;
      *out_per_sm = x.per_sm;
      return cudaSuccess;
    }
  // the attribute only ever grows: an earlier size stays launchable
  size_t most = smem;
  for (const Entry& x : known)
    if (x.k == kernel && x.dev == dev) most = std::max(most, x.smem);
  if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most)) != cudaSuccess) return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem)) != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  *out_per_sm = per_sm;
  *out = device_sm_count() * per_sm;
  if (known.size() >= 4096) known.clear();
  known.push_back(Entry{kernel, dev, smem, *out, per_sm});
  return cudaSuccess;
}
}  // namespace fft

int device_sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  if (!cached[dev]) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    cached[dev] = sms;
  }
  return cached[dev];
}

TwiddleTables twiddle_layout(int log2n1, int log2n2, void* base) {
  TwiddleTables t{};
  double2* p = (double2*)base;
  t.a = p;
  t.b = p + ((size_t)1 << log2n2);
  t.bytes = (((size_t)5 << log2n2) + ((size_t)1 << log2n1)) * sizeof(double2);
  return t;
}

cudaError_t build_twiddles(int log2n1, int log2n2, void* base, cudaStream_t st) {
  const TwiddleTables t = twiddle_layout(log2n1, log2n2, base);
  roots((double2*)t.a, 1 << log2n2, log2n2, st);
  roots((double2*)t.b, 1 << log2n1, log2n1, st);
  double2* twist = (double2*)t.b + ((size_t)1 << log2n1);
  for (int p = 0; p < 4; ++p)
    roots(twist + ((size_t)p << log2n2), 1 << log2n2, log2n2 + pass_span_log2(log2n1, p), st);
  return cudaGetLastError();
}

}  // namespace fstat
