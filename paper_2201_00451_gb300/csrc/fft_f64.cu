// FP64 (comparison path) instantiations of the FFT passes.
#include "fft_impl.cuh"

namespace fstat {

cudaError_t launch_pass_a_f64(int log2_n2, int ca, int va, const void* G, GCol gc, int64_t n, int n1, const void* twA,
                              const TmplCoef* coef, void* Z, cudaStream_t st, int res) {
  return fft::dispatch_a<double>(log2_n2, ca, va, G, gc, n, n1, twA, coef, Z, st, res);
}

cudaError_t launch_pass_b_f64(int log2_n1, int cb, int vb, const void* Z, int n2, const void* twB,
                              const SkyConst* sky, float* out, cudaStream_t st, const PeakArgs* pk, int res) {
  if (pk) return launch_pass_b_peak_f64(log2_n1, cb, vb, Z, n2, twB, sky, *pk, st, res);
  return fft::dispatch_b<double, fft::kStore>(log2_n1, cb, vb, Z, n2, twB, sky, out, PeakArgs{}, st, res);
}

}  // namespace fstat
