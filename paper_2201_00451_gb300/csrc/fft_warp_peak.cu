// Warp-local FFT pass B (fft_warp.cuh) with 2F reduced in the kernel.
#include "fft_warp.cuh"

namespace fstat {

// pk: the call's request; template k of the launch is the call's template
// ord[k] (added to pk.tmpl, its band keys at pk.band_key + ord[k] n_bands),
// or the only one without ord.
cudaError_t launch_wpass_b_peak(int log2_n1, int cb, void* Z, int n_tmpl, int n2, const SkyConst* sky,
                                const int* ord, int n_bands, const PeakArgs& pk, int* err, int wait_limit,
                                cudaStream_t st, int res) {
  fft::WBArgs a{sky, nullptr, ord, 1, n_tmpl, n_bands, pk};
  if (!a.pk.err) a.pk.err = err;
  set_wait(a.pk, wait_limit);
  return fft::dispatch_wb<fft::kPeaks>(log2_n1, cb, (float4*)Z, n2, a, st, res);
}

}  // namespace fstat
