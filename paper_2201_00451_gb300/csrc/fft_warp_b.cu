// Warp-local FFT pass B (fft_warp.cuh): dense 2F, and added to shifted rows.
#include "fft_warp.cuh"

namespace fstat {

namespace {
template <int L, int CB> ZLayout layout_of() {
  using S = fft::WB<L, CB>;
  return ZLayout{fft::log2c(CB), fft::log2c(S::RL), S::SUB};
}
template <int L> ZLayout layout_len(int cb) {
  switch (fft::wb_rows<L>(cb)) {
    case 1: return layout_of<L, 1>();
    case 2: return layout_of<L, 2>();
    case 4: return layout_of<L, 4>();
    case 8: return layout_of<L, 8>();
    default: return layout_of<L, fft::default_wcb<L>()>();
  }
}
}  // namespace

ZLayout wpass_z_layout(int log2_n1, int cb) {
  switch (log2_n1) {
    case 5: return layout_len<32>(cb);
    case 6: return layout_len<64>(cb);
    case 7: return layout_len<128>(cb);
    case 8: return layout_len<256>(cb);
    case 9: return layout_len<512>(cb);
    case 10: return layout_len<1024>(cb);
    case 11: return layout_len<2048>(cb);
    default: return layout_len<4096>(cb);
  }
}
int wpass_b_rows(int log2_n1, int cb) { return 1 << wpass_z_layout(log2_n1, cb).cb; }

cudaError_t launch_wpass_b(int log2_n1, int cb, void* Z, int n_tmpl, int n2, const SkyConst* sky, float* out,
                           const int* ord, int64_t out_rows, int* err, int wait_limit, cudaStream_t st, int res) {
  fft::WBArgs a{sky, out, ord, out_rows, n_tmpl, 0, PeakArgs{}};
  a.pk.err = err;
  set_wait(a.pk, wait_limit);
  return fft::dispatch_wb<fft::kStore>(log2_n1, cb, (float4*)Z, n2, a, st, res);
}

cudaError_t launch_wpass_b_acc(int log2_n1, int cb, void* Z, int n2, const SkyConst* sky, float* out, int shift,
                               bool first, int* err, int wait_limit, cudaStream_t st, int res) {
  fft::WBArgs a{sky, out, nullptr, 1, 1, 0, PeakArgs{}};
  a.pk.err = err;
  a.pk.shift = shift;
  a.pk.first = first;
  set_wait(a.pk, wait_limit);
  return fft::dispatch_wb<fft::kAccumulate>(log2_n1, cb, (float4*)Z, n2, a, st, res);
}

}  // namespace fstat
