// Warp-local FFT pass A (fft_warp.cuh) for every column length.
#include "fft_warp.cuh"

namespace fstat {

cudaError_t launch_wpass_a(int log2_n2, int staging, const void* G, GCol gc, int64_t n, int n1, const TmplCoef* coef,
                           void* Z, ZLayout zy, int n_tmpl, int* err, int wait_limit, cudaStream_t st, int res) {
  float4* z = (float4*)Z;
  const float4* g = (const float4*)G;
  switch (log2_n2) {
#define FSTAT_WA(B) \
  case B: return fft::run_wa<(1 << B)>(g, gc.lcs, n, n1, coef, z, zy, n_tmpl, staging, err, wait_limit, st, res);
    FSTAT_WA(5) FSTAT_WA(6) FSTAT_WA(7) FSTAT_WA(8) FSTAT_WA(9) FSTAT_WA(10) FSTAT_WA(11) FSTAT_WA(12) FSTAT_WA(13)
#undef FSTAT_WA
    default: return cudaErrorInvalidValue;
  }
}

// Residues of a column's sample index that G keeps together: the last radix.
int wpass_a_residues_log2(int log2_n2) {
  switch (log2_n2) {
    case 10: return fft::log2c(fft::WA<1024>::RL);
    case 11: return fft::log2c(fft::WA<2048>::RL);
    case 12: return fft::log2c(fft::WA<4096>::RL);
    case 13: return fft::log2c(fft::WA<8192>::RL);
    default: return 0;  // up to 512 points: the whole column in one warp
  }
}

}  // namespace fstat
