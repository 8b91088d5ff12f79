// Shape codes of the FFT passes (fstat_set_cta): which name a compiled shape,
// and what 0 stands for.
#include "fft_warp.cuh"

namespace fstat {

namespace {

// Columns or rows per CTA c that the CTA-wide passes offered at a length,
// with radix 16 or (odd schedules, 1024 points or more) 8 first: 32 to 1024
// threads and a padded buffer of at most 220 KB.  FP32 plans run the
// warp-local passes for all of them.
int first_radix(int log2_len, int v) {
  if (v & 1) return 8;
  return log2_len == 5 || log2_len == 6 || log2_len == 9 ? 8 : 16;
}
bool fits(int log2_len, int c, int v) {
  const int len = 1 << log2_len, r0 = first_radix(log2_len, v), threads = c * (len / r0);
  return threads >= 32 && threads <= 1024 && (int64_t)c * (len + len / r0) * 16 <= 220 * 1024;
}
bool offered(int log2_len, int c, int v, int max_c) {
  if (log2_len < 9 || ((v & 1) && log2_len < 10)) return false;
  return (c == 1 || c == 2 || c == 4 || c == 8) && c <= max_c && fits(log2_len, c, v);
}
// their default: 128 threads, at least two rows in pass B
int wide_default(int log2_len, bool pass_b) {
  const int tpc = (1 << log2_len) / first_radix(log2_len, 0), c = tpc >= 128 ? 1 : 128 / tpc;
  return pass_b && c < 2 ? 2 : c;
}

template <typename T, int L> int default_c(bool pass_b) {
  if (sizeof(T) == 4) return pass_b ? wpass_b_rows(fft::log2c(L), 0) : fft::WA<L>::COLS;
  return pass_b ? fft::Shape<double, L, 0>::CB_DEF : fft::Shape<double, L, 0>::CA_DEF;
}
template <typename T> int default_c_len(int log2_len, bool pass_b) {
  switch (log2_len) {
    case 5: return default_c<T, 32>(pass_b);
    case 6: return default_c<T, 64>(pass_b);
    case 7: return default_c<T, 128>(pass_b);
    case 8: return default_c<T, 256>(pass_b);
    case 9: return default_c<T, 512>(pass_b);
    case 10: return default_c<T, 1024>(pass_b);
    case 11: return default_c<T, 2048>(pass_b);
    case 12: return default_c<T, 4096>(pass_b);
    case 13: return pass_b ? 0 : 1;  // 8192-point columns: one per CTA
    default: return 0;
  }
}

}  // namespace

bool pass_a_shape(int log2_n2, int ca, int va) {
  if (va == 16 || va == 18) return log2_n2 == (va == 16 ? 13 : 12) && ca <= 1;
  const int def = log2_n2 == 13 ? 1 : wide_default(log2_n2, false);
  if (ca <= 0) ca = def;
  if (va == 0 && ca == def) return true;
  return offered(log2_n2, ca, va, 4) && (va != 10 || log2_n2 >= 10);
}
bool pass_b_shape(int log2_n1, int cb, int vb) {
  const int def = wide_default(log2_n1, true);
  if (cb <= 0) cb = def;
  if (vb == 0 && cb == def) return true;
  return log2_n1 <= 12 && offered(log2_n1, cb, vb, 8) && (vb <= 3 || log2_n1 >= 10);
}

int64_t pass_a_spacing(int log2n, int log2_n2) { return ((int64_t)1 << log2n) / fft::r_of(1 << log2_n2, 0, 0); }

// Columns (pass A, pass_b = 0) or rows (pass B) per CTA that shape 0 stands
// for at a pass length 2^log2_len.
int fft_default_c(int log2_len, int pass_b, int precision) {
  return precision == FSTAT_FP64 ? default_c_len<double>(log2_len, pass_b != 0)
                                 : default_c_len<float>(log2_len, pass_b != 0);
}

}  // namespace fstat
