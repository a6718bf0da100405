// Which kernels transform a line: f_hat_l = sum_k e^{-2 pi i (k-1)(l-1)/n} f_k
// (eq. step1FFTfcoeff) and its inverse with 1/n (eq. step3IFFTz3coeff) go to
// the tensor-core product (short rows, by choice of the plan), to the
// power-of-two kernels, or to the mixed-radix ones (any other length).
#include <algorithm>

#include "helm_dft.h"
#include "helm_kernels.cuh"

namespace helm {

namespace {
// Primes up to this are passes of the mixed-radix kernels.
constexpr int kMaxGenericRadix = 64;
}  // namespace

bool dft_needs_bluestein(const DftPlan& p) {
  for (int s = 0; s < p.nstages; ++s)
    if (p.radix[s] > kMaxGenericRadix) return true;
  return false;
}

int64_t bluestein_length(int64_t n) {
  int64_t m = 1;
  while (m < 2 * n - 1) m <<= 1;
  return m;
}

bool dft_supported(const DftPlan& p, size_t elem_bytes, int max_smem) {
  if (dft_needs_bluestein(p)) {
    const int64_t m = bluestein_length(p.n);
    return m <= 8192 && (size_t)2 * m * elem_bytes <= (size_t)max_smem;
  }
  // two bare lines: all that the row kernels need (they pad them where there is room)
  return (size_t)2 * p.n * elem_bytes <= (size_t)max_smem;
}

cudaError_t launch_dft_rows(int prec, const void* in, int in_is_double, void* out, int out_mode,
                            int64_t nrows, const DftPlan& p, const void* tw, int sign, double scale,
                            double accum_scale, const void* sc_in, const void* sc_out, const int* skip,
                            cudaStream_t st, int* err) {
  // the tensor-core variant, for calls whose scalings are those its tables hold
  if (prec == kPrecF32 && p.gw[sign < 0 ? 0 : 1] && (in_is_double == kInC64 || in_is_double == kInC128) &&
      (out_mode == kOutC64 || out_mode == kOutC128 || out_mode == kOutAccumC128)) {
    const bool fwd = sign < 0;
    const bool same = fwd ? (sc_in == p.gsc[0] && !sc_out && scale == 1.0)
                          : (sc_out == p.gsc[1] && !sc_in && scale == p.gscale);
    if (same)
      return launch_dft_rows_tc(p.gw[fwd ? 0 : 1], p.n, in, in_is_double, out, out_mode, nrows, accum_scale, skip, st,
                                err);
  }
  if (dft_needs_bluestein(p) && !p.bm) return cudaErrorInvalidValue;  // large prime without its chirp tables
  if (dft_rows_pow2_supported(p.n))
    return launch_dft_rows_pow2(prec, in, in_is_double, out, out_mode, nrows, p.n, tw, sign, scale, accum_scale,
                                sc_in, sc_out, skip, st, err);
  return launch_dft_rows_mix(prec, in, in_is_double, out, out_mode, nrows, p, tw, sign, scale, accum_scale, sc_in,
                             sc_out, skip, st);
}

cudaError_t launch_dft_cols(int prec, const void* in, int in_is_double, void* out, int out_mode,
                            int64_t outer, int64_t inner, const DftPlan& p, const void* tw, int sign,
                            double scale, double accum_scale, const void* sc_in, const void* sc_out,
                            const int* skip, cudaStream_t st) {
  if (dft_needs_bluestein(p) && !p.bm) return cudaErrorInvalidValue;
  if (dft_cols_pow2_supported(p.n))
    return launch_dft_cols_pow2(prec, in, in_is_double, out, out_mode, outer, inner, p.n, tw, sign, scale,
                                accum_scale, sc_in, sc_out, skip, st);
  return launch_dft_cols_mix(prec, in, in_is_double, out, out_mode, outer, inner, p, tw, sign, scale, accum_scale,
                             sc_in, sc_out, skip, st);
}

}  // namespace helm
