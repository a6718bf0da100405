// Coefficients of the fixed-point residual as two 32-bit limbs (host).
#pragma once

#include <cmath>

namespace helm {

// h 2^32 + l, l signed.  l = -2^31 is among its values and has no 32-bit
// negative: a negated coefficient is split anew, never negated limb by limb.
struct Limb {
  int h, l;
};

// v 2^(62 - es), rounded, for |v| < 2^es (0 for an infinity or a NaN).
inline Limb fx_limb(double v, int es) {
  const long long c = std::isfinite(v) ? std::llround(std::ldexp(v, 62 - es)) : 0;
  const long long h = (c + (1ll << 31)) >> 32;
  return {(int)h, (int)(c - h * (1ll << 32))};
}

// A complex coefficient: real and imaginary part, and the latter's negative.
struct LimbC {
  Limb re, im, nim;
};
inline LimbC fx_limb_c(double re, double im, int es) {
  return {fx_limb(re, es), fx_limb(im, es), fx_limb(-im, es)};
}

}  // namespace helm
