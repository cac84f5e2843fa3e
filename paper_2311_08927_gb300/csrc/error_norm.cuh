// Scaled error norm of the FP64 forms' embedded estimate,
//   max_i |k1 - 2 k2 + k3|_i / (atol_i + rtol max(|y_i|, |y1_i|)),
// in FP64, as the oracle's (besides the rounding of each ratio).
//
// The species with the largest ratio is found in FP32 on truncated high words,
// and its ratio alone formed in FP64: comparing 29 ratios in FP64 took five
// slots of the FP64 pipe per species.  Truncation (2^-20 in the error and in
// the scale), the approximate reciprocal and the roundings leave each FP32
// ratio within 1.3e-6 of the true one, so where no other comes within 1e-5 of
// the largest the choice is the right one.  Where one does (a near tie), where
// a scale or an error leaves the float range or all errors are next to nothing,
// and where a value is not finite, the ratios are compared in FP64 by cross
// products.  Not finite: an infinite norm.  60,000 particles FP64: 15.8 ms per
// call, 15.6 with the FP32 choice alone.
#pragma once
#include "adm1_device.cuh"

namespace chad {

// |d| as a float from its high word: truncated to 20 significand bits, below
// the normal float range zero, above it (and for infinities and NaN) infinite.
CHAD_HD float magf(double d) {
  int m = maghi(d) - 0x38000000;
  m = m < 0 ? 0 : m > 0x0ff00000 ? 0x0ff00000 : m;
  const unsigned u = (unsigned)m << 3;
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  memcpy(&f, &u, sizeof(f));
  return f;
#endif
}

// A copy that the compiler cannot tell from another value: the rare path below
// forms its errors anew instead of having them kept (and spilled) for it.
CHAD_HD double opaque(double x) {
#ifdef __CUDA_ARCH__
  asm volatile("" : "+d"(x));
#endif
  return x;
}

// The ratio of the species that sets the norm, by FP64 comparisons alone.
CHAD_HD double error_ratio_exact(const double* y, const double* y1, const double* k1,
                                 const double* k2, const double* k3, double rtol,
                                 const double* atol) {
  double en = 0.0, sn = 1.0;
  bool bad = false;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const double e = fabs(fma(-2.0, k2[i], opaque(k1[i])) + k3[i]), yi = opaque(y[i]);
    const double sc = fma(rtol, fabs(mag64(yi) > mag64(y1[i]) ? yi : y1[i]), atol[i]);
    bad = bad || mag64(e) >= kInfBits || mag64(sc) >= kInfBits;
    if (e * sn > en * sc) {
      en = e;
      sn = sc;
    }
  }
  return bad ? double(INFINITY) : en / sn;
}

CHAD_HD double error_ratio(const double* y, const double* y1, const double* k1, const double* k2,
                           const double* k3, double rtol, const double* atol) {
  double en = 0.0, ym = 0.0, at = 1.0;
  float best = 0.0f, next = 0.0f;  // the two largest ratios
  bool in_range = true;
  const float rt = cvt<float>(rtol);
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const double e = fma(-2.0, k2[i], k1[i]) + k3[i];
    const double yi = mag64(y[i]) > mag64(y1[i]) ? y[i] : y1[i];
    const float ef = magf(e), sc = fmaf(rt, magf(yi), magf(atol[i]));
    const float r = ef * rcp_approx(sc);
    in_range = in_range && sc >= 1e-30f && fmaxf(sc, ef) <= 1e30f;
    next = fmaxf(next, fminf(r, best));
    if (r > best) {
      best = r;
      en = e;
      ym = yi;
      at = atol[i];
    }
  }
  if (!in_range || !(best >= 1e-6f) || next >= best * (1.0f - 1e-5f))
    return error_ratio_exact(y, y1, k1, k2, k3, rtol, atol);
  return fabs(en) * rcp<double>(fma(rtol, fabs(ym), at));
}

}  // namespace chad
