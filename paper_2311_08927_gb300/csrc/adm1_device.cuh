// Device-side ADM1 model for one particle per thread (Sec. 2.2-2.3).
//
//   * part_const   : temperature-dependent constants of a particle (van 't
//                    Hoff acid-base and Henry constants, Arrhenius kinetics).
//   * solve_SH     : Eq. 7 charge balance for S_H+ by Newton, with a
//                    bracketed geometric bisection fallback (FP64 always).
//   * model_f      : rate vector f(y) (Eq. 2 mass balances, Eq. 3-6 rates).
//   * model_fj     : f(y) and the analytic Jacobian df/dy, including the
//                    rank-1 coupling through S_H(y) given by the implicit
//                    function theorem on Eq. 7.
// R is the arithmetic type of rates, Jacobian and LU (double for the plain
// path, float for the mixed path); the charge balance is always FP64.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "model.h"

#ifndef CHAD_HD
#define CHAD_HD __host__ __device__ __forceinline__
#endif

namespace chad {

// Dense row-major storage of a NS x NS matrix (slot of entry (r, c)).
struct DenseIdx {
  static CHAD_HD constexpr int at(int r, int c) { return r * NS + c; }
  static constexpr int size = NS * NS;
};

// Conversions between binary64 and binary32 (IEEE 754).  On the GPU a
// hardware FP64<->FP32 conversion occupies the FP64 pipe as long as an FP64
// FMA (measured on GB300: both ~600 G lane-ops/s, the DFMA rate), so the
// device versions below work on the bit patterns with integer operations:
//   widen  (float -> double): exact for normal numbers; zero and subnormal
//          inputs give a signed zero; Inf and NaN keep their class.
//   narrow (double -> float): the significand truncated to 23 bits (round
//          toward zero, relative error below 2^-23); magnitudes below the
//          normal float range give a signed zero, above it +-Inf; NaN stays
//          NaN.
// Host code and other types use the plain casts.
template <class To, class From>
CHAD_HD To cvt(From x) {
  return To(x);
}
#ifdef __CUDA_ARCH__
template <>
__device__ __forceinline__ double cvt<double, float>(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xffu;
  const unsigned m = (e == 0u) ? 0u : (u & 0x7fffffu);
  const unsigned ee = (e == 0u) ? 0u : ((e == 0xffu) ? 0x7ffu : e + 896u);
  const unsigned hi = (u & 0x80000000u) | (ee << 20) | (m >> 3);
  return __hiloint2double((int)hi, (int)(m << 29));
}
template <>
__device__ __forceinline__ float cvt<float, double>(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned sgn = hi & 0x80000000u;
  const int E = (int)((hi >> 20) & 0x7ffu);
  const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
  const int e = E - 896;
  const bool nan = (E == 0x7ff) && (((hi & 0xfffffu) | lo) != 0u);
  unsigned u = sgn | ((unsigned)e << 23) | m;
  u = (e <= 0) ? sgn : u;
  u = (e >= 255) ? (sgn | 0x7f800000u | (nan ? 0x400000u : 0u)) : u;
  return __uint_as_float(u);
}
#endif

// 1/d.  On the GPU without branches, so that the some 170 reciprocals of a
// step attempt leave the straight-line code in one piece (the compiler can
// schedule across them and share equal ones).
//   FP64: the significand of d as a float in [1, 2), the hardware's
//     approximate FP32 reciprocal of it widened and rescaled by integer
//     operations into the seed r0 (relative error e = 1 - d r0 below 2^-21),
//     then one polynomial correction r0 (1 + e + e^2) of the Newton-Raphson
//     family for the reciprocal, whose relative error is O(e^3) (below
//     1e-18): three FMAs on the FP64 pipe.  |d| below 2^-1022 gives a
//     signed infinity, |d| from 2^1022 on a signed zero.  A NaN stays one as
//     long as its high word says so, which every operation's result does (a
//     payload in the low word alone would read as an infinity).
//   FP32: the approximate reciprocal and one Newton-Raphson step with the
//     residual from an FMA: correctly rounded for all normal d with a normal
//     reciprocal (all 2^32 arguments tested).  d = 0, infinite or NaN keeps
//     the approximation, which is exact there, and so do subnormal d (signed
//     infinity) and |d| above 2^126 (signed zero): the kernels' arguments are
//     sums with a half-saturation or scale constant, pivots near 1 and slopes.
// Elsewhere (host, counting types): the plain division.
template <class R>
CHAD_HD R rcp(R d) {
  return R(1) / d;
}
CHAD_HD float rcp_approx(float d) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
#else
  return 1.0f / d;
#endif
}
#ifdef __CUDA_ARCH__
template <>
__device__ __forceinline__ float rcp<float>(float d) {
  const float r = rcp_approx(d);
  const float e = fmaf(-d, r, 1.0f);
  const float x = fmaf(r, e, r);
  return fabsf(e) < 0.5f ? x : r;
}
template <>
__device__ __forceinline__ double rcp<double>(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned sgn = hi & 0x80000000u, mag = hi & 0x7fffffffu;
  const float m = __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29));
  const unsigned s = __float_as_uint(rcp_approx(m));  // in [1/2, 1]
  // exponents: the seed's (bias 127 -> 1023) minus that of d
  const unsigned rh = sgn | ((s >> 3) + 0x77f00000u - (mag & 0x7ff00000u));
  const double r = __hiloint2double((int)rh, (int)(s << 29));
  const double e = fma(-d, r, 1.0);
  const double x = fma(r, fma(e, e, e), r);
  // on the bit patterns: tiny -> infinity, huge or infinite -> zero
  const bool tiny = mag < 0x00100000u, huge = mag - 0x7fd00000u <= 0x00200000u;
  const unsigned xh = tiny ? (sgn | 0x7ff00000u) : huge ? sgn : (unsigned)__double2hiint(x);
  return __hiloint2double((int)xh, tiny || huge ? 0 : __double2loint(x));
}
#endif

// Threshold pivot test of the static-order LU: a pivot p is accepted when
// it is finite, nonzero and |p| >= 0.1 max_i |l_i| over its sub-column.
// key() maps an entry to a comparable magnitude, kmax() combines keys,
// good() takes the decision.  Host and counting types: the exact test.  On
// the GPU (FP64 and FP32) it runs on the IEEE-754 bit patterns with integer
// operations, because FP64 compares and min/max occupy the FP64 pipe: the
// sign-cleared pattern (the high word for a double) orders finite
// magnitudes like their values, and read as an integer it is a
// piecewise-linear log2 of the magnitude in units of 2^-20 (double high
// word) or 2^-23 (float), so the factor 0.1 becomes a shift by log2(10) in
// those units; the effective threshold is 0.1 up to the error of that
// linear log2, i.e. between 0.094 and 0.106.
template <class R>
struct PivTest {
  using K = R;
  static CHAD_HD K key(R x) { return fabs(x); }
  static CHAD_HD K kmax(K a, K b) { return fmax(a, b); }
  static CHAD_HD bool good(K p) { return p != R(0) && isfinite(p); }
  static CHAD_HD bool good(K p, K cm) { return good(p) && p >= R(0.1) * cm; }
};
#ifdef __CUDA_ARCH__
template <>
struct PivTest<double> {
  using K = unsigned;
  static __device__ __forceinline__ K key(double x) {
    return (unsigned)__double2hiint(x) & 0x7fffffffu;
  }
  static __device__ __forceinline__ K kmax(K a, K b) { return max(a, b); }
  static __device__ __forceinline__ bool good(K p) { return p != 0u && p < 0x7ff00000u; }
  static __device__ __forceinline__ bool good(K p, K cm) {
    return good(p) && p + 3483294u >= cm;  // log2(10) * 2^20
  }
};
template <>
struct PivTest<float> {
  using K = unsigned;
  static __device__ __forceinline__ K key(float x) { return __float_as_uint(x) & 0x7fffffffu; }
  static __device__ __forceinline__ K kmax(K a, K b) { return max(a, b); }
  static __device__ __forceinline__ bool good(K p) { return p != 0u && p < 0x7f800000u; }
  static __device__ __forceinline__ bool good(K p, K cm) {
    return good(p) && p + 27866353u >= cm;  // log2(10) * 2^23
  }
};
#endif

constexpr double kVfaCod_ac = 64.0, kVfaCod_pro = 112.0, kVfaCod_bu = 160.0, kVfaCod_va = 208.0;
constexpr double kC4Guard = 1e-6;  // division guard of the c4 uptake split
constexpr double kSH_lo = 1e-14, kSH_hi = 1.0;

template <class T>
struct PartConstT {
  T arr;  // Arrhenius factor of the kinetic constants
  T K_w, K_a_co2, K_a_IN, K_H_co2, K_H_ch4, K_H_h2, p_h2o, RT;
};
using PartConst = PartConstT<double>;
// float copy for FP32 rate evaluations (converted once per particle load
// instead of at every use)
using PartConstF = PartConstT<float>;
CHAD_HD void narrow_pc(const PartConst& q, PartConstF& f) {
  f.arr = float(q.arr);
  f.K_w = float(q.K_w);
  f.K_a_co2 = float(q.K_a_co2);
  f.K_a_IN = float(q.K_a_IN);
  f.K_H_co2 = float(q.K_H_co2);
  f.K_H_ch4 = float(q.K_H_ch4);
  f.K_H_h2 = float(q.K_H_h2);
  f.p_h2o = float(q.p_h2o);
  f.RT = float(q.RT);
}

CHAD_HD void part_const(const DigConst& c, double T, PartConst& q) {
  const double invT = 1.0 / T;
  const double dT = c.inv_T_base - invT;
  q.arr = exp(-c.Ea_over_R * (invT - c.inv_T_ref));
  q.K_w = c.K_w_b * exp(c.th_w * dT);
  q.K_a_co2 = c.K_a_co2_b * exp(c.th_a_co2 * dT);
  q.K_a_IN = c.K_a_IN_b * exp(c.th_a_IN * dT);
  q.K_H_co2 = c.K_H_co2_b * exp(c.th_H_co2 * dT);
  q.K_H_ch4 = c.K_H_ch4_b * exp(c.th_H_ch4 * dT);
  q.K_H_h2 = c.K_H_h2_b * exp(c.th_H_h2 * dT);
  q.p_h2o = c.p_h2o_b * exp(c.th_h2o * dT);
  q.RT = c.R * T;
}

// PartConst in structure-of-arrays form, field f of particle p at
// pc[f * ld + p]: computed once per load (the temperature of a particle is
// fixed while it is loaded) instead of by every lane that takes a new
// particle, which would leave the rest of its warp idle during nine FP64
// exponentials.
CHAD_HD void pc_store(const PartConst& q, double* pc, int64_t ld, int64_t p) {
  pc[0 * ld + p] = q.arr;
  pc[1 * ld + p] = q.K_w;
  pc[2 * ld + p] = q.K_a_co2;
  pc[3 * ld + p] = q.K_a_IN;
  pc[4 * ld + p] = q.K_H_co2;
  pc[5 * ld + p] = q.K_H_ch4;
  pc[6 * ld + p] = q.K_H_h2;
  pc[7 * ld + p] = q.p_h2o;
  pc[8 * ld + p] = q.RT;
}
CHAD_HD void pc_load(const double* pc, int64_t ld, int64_t p, PartConst& q) {
  q.arr = pc[0 * ld + p];
  q.K_w = pc[1 * ld + p];
  q.K_a_co2 = pc[2 * ld + p];
  q.K_a_IN = pc[3 * ld + p];
  q.K_H_co2 = pc[4 * ld + p];
  q.K_H_ch4 = pc[5 * ld + p];
  q.K_H_h2 = pc[6 * ld + p];
  q.p_h2o = pc[7 * ld + p];
  q.RT = pc[8 * ld + p];
}

// ----------------------------------------------------------- Eq. 7 (FP64)
struct AcidBase {
  double SH;     // root
  double dEdS;   // dE/dS_H at the root
  double r_IN, r_co2, r_ac, r_pro, r_bu, r_va;  // 1/(K_a + S_H) at the root
  double rS;     // 1/S_H
};

struct NewtonCounters {
  int iters;
  int fallbacks;
  int failed;
};

// The bit pattern of a double, its magnitude's pattern, and the high word of
// the latter: finite magnitudes order like their patterns, and on the GPU an
// FP64 compare takes an FP64 pipe slot where an integer compare does not.
CHAD_HD long long bits64(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long b;
  memcpy(&b, &x, sizeof(b));
  return b;
#endif
}
CHAD_HD long long mag64(double x) { return bits64(x) & 0x7fffffffffffffffll; }
CHAD_HD int maghi(double x) { return (int)(mag64(x) >> 32); }
constexpr long long kInfBits = 0x7ff0000000000000ll;
CHAD_HD bool pos_finite(double x) { return (unsigned long long)bits64(x) - 1ull < (unsigned long long)kInfBits - 1ull; }
// |t| <= 2^-18 |S| to within the piecewise-linear log2 of the patterns (6 %)
CHAD_HD bool third_order_close(double t, double S) { return maghi(t) + (18 << 20) <= maghi(S); }

// Eq. 7 with the products that do not change with S_H formed once per solve:
//   E(S) = base + S - sum_k P_k / (K_k + S) - K_w / S
// over IN, co2, ac, pro, bu, va (P = K_a times the concentration in charge
// equivalents).
template <class F>
struct ChargeBalT {
  F base, P[6];
};
using ChargeBal = ChargeBalT<double>;
template <class F>
CHAD_HD void charge_bal(const DigConst& c, const PartConst& q, const double* y, ChargeBalT<F>& e) {
  e.base = (F(y[iS_cat]) - F(y[iS_an])) + F(y[iS_IN]);
  e.P[0] = F(q.K_a_IN) * F(y[iS_IN]);
  e.P[1] = F(q.K_a_co2) * F(y[iS_IC]);
  e.P[2] = F(c.K_a_ac) * F(y[iS_ac]) * F(1.0 / kVfaCod_ac);
  e.P[3] = F(c.K_a_pro) * F(y[iS_pro]) * F(1.0 / kVfaCod_pro);
  e.P[4] = F(c.K_a_bu) * F(y[iS_bu]) * F(1.0 / kVfaCod_bu);
  e.P[5] = F(c.K_a_va) * F(y[iS_va]) * F(1.0 / kVfaCod_va);
}
// E and dE/dS from the reciprocals rS = 1/S and r_k = 1/(K_k + S).  The
// routines of the balance are templates on the scalar type so that their
// operations can be counted on the host.
template <class F>
CHAD_HD F charge_sums(const ChargeBalT<F>& e, F K_w, F S, F rS, const F* r, F& dEdS) {
  const F kw = K_w * rS;
  F E = (e.base - kw) + S, d = F(1.0) + kw * rS;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const F t = e.P[k] * r[k];
    E = E - t;
    d = d + t * r[k];
  }
  dEdS = d;
  return E;
}
// E and dE/dS at S with the reciprocals.
template <class F>
CHAD_HD F charge_eval(const DigConst& c, const PartConst& q, const ChargeBalT<F>& e, F S, F* r,
                      F& rS, F& dEdS) {
  rS = rcp<F>(S);
  r[0] = rcp<F>(F(q.K_a_IN) + S);
  r[1] = rcp<F>(F(q.K_a_co2) + S);
  r[2] = rcp<F>(F(c.K_a_ac) + S);
  r[3] = rcp<F>(F(c.K_a_pro) + S);
  r[4] = rcp<F>(F(c.K_a_bu) + S);
  r[5] = rcp<F>(F(c.K_a_va) + S);
  return charge_sums<F>(e, F(q.K_w), S, rS, r, dEdS);
}
// Chebyshev's third-order correction at a Newton update t = E inv, inv =
// 1/E': the move d of the root, -t + t^2 h / E' with h = -E''/2.
template <class F>
CHAD_HD F charge_step(const ChargeBalT<F>& e, F K_w, F rS, const F* r, F t, F inv) {
  F h = K_w * rS * (rS * rS);
#pragma unroll
  for (int k = 0; k < 6; ++k) h = h + e.P[k] * r[k] * (r[k] * r[k]);
  return t * (t * (h * inv)) - t;
}
// The reciprocals moved from S to S + d to second order in x = r d,
// 1/(K + S + d) = r / (1 + x) = r (1 - x + x^2 - ..), and dE/dS there.
template <class F>
CHAD_HD void charge_move(const ChargeBalT<F>& e, F K_w, F S, F d, F* r, F& rS, F& dEdS) {
  F x = rS * d;
  rS = rS + rS * (x * x - x);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    x = r[k] * d;
    r[k] = r[k] + r[k] * (x * x - x);
  }
  charge_sums<F>(e, K_w, S + d, rS, r, dEdS);
}
CHAD_HD void charge_fill(AcidBase& ab, double SH, double rS, const double* r, double dEdS) {
  ab.SH = SH;
  ab.dEdS = dEdS;
  ab.rS = rS;
  ab.r_IN = r[0];
  ab.r_co2 = r[1];
  ab.r_ac = r[2];
  ab.r_pro = r[3];
  ab.r_bu = r[4];
  ab.r_va = r[5];
}

// Newton from `guess` without a fallback: true if it converged within
// max_iters with |E| <= max_resid at the returned root (ab then describes
// it).  E is increasing and concave, Newton converges quadratically with a
// relative contraction factor below 1 near the root: an update below 1e-8
// relative leaves the new iterate within ~1e-16 of the root.
__host__ __device__ inline bool newton_only(const DigConst& c, const PartConst& q,
                                            const double* y, double guess, int max_iters,
                                            double max_resid, AcidBase& ab, int& iters) {
  ChargeBal cb;
  charge_bal<double>(c, q, y, cb);
  double S = (guess > 0.0 && isfinite(guess)) ? guess : 1e-7;
  double prevE = INFINITY, Ec = INFINITY;
  bool last = false;
  for (int it = 0;; ++it) {
    double r[6], rS, dE;
    const double E = charge_eval<double>(c, q, cb, S, r, rS, dE);
    if (last) {  // at the root: the residual bound
      charge_fill(ab, S, rS, r, dE);
      return fabs(E) <= max_resid || Ec <= max_resid;
    }
    if (it >= max_iters) return false;
    iters++;
    if (!isfinite(E) || fabs(E) > fabs(prevE)) return false;
    const double dS = E * rcp<double>(dE);
    const double Sn = S - dS;
    if (!(Sn > 0.0) || !isfinite(Sn)) return false;
    last = fabs(dS) <= 1e-8 * Sn || fabs(E) <= 1e-15;
    Ec = fabs(E);
    prevE = E;
    S = Sn;
  }
}

// Root of Eq. 7: Newton from `guess`; an iterate leaving (0, inf) or a
// growing |E| switches to a bracket on [1e-14, 1].  One loop around a single
// evaluation of Eq. 7: each evaluation inlines seven reciprocals, and one
// copy keeps the integrator's code within reach of the instruction cache.
//   * A Newton update t with |t| <= 2^-18 S ends the solve with the
//     third-order step of Chebyshev, S - t + t^2 h / E' with h = -E''/2 =
//     sum P r^3 + K_w / S^3: |E''/E'| <= 2/S and its higher relatives bound
//     the remainder by a few (t/S)^3, below 1e-16.  The reciprocals move
//     with the root, 1/(K + S + d) = r (1 - x + x^2) with x = r d and
//     relative error x^3.  Plain Newton would need another evaluation (75
//     FP64 instructions) in nearly every warp, since some lane's tangent
//     guess is off by more than 1e-8.
//   * Bracket: geometric midpoints halve its ratio's logarithm until
//     hi <= 4 lo, then Newton inside it (E is increasing and concave: from
//     the left Newton climbs to the root without passing it).  A dozen
//     evaluations, where bisection to the last bit took over fifty.
__host__ __device__ inline void solve_SH(const DigConst& c, const PartConst& q, const double* y,
                                         double guess, int max_iters, AcidBase& ab,
                                         NewtonCounters& nc) {
  enum { kNewton, kLo, kHi, kBracket, kFinal };
  ChargeBal cb;
  charge_bal<double>(c, q, y, cb);
  const double start = pos_finite(guess) ? guess : 1e-7;
  int phase = max_iters > 0 ? kNewton : kLo;
  if (phase == kLo) nc.fallbacks++;
  double S = phase == kNewton ? start : kSH_lo;  // point of the next evaluation
  long long prevE = kInfBits;
  double lo = kSH_lo, hi = kSH_hi;
  bool lo_neg = false;
  int it = 0;
  for (;;) {
    double r[6], rS, dE;
    const double E = charge_eval<double>(c, q, cb, S, r, rS, dE);
    const double inv = rcp<double>(dE);
    const double t = E * inv;
    bool done = phase == kFinal;
    double d = 0.0;
    if (phase == kNewton || phase == kBracket) {
      const long long mE = mag64(E);
      const bool close = mE < kInfBits && third_order_close(t, S);
      if (phase == kNewton) nc.iters++;
      if (close && !(phase == kNewton && mE > prevE)) {
        d = charge_step<double>(cb, q.K_w, rS, r, t, inv);
        done = true;
      } else if (phase == kNewton) {
        const double Sn = S - t;
        bool fail = mE >= kInfBits || mE > prevE || !pos_finite(Sn);
        if (!fail) {
          prevE = mE;
          S = Sn;
          fail = ++it >= max_iters;
        }
        if (fail) {
          nc.fallbacks++;
          phase = kLo;
          S = lo;
        }
      } else {
        ++it;
        if (bits64(E) < 0) lo = S; else hi = S;
        const double mid = sqrt(lo * hi), Sn = S - t;
        if (it >= 200 || !(mid > lo && mid < hi)) {
          phase = kFinal;
          S = mid;
        } else {
          S = hi <= 4.0 * lo && Sn > lo && Sn < hi ? Sn : mid;
        }
      }
    } else if (phase == kLo) {
      lo_neg = E < 0.0;
      phase = kHi;
      S = hi;
    } else if (phase == kHi) {
      if (!(lo_neg && E > 0.0)) {  // no sign change: keep the guess
        nc.failed = 1;
        phase = kFinal;
        S = start;
      } else {
        phase = kBracket;
        it = 0;
        S = sqrt(lo * hi);
      }
    }
    if (done) {
      charge_move<double>(cb, q.K_w, S, d, r, rS, dE);
      charge_fill(ab, S + d, rS, r, dE);
      return;
    }
  }
}

// dS_H/dy_k = -(dE/dy_k) / (dE/dS_H) (implicit function theorem on Eq. 7)
// for the 8 states that enter Eq. 7, in the order of kShStates.
constexpr int kShStates[8] = {iS_va, iS_bu, iS_pro, iS_ac, iS_IC, iS_IN, iS_cat, iS_an};
template <class DC, class PQ>
CHAD_HD void sh_tangent(const DC& c, const PQ& q, const AcidBase& ab, double* v) {
  const double inv = -rcp<double>(ab.dEdS);
  v[0] = inv * (-c.K_a_va * ab.r_va * (1.0 / kVfaCod_va));
  v[1] = inv * (-c.K_a_bu * ab.r_bu * (1.0 / kVfaCod_bu));
  v[2] = inv * (-c.K_a_pro * ab.r_pro * (1.0 / kVfaCod_pro));
  v[3] = inv * (-c.K_a_ac * ab.r_ac * (1.0 / kVfaCod_ac));
  v[4] = inv * (-q.K_a_co2 * ab.r_co2);
  v[5] = inv * (ab.SH * ab.r_IN);
  v[6] = inv;
  v[7] = -inv;
}

// ----------------------------------------------------------- inhibition helpers
// Hill pH inhibition I = 1 / (1 + (S/K)^n) and dI/dS
template <class R>
CHAD_HD void hill(R S, R invK, R n, int ni, R& I, R& dI) {
  const R x = S * invK;
  R xn1, xn;
  switch (ni) {
    case 1: xn1 = R(1); xn = x; break;
    case 2: xn1 = x; xn = x * x; break;
    case 3: xn1 = x * x; xn = xn1 * x; break;
    case 4: xn1 = x * x * x; xn = xn1 * x; break;
    default: xn = pow(x, n); xn1 = xn / x; break;
  }
  I = rcp<R>(R(1) + xn);
  dI = -n * xn1 * invK * I * I;
}

// ----------------------------------------------------------- Eq. 8 (FP64)
// S_h2 as an algebraic variable: its mass balance (Eq. 8) as a function of
// S_h2 alone, every other state and S_H fixed.  These are the hydrogen terms
// of rates() and balances() written out: the fa, c4 and pro uptakes carry
// the inhibition K_I/(K_I + S_h2), the hydrogen uptake the Monod factor
// S_h2/(K_S + S_h2), the transfer and the outflow are linear, so
//   E(S) = C0 + P_fa I_fa(S) + P_c4 I_c4(S) + P_pro I_pro(S) - P_h2 M(S) - kD S
// with P >= 0: E decreases in S and the root is unique.
template <class F>
struct H2Bal {
  F C0, Pfa, Pc4, Ppro, Ph2, kD, Kfa, Kc4, Kpro, Kh2;  // Pfa, Pc4, Ppro: times their K in FP64
};

// Factors of the rates that do not hold S_h2 (Eq. 3-6 inhibitions and Monod
// terms): formed once per evaluation point and shared by the Eq. 8 balance
// and the rates, ten reciprocals and about 60 operations fewer than forming
// them in both.  In FP64, B5 and B12 carry the Arrhenius factor (one product
// instead of one per rate constant).  FP32 products keep the association that
// they have had: the mixed forms' error estimates, and with them the choice
// of a step, hang on the last bits of the FP32 rates.  The FP64 forms are
// bound by the FP64 pipe, one warp instruction per 64 cycles and
// sub-partition, so each instruction saved counts: with the partials below
// and the products of structural zeros left out, 100,000 particles in the
// shared-headspace cylinder take 54.5 ms instead of 58.0, ten fixed substeps
// of 111,000 particles 8.54 instead of 9.18.
template <class R>
constexpr bool is_f32() {
  return std::is_same<R, float>::value;
}
template <class R>
struct Factors {
  R Ipaa, dIpaa, Iph2, dIph2;  // pH inhibitions (the aa form also of su, fa, c4, pro)
  R rIN, IIN;
  R rsu, raa, rfs, rva, rbu, rpo;  // 1/(K_S + S)
  R msu, maa, mfa, mva, mbu, mpo;  // Monod terms
  R rden, gva, gbu;                // c4 uptake split
  R B5, B12;                       // arr I_pH I_IN
};

template <class R, class DC, class PQ, class Y>
CHAD_HD void factors(const DC& c, const PQ& q, const Y* y, const AcidBase& ab, Factors<R>& k) {
  hill<R>(R(ab.SH), R(c.inv_K_pH_aa), R(c.n_aa), c.ni_aa, k.Ipaa, k.dIpaa);
  hill<R>(R(ab.SH), R(c.inv_K_pH_h2), R(c.n_h2), c.ni_h2, k.Iph2, k.dIph2);
  const R S_IN = R(y[iS_IN]), S_va = R(y[iS_va]), S_bu = R(y[iS_bu]);
  k.rIN = rcp<R>(S_IN + R(c.K_S_IN));
  k.IIN = S_IN * k.rIN;
  k.rsu = rcp<R>(R(c.K_S_su) + R(y[iS_su]));
  k.raa = rcp<R>(R(c.K_S_aa) + R(y[iS_aa]));
  k.rfs = rcp<R>(R(c.K_S_fa) + R(y[iS_fa]));
  k.rva = rcp<R>(R(c.K_S_c4) + S_va);
  k.rbu = rcp<R>(R(c.K_S_c4) + S_bu);
  k.rpo = rcp<R>(R(c.K_S_pro) + R(y[iS_pro]));
  k.msu = R(y[iS_su]) * k.rsu;
  k.maa = R(y[iS_aa]) * k.raa;
  k.mfa = R(y[iS_fa]) * k.rfs;
  k.mva = S_va * k.rva;
  k.mbu = S_bu * k.rbu;
  k.mpo = R(y[iS_pro]) * k.rpo;
  k.rden = rcp<R>(S_bu + S_va + R(kC4Guard));
  k.gva = S_va * k.rden;
  k.gbu = S_bu * k.rden;
  const R aN = is_f32<R>() ? k.IIN : R(q.arr) * k.IIN;
  k.B5 = k.Ipaa * aN;
  k.B12 = k.Iph2 * aN;
}

template <class F, class DC, class PQ, class Y>
CHAD_HD void h2_coeffs(const DC& c, const PQ& q, const Y* y, F D, const Factors<F>& k,
                       H2Bal<F>& e) {
  const F kLa = F(c.k_La);
  const F KH2 = F(q.K_H_h2) * F(q.RT);
  if constexpr (is_f32<F>()) {
    const F a = F(q.arr);
    const F r4 = F(c.k_m_su) * a * F(y[iX_su]) * k.msu * k.B5;
    const F r5 = F(c.k_m_aa) * a * F(y[iX_aa]) * k.maa * k.B5;
    e.C0 = D * F(c.y_in[iS_h2]) + F(c.su_h2) * r4 + F(c.aa_h2) * r5 + kLa * KH2 * F(y[iG_h2]);
    e.Pfa = F(c.fa_h2) * F(c.k_m_fa) * a * F(y[iX_fa]) * k.mfa * k.B5;
    e.Pc4 = (F(c.va_h2) * k.mva * k.gva + F(c.bu_h2) * k.mbu * k.gbu) * F(c.k_m_c4) * a * F(y[iX_c4]) * k.B5;
    e.Ppro = F(c.pro_h2) * F(c.k_m_pro) * a * F(y[iX_pro]) * k.mpo * k.B5;
    e.Ph2 = F(c.k_m_h2) * a * F(y[iX_h2]) * k.B12;
  } else {
    const F r4 = F(c.k_m_su) * F(y[iX_su]) * k.msu;
    const F r5 = F(c.k_m_aa) * F(y[iX_aa]) * k.maa;
    e.C0 = D * F(c.y_in[iS_h2]) + (F(c.su_h2) * r4 + F(c.aa_h2) * r5) * k.B5 + kLa * KH2 * F(y[iG_h2]);
    e.Pfa = F(c.fa_h2) * (F(c.k_m_fa) * F(y[iX_fa]) * k.mfa) * k.B5 * F(c.K_I_h2_fa);
    e.Pc4 = (F(c.va_h2) * (k.mva * k.gva) + F(c.bu_h2) * (k.mbu * k.gbu)) *
            (F(c.k_m_c4) * F(y[iX_c4])) * k.B5 * F(c.K_I_h2_c4);
    e.Ppro = F(c.pro_h2) * (F(c.k_m_pro) * F(y[iX_pro]) * k.mpo) * k.B5 * F(c.K_I_h2_pro);
    e.Ph2 = F(c.k_m_h2) * F(y[iX_h2]) * k.B12;
  }
  e.kD = kLa + D;
  e.Kfa = F(c.K_I_h2_fa);
  e.Kc4 = F(c.K_I_h2_c4);
  e.Kpro = F(c.K_I_h2_pro);
  e.Kh2 = F(c.K_S_h2);
}

// E(S) and dE/dS of Eq. 8 from the coefficients; h (may be null; FP64)
// receives E''/2.
template <class F>
CHAD_HD F h2_eval(const H2Bal<F>& e, F S, F& dE, F* h = nullptr) {
  const F rfa = rcp<F>(e.Kfa + S), rc4 = rcp<F>(e.Kc4 + S), rpr = rcp<F>(e.Kpro + S);
  const F rh = rcp<F>(e.Kh2 + S);
  if constexpr (is_f32<F>()) {
    const F Ifa = e.Kfa * rfa, Ic4 = e.Kc4 * rc4, Ipr = e.Kpro * rpr;
    dE = F(0) - (e.Pfa * Ifa * rfa + e.Pc4 * Ic4 * rc4 + e.Ppro * Ipr * rpr +
                 e.Ph2 * e.Kh2 * rh * rh + e.kD);
    return e.C0 + e.Pfa * Ifa + e.Pc4 * Ic4 + e.Ppro * Ipr - e.Ph2 * S * rh - e.kD * S;
  }
  const F tfa = e.Pfa * rfa, tc4 = e.Pc4 * rc4, tpr = e.Ppro * rpr, th = e.Ph2 * rh;
  const F dfa = tfa * rfa, dc4 = tc4 * rc4, dpr = tpr * rpr, dh = th * (e.Kh2 * rh);
  dE = F(0) - (dfa + dc4 + dpr + dh + e.kD);
  if (h) *h = dfa * rfa + dc4 * rc4 + dpr * rpr + dh * rh;
  return e.C0 + tfa + tc4 + tpr - (th + e.kD) * S;
}

// Root of Eq. 8 by Newton from the guess, ended by Chebyshev's third-order
// step as in solve_SH (|E''/E'| <= 2/S here too).  An iterate leaving (0,
// inf), a growing |E| or a non-negative slope switches to bisection on [0,
// hi], hi doubled from the guess until E(hi) <= 0 (E decreases, and E(0) >=
// 0: at S = 0 nothing removes hydrogen but the transfer from a gas that
// holds some).
__host__ __device__ inline double solve_h2(const H2Bal<double>& e, double guess, int max_iters,
                                           NewtonCounters& nc) {
  double S = pos_finite(guess) ? guess : 1e-8;
  long long prevE = kInfBits;
  for (int it = 0; it < max_iters; ++it) {
    double dE, h;
    const double E = h2_eval<double>(e, S, dE, &h);
    const long long mE = mag64(E);
    nc.iters++;
    if (mE >= kInfBits || mE > prevE || bits64(dE) >= 0 || mag64(dE) > kInfBits) break;
    const double inv = rcp<double>(dE);
    const double t = E * inv;
    if (third_order_close(t, S)) return S - t - t * (t * (h * inv));
    const double Sn = S - t;
    if (!pos_finite(Sn)) break;
    prevE = mE;
    S = Sn;
  }
  nc.fallbacks++;
  double lo = 0.0, hi = fmax(pos_finite(guess) ? guess : 0.0, 1e-12), dE;
  int k = 0;
  while (k < 200 && h2_eval<double>(e, hi, dE) > 0.0) {
    hi *= 2.0;
    ++k;
  }
  if (k == 200) {
    nc.failed = 1;
    return pos_finite(guess) ? guess : 1e-8;
  }
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (!(mid > lo && mid < hi)) break;
    if (h2_eval<double>(e, mid, dE) > 0.0) lo = mid; else hi = mid;
  }
  return 0.5 * (lo + hi);
}

// Rates of the 19 biochemical processes, the 3 transfers and their partial
// derivatives.  Column lists are fixed per process.
template <class R>
struct Rates {
  R r[22];
  // partials (d*) -- only filled by the Jacobian variant
  R d1, d2, d3, d4;                                   // wrt X_c, X_ch, X_pr, X_li
  R d5[3], d6[3], d7[4], d8[5], d9[5], d10[4], d11[3], d12[3];
  R s5, s6, s7, s8, s9, s10, s11, s12;                // wrt S_H
  R ddec[7];
  R dT8[2], dT9[2], dT10[2], sT10;
  R qv, qvs, dqv;                                     // q_gas/V_gas (qvs scaled), its dP derivative
  R P_h2, P_ch4, P_co2;                               // dP/dG
};

// k: the factors at y (factors()).  J: the partials too, multiplied by sc
// (the FP64 forms take sc = -g, so that the Jacobian scatter yields -g J_d
// and -g u): sc goes into the few factors that all partials of a process
// share instead of multiplying each of some 60 partials.
template <class R, bool J, class DC, class PQ>
CHAD_HD void rates(const DC& c, const PQ& q, const R* y, const AcidBase& ab, const Factors<R>& k,
                   Rates<R>& o, R sc = R(1)) {
  const R a = R(q.arr);
  const R SH = R(ab.SH);
  R Ipac, dIpac;
  hill<R>(SH, R(c.inv_K_pH_ac), R(c.n_ac), c.ni_ac, Ipac, dIpac);
  const R S_IN = y[iS_IN], S_h2 = y[iS_h2];
  const R rfa = rcp<R>(R(c.K_I_h2_fa) + S_h2), rc4 = rcp<R>(R(c.K_I_h2_c4) + S_h2);
  const R rpr = rcp<R>(R(c.K_I_h2_pro) + S_h2);
  const R Ih2fa = R(c.K_I_h2_fa) * rfa, Ih2c4 = R(c.K_I_h2_c4) * rc4, Ih2pro = R(c.K_I_h2_pro) * rpr;
  const R r_nh3 = R(q.K_a_IN) * R(ab.r_IN);
  const R nh3 = r_nh3 * S_IN;  // free ammonia
  const R rnh = rcp<R>(R(c.K_I_nh3) + nh3);
  const R Inh3 = R(c.K_I_nh3) * rnh;

  // first-order processes
  const R kdis = R(c.k_dis) * a, kch = R(c.k_hyd_ch) * a, kpr = R(c.k_hyd_pr) * a,
          kli = R(c.k_hyd_li) * a;
  o.r[0] = kdis * y[iX_c];
  o.r[1] = kch * y[iX_ch];
  o.r[2] = kpr * y[iX_pr];
  o.r[3] = kli * y[iX_li];
  // uptakes: p = k_m X x Monod terms, the rate p B
  const R rac = rcp<R>(R(c.K_S_ac) + y[iS_ac]), rh2 = rcp<R>(R(c.K_S_h2) + S_h2);
  const R mac = y[iS_ac] * rac, mh2 = S_h2 * rh2;
  const R B7 = k.B5 * Ih2fa, B8 = k.B5 * Ih2c4, B10 = k.B5 * Ih2pro;
  // the Arrhenius factor: in the rate constants (FP32) or in the B (FP64)
  const R aK = is_f32<R>() ? a : R(1), aB = is_f32<R>() ? R(1) : a;
  const R B11 = Ipac * (aB * k.IIN) * Inh3;
  const R ksu = R(c.k_m_su) * aK, kaa = R(c.k_m_aa) * aK, kfa = R(c.k_m_fa) * aK,
          kc4 = R(c.k_m_c4) * aK, kpo = R(c.k_m_pro) * aK, kac = R(c.k_m_ac) * aK,
          kh2 = R(c.k_m_h2) * aK;
  const R A5 = ksu * y[iX_su], A6 = kaa * y[iX_aa], A7 = kfa * y[iX_fa], A8 = kc4 * y[iX_c4];
  const R A10 = kpo * y[iX_pro], A11 = kac * y[iX_ac], A12 = kh2 * y[iX_h2];
  const R tva = k.mva * k.gva, tbu = k.mbu * k.gbu;
  const R p5 = A5 * k.msu, p6 = A6 * k.maa, p7 = A7 * k.mfa;
  const R p8 = is_f32<R>() ? A8 * k.mva * k.gva : A8 * tva;
  const R p9 = is_f32<R>() ? A8 * k.mbu * k.gbu : A8 * tbu;
  const R p10 = A10 * k.mpo, p11 = A11 * mac, p12 = A12 * mh2;
  o.r[4] = p5 * k.B5;
  o.r[5] = p6 * k.B5;
  o.r[6] = p7 * B7;
  o.r[7] = p8 * B8;
  o.r[8] = p9 * B8;
  o.r[9] = p10 * B10;
  o.r[10] = p11 * B11;
  o.r[11] = p12 * k.B12;
  R kd[7];
#pragma unroll
  for (int i = 0; i < 7; ++i) {
    kd[i] = R(c.k_dec[i]) * a;
    o.r[12 + i] = kd[i] * y[iX_su + i];
  }
  // gas phase
  const R RT = R(q.RT);
  const R P_h2 = RT * R(1.0 / 16.0), P_ch4 = RT * R(1.0 / 64.0), P_co2 = RT;
  const R P = P_h2 * y[iG_h2] + P_ch4 * y[iG_ch4] + P_co2 * y[iG_co2] + R(q.p_h2o);
  const R kpv = R(c.kp_over_Vgas), invPa = rcp<R>(R(c.P_atm));
  o.qv = kpv * (P - R(c.P_atm)) * P * invPa;
  const R kLa = R(c.k_La);
  const R KH2 = R(q.K_H_h2) * RT, KCH4 = R(q.K_H_ch4) * RT, KCO2 = R(q.K_H_co2) * RT;
  const R rco2 = R(ab.r_co2);
  const R fco2 = SH * rco2;  // S_co2 / S_IC
  o.r[19] = kLa * (S_h2 - KH2 * y[iG_h2]);
  o.r[20] = kLa * (y[iS_ch4] - KCH4 * y[iG_ch4]);
  o.r[21] = kLa * (y[iS_IC] * fco2 - KCO2 * y[iG_co2]);

  if constexpr (J && is_f32<R>()) {
    // FP32 partials (sc is 1 here), each product associated from the left
    const R dIIN = R(c.K_S_IN) * k.rIN * k.rIN;
    o.d1 = kdis; o.d2 = kch; o.d3 = kpr; o.d4 = kli;
    // rho5: S_su, X_su, S_IN
    o.d5[0] = A5 * (R(c.K_S_su) * k.rsu * k.rsu) * k.B5;
    o.d5[1] = ksu * k.msu * k.B5;
    o.d5[2] = A5 * k.msu * k.Ipaa * dIIN;
    o.s5 = A5 * k.msu * k.dIpaa * k.IIN;
    // rho6: S_aa, X_aa, S_IN
    o.d6[0] = A6 * (R(c.K_S_aa) * k.raa * k.raa) * k.B5;
    o.d6[1] = kaa * k.maa * k.B5;
    o.d6[2] = A6 * k.maa * k.Ipaa * dIIN;
    o.s6 = A6 * k.maa * k.dIpaa * k.IIN;
    // rho7: S_fa, X_fa, S_IN, S_h2
    o.d7[0] = A7 * (R(c.K_S_fa) * k.rfs * k.rfs) * B7;
    o.d7[1] = kfa * k.mfa * B7;
    o.d7[2] = A7 * k.mfa * k.Ipaa * dIIN * Ih2fa;
    o.d7[3] = -A7 * k.mfa * k.B5 * Ih2fa * rfa;   // dI/dS_h2 = -K/(K+S)^2 = -I r
    o.s7 = A7 * k.mfa * k.dIpaa * k.IIN * Ih2fa;
    // rho8, rho9: S_va, S_bu, X_c4, S_IN, S_h2
    const R rd2 = k.rden * k.rden;
    const R dgva_va = (y[iS_bu] + R(kC4Guard)) * rd2, dgva_bu = -y[iS_va] * rd2;
    const R dgbu_bu = (y[iS_va] + R(kC4Guard)) * rd2, dgbu_va = -y[iS_bu] * rd2;
    const R dmva = R(c.K_S_c4) * k.rva * k.rva, dmbu = R(c.K_S_c4) * k.rbu * k.rbu;
    o.d8[0] = A8 * B8 * (dmva * k.gva + k.mva * dgva_va);
    o.d8[1] = A8 * B8 * k.mva * dgva_bu;
    o.d8[2] = kc4 * k.mva * k.gva * B8;
    o.d8[3] = A8 * k.mva * k.gva * k.Ipaa * dIIN * Ih2c4;
    o.d8[4] = -A8 * k.mva * k.gva * k.B5 * Ih2c4 * rc4;
    o.s8 = A8 * k.mva * k.gva * k.dIpaa * k.IIN * Ih2c4;
    o.d9[0] = A8 * B8 * k.mbu * dgbu_va;
    o.d9[1] = A8 * B8 * (dmbu * k.gbu + k.mbu * dgbu_bu);
    o.d9[2] = kc4 * k.mbu * k.gbu * B8;
    o.d9[3] = A8 * k.mbu * k.gbu * k.Ipaa * dIIN * Ih2c4;
    o.d9[4] = -A8 * k.mbu * k.gbu * k.B5 * Ih2c4 * rc4;
    o.s9 = A8 * k.mbu * k.gbu * k.dIpaa * k.IIN * Ih2c4;
    // rho10: S_pro, X_pro, S_IN, S_h2
    o.d10[0] = A10 * (R(c.K_S_pro) * k.rpo * k.rpo) * B10;
    o.d10[1] = kpo * k.mpo * B10;
    o.d10[2] = A10 * k.mpo * k.Ipaa * dIIN * Ih2pro;
    o.d10[3] = -A10 * k.mpo * k.B5 * Ih2pro * rpr;
    o.s10 = A10 * k.mpo * k.dIpaa * k.IIN * Ih2pro;
    // rho11: S_ac, X_ac, S_IN (I_IN and free ammonia)
    const R dInh3 = -Inh3 * rnh;  // dI_nh3 / dS_nh3
    o.d11[0] = A11 * (R(c.K_S_ac) * rac * rac) * B11;
    o.d11[1] = kac * mac * B11;
    o.d11[2] = A11 * mac * Ipac * (dIIN * Inh3 + k.IIN * dInh3 * r_nh3);
    o.s11 = A11 * mac * k.IIN * (dIpac * Inh3 - Ipac * dInh3 * nh3 * R(ab.r_IN));
    // rho12: S_h2, X_h2, S_IN
    o.d12[0] = A12 * (R(c.K_S_h2) * rh2 * rh2) * k.B12;
    o.d12[1] = kh2 * mh2 * k.B12;
    o.d12[2] = A12 * mh2 * k.Iph2 * dIIN;
    o.s12 = A12 * mh2 * k.dIph2 * k.IIN;
#pragma unroll
    for (int i = 0; i < 7; ++i) o.ddec[i] = kd[i];
    // transfers
    o.dT8[0] = kLa; o.dT8[1] = -kLa * KH2;
    o.dT9[0] = kLa; o.dT9[1] = -kLa * KCH4;
    o.dT10[0] = kLa * fco2; o.dT10[1] = -kLa * KCO2;
    o.sT10 = kLa * y[iS_IC] * R(q.K_a_co2) * rco2 * rco2;
    o.qvs = o.qv;
    o.dqv = kpv * (R(2) * P - R(c.P_atm)) * invPa;
    o.P_h2 = P_h2; o.P_ch4 = P_ch4; o.P_co2 = P_co2;
  } else if constexpr (J) {
    o.d1 = kdis * sc; o.d2 = kch * sc; o.d3 = kpr * sc; o.d4 = kli * sc;
    // scaled factors of the uptakes and their derivatives to S_IN (G) and S_H (H)
    const R as = a * sc, aN = as * k.IIN;
    const R dIIN = as * (R(c.K_S_IN) * k.rIN * k.rIN);
    const R Bs = k.B5 * sc, G = k.Ipaa * dIIN, H = k.dIpaa * aN;
    // rho5: S_su, X_su, S_IN
    o.d5[0] = A5 * Bs * (R(c.K_S_su) * k.rsu * k.rsu);
    o.d5[1] = ksu * k.msu * Bs;
    o.d5[2] = p5 * G;
    o.s5 = p5 * H;
    // rho6: S_aa, X_aa, S_IN
    o.d6[0] = A6 * Bs * (R(c.K_S_aa) * k.raa * k.raa);
    o.d6[1] = kaa * k.maa * Bs;
    o.d6[2] = p6 * G;
    o.s6 = p6 * H;
    // rho7: S_fa, X_fa, S_IN, S_h2 (dI/dS_h2 = -K/(K+S)^2 = -I r)
    const R Bs7 = Bs * Ih2fa, p7i = p7 * Ih2fa;
    o.d7[0] = A7 * Bs7 * (R(c.K_S_fa) * k.rfs * k.rfs);
    o.d7[1] = kfa * k.mfa * Bs7;
    o.d7[2] = p7i * G;
    o.d7[3] = -p7i * Bs * rfa;
    o.s7 = p7i * H;
    // rho8, rho9: S_va, S_bu, X_c4, S_IN, S_h2
    const R rd2 = k.rden * k.rden;
    const R dgva_va = (y[iS_bu] + R(kC4Guard)) * rd2, dgva_bu = -y[iS_va] * rd2;
    const R dgbu_bu = (y[iS_va] + R(kC4Guard)) * rd2, dgbu_va = -y[iS_bu] * rd2;
    const R dmva = R(c.K_S_c4) * k.rva * k.rva, dmbu = R(c.K_S_c4) * k.rbu * k.rbu;
    const R Bs8 = Bs * Ih2c4, AB8 = A8 * Bs8, kB8 = kc4 * Bs8, Bsr = Bs * rc4;
    const R p8i = p8 * Ih2c4, p9i = p9 * Ih2c4;
    o.d8[0] = AB8 * (dmva * k.gva + k.mva * dgva_va);
    o.d8[1] = AB8 * (k.mva * dgva_bu);
    o.d8[2] = kB8 * tva;
    o.d8[3] = p8i * G;
    o.d8[4] = -p8i * Bsr;
    o.s8 = p8i * H;
    o.d9[0] = AB8 * (k.mbu * dgbu_va);
    o.d9[1] = AB8 * (dmbu * k.gbu + k.mbu * dgbu_bu);
    o.d9[2] = kB8 * tbu;
    o.d9[3] = p9i * G;
    o.d9[4] = -p9i * Bsr;
    o.s9 = p9i * H;
    // rho10: S_pro, X_pro, S_IN, S_h2
    const R Bs10 = Bs * Ih2pro, p10i = p10 * Ih2pro;
    o.d10[0] = A10 * Bs10 * (R(c.K_S_pro) * k.rpo * k.rpo);
    o.d10[1] = kpo * k.mpo * Bs10;
    o.d10[2] = p10i * G;
    o.d10[3] = -p10i * Bs * rpr;
    o.s10 = p10i * H;
    // rho11: S_ac, X_ac, S_IN (I_IN and free ammonia)
    const R dInh3 = -Inh3 * rnh;  // dI_nh3 / dS_nh3
    const R Bs11 = B11 * sc;
    o.d11[0] = A11 * Bs11 * (R(c.K_S_ac) * rac * rac);
    o.d11[1] = kac * mac * Bs11;
    o.d11[2] = p11 * (Ipac * (dIIN * Inh3 + aN * (dInh3 * r_nh3)));
    o.s11 = p11 * (aN * (dIpac * Inh3 - Ipac * dInh3 * nh3 * R(ab.r_IN)));
    // rho12: S_h2, X_h2, S_IN
    const R Bs12 = k.B12 * sc;
    o.d12[0] = A12 * Bs12 * (R(c.K_S_h2) * rh2 * rh2);
    o.d12[1] = kh2 * mh2 * Bs12;
    o.d12[2] = p12 * (k.Iph2 * dIIN);
    o.s12 = p12 * (k.dIph2 * aN);
#pragma unroll
    for (int i = 0; i < 7; ++i) o.ddec[i] = kd[i] * sc;
    // transfers and gas outflow
    const R kLs = kLa * sc, kps = kpv * invPa * sc;
    o.dT8[0] = kLs; o.dT8[1] = -kLs * KH2;
    o.dT9[0] = kLs; o.dT9[1] = -kLs * KCH4;
    o.dT10[0] = kLs * fco2; o.dT10[1] = -kLs * KCO2;
    o.sT10 = kLs * y[iS_IC] * (R(q.K_a_co2) * rco2 * rco2);
    o.qvs = o.qv * sc;
    o.dqv = kps * (R(2) * P - R(c.P_atm));
    o.P_h2 = P_h2; o.P_ch4 = P_ch4; o.P_co2 = P_co2;
  }
}

// Stoichiometric part of the mass balances of Eq. 2: f = dil + N r, where
// dil holds the transport terms of every state (liquid: dilution; gas:
// outflow) and N the ADM1 stoichiometry of the 19 processes and the three
// gas transfers (r[19..21]).
// C: type of the stoichiometric coefficients in the products (R itself,
// or float for a two-float accumulator R).
template <class R, class DC, class C = R>
CHAD_HD void stoich(const DC& c, const R* r, const R* dil, R* f) {
  const R dec = r[12] + r[13] + r[14] + r[15] + r[16] + r[17] + r[18];
  f[iS_su] = dil[iS_su] + r[1] + C(c.c_su_li) * r[3] - r[4];
  f[iS_aa] = dil[iS_aa] + r[2] - r[5];
  f[iS_fa] = dil[iS_fa] + C(c.f_fa_li) * r[3] - r[6];
  f[iS_va] = dil[iS_va] + C(c.aa_va) * r[5] - r[7];
  f[iS_bu] = dil[iS_bu] + C(c.su_bu) * r[4] + C(c.aa_bu) * r[5] - r[8];
  f[iS_pro] = dil[iS_pro] + C(c.su_pro) * r[4] + C(c.aa_pro) * r[5] + C(c.va_pro) * r[7] - r[9];
  f[iS_ac] = dil[iS_ac] + C(c.su_ac) * r[4] + C(c.aa_ac) * r[5] + C(c.fa_ac) * r[6] +
             C(c.va_ac) * r[7] + C(c.bu_ac) * r[8] + C(c.pro_ac) * r[9] - r[10];
  f[iS_h2] = dil[iS_h2] + C(c.su_h2) * r[4] + C(c.aa_h2) * r[5] + C(c.fa_h2) * r[6] +
             C(c.va_h2) * r[7] + C(c.bu_h2) * r[8] + C(c.pro_h2) * r[9] - r[11] - r[19];
  f[iS_ch4] = dil[iS_ch4] + C(c.ac_ch4) * r[10] + C(c.h2_ch4) * r[11] - r[20];
  R ic = dil[iS_IC] + C(c.cIC[12]) * dec - r[21];
#pragma unroll
  for (int j = 0; j < 12; ++j) ic += C(c.cIC[j]) * r[j];
  f[iS_IC] = ic;
  R in = dil[iS_IN] + C(c.nIN[0]) * r[0] + C(c.nIN[12]) * dec;
#pragma unroll
  for (int j = 4; j < 12; ++j) in += C(c.nIN[j]) * r[j];
  f[iS_IN] = in;
  f[iS_I] = dil[iS_I] + C(c.f_sI) * r[0];
  f[iX_c] = dil[iX_c] - r[0] + dec;
  f[iX_ch] = dil[iX_ch] + C(c.f_ch) * r[0] - r[1];
  f[iX_pr] = dil[iX_pr] + C(c.f_pr) * r[0] - r[2];
  f[iX_li] = dil[iX_li] + C(c.f_li) * r[0] - r[3];
  f[iX_su] = dil[iX_su] + C(c.Y_su) * r[4] - r[12];
  f[iX_aa] = dil[iX_aa] + C(c.Y_aa) * r[5] - r[13];
  f[iX_fa] = dil[iX_fa] + C(c.Y_fa) * r[6] - r[14];
  f[iX_c4] = dil[iX_c4] + C(c.Y_c4) * (r[7] + r[8]) - r[15];
  f[iX_pro] = dil[iX_pro] + C(c.Y_pro) * r[9] - r[16];
  f[iX_ac] = dil[iX_ac] + C(c.Y_ac) * r[10] - r[17];
  f[iX_h2] = dil[iX_h2] + C(c.Y_h2) * r[11] - r[18];
  f[iX_I] = dil[iX_I] + C(c.f_xI) * r[0];
  f[iS_cat] = dil[iS_cat];
  f[iS_an] = dil[iS_an];
  const C vr = C(c.Vliq_over_Vgas);
  f[iG_h2] = dil[iG_h2] + vr * r[19];
  f[iG_ch4] = dil[iG_ch4] + vr * r[20];
  f[iG_co2] = dil[iG_co2] + vr * r[21];
}

// f(y): mass balances of Eq. 2 with the ADM1 stoichiometry
template <class R, class DC>
CHAD_HD void balances(const DC& c, const R* y, R D, const Rates<R>& o, R* f) {
  R dil[NS];
#pragma unroll
  for (int i = 0; i < 26; ++i) dil[i] = D * (R(c.y_in[i]) - y[i]);
  dil[iG_h2] = -y[iG_h2] * o.qv;
  dil[iG_ch4] = -y[iG_ch4] * o.qv;
  dil[iG_co2] = -y[iG_co2] * o.qv;
  stoich<R>(c, o.r, dil, f);
}

// Jacobian-vector product J x = J_d x + u (v^T x) without a matrix: the
// rate partials of rates<RO, true> give the linearised rates
// dr = (d rho / dy) x + (d rho / dS_H) s with s = v^T x, which go through the
// same stoichiometry as the rates; the transport terms are linearised
// directly.  Arithmetic in precision RD (FP64 in the kernels) whatever the
// precision RO of the partials.
template <class RO, class RD, class DC, class C = RD>
CHAD_HD void jvp(const DC& c, const C* y, C D, const Rates<RO>& o, const RD* x, RD s,
                 RD* out) {
  RD dr[22];
  dr[0] = C(o.d1) * x[iX_c];
  dr[1] = C(o.d2) * x[iX_ch];
  dr[2] = C(o.d3) * x[iX_pr];
  dr[3] = C(o.d4) * x[iX_li];
  dr[4] = C(o.d5[0]) * x[iS_su] + C(o.d5[1]) * x[iX_su] + C(o.d5[2]) * x[iS_IN] +
          C(o.s5) * s;
  dr[5] = C(o.d6[0]) * x[iS_aa] + C(o.d6[1]) * x[iX_aa] + C(o.d6[2]) * x[iS_IN] +
          C(o.s6) * s;
  dr[6] = C(o.d7[0]) * x[iS_fa] + C(o.d7[1]) * x[iX_fa] + C(o.d7[2]) * x[iS_IN] +
          C(o.d7[3]) * x[iS_h2] + C(o.s7) * s;
  dr[7] = C(o.d8[0]) * x[iS_va] + C(o.d8[1]) * x[iS_bu] + C(o.d8[2]) * x[iX_c4] +
          C(o.d8[3]) * x[iS_IN] + C(o.d8[4]) * x[iS_h2] + C(o.s8) * s;
  dr[8] = C(o.d9[0]) * x[iS_va] + C(o.d9[1]) * x[iS_bu] + C(o.d9[2]) * x[iX_c4] +
          C(o.d9[3]) * x[iS_IN] + C(o.d9[4]) * x[iS_h2] + C(o.s9) * s;
  dr[9] = C(o.d10[0]) * x[iS_pro] + C(o.d10[1]) * x[iX_pro] +
          C(o.d10[2]) * x[iS_IN] + C(o.d10[3]) * x[iS_h2] + C(o.s10) * s;
  dr[10] = C(o.d11[0]) * x[iS_ac] + C(o.d11[1]) * x[iX_ac] +
           C(o.d11[2]) * x[iS_IN] + C(o.s11) * s;
  dr[11] = C(o.d12[0]) * x[iS_h2] + C(o.d12[1]) * x[iX_h2] +
           C(o.d12[2]) * x[iS_IN] + C(o.s12) * s;
#pragma unroll
  for (int k = 0; k < 7; ++k) dr[12 + k] = C(o.ddec[k]) * x[iX_su + k];
  dr[19] = C(o.dT8[0]) * x[iS_h2] + C(o.dT8[1]) * x[iG_h2];
  dr[20] = C(o.dT9[0]) * x[iS_ch4] + C(o.dT9[1]) * x[iG_ch4];
  dr[21] = C(o.dT10[0]) * x[iS_IC] + C(o.dT10[1]) * x[iG_co2] + C(o.sT10) * s;
  RD dil[NS];
#pragma unroll
  for (int i = 0; i < 26; ++i) dil[i] = -D * x[i];
  const C qv = C(o.qvs);
  const RD dq =
      C(o.dqv) * (C(o.P_h2) * x[iG_h2] + C(o.P_ch4) * x[iG_ch4] + C(o.P_co2) * x[iG_co2]);
  dil[iG_h2] = -x[iG_h2] * qv - y[iG_h2] * dq;
  dil[iG_ch4] = -x[iG_ch4] * qv - y[iG_ch4] * dq;
  dil[iG_co2] = -x[iG_co2] * qv - y[iG_co2] * dq;
  stoich<RD, DC, C>(c, dr, dil, out);
}


// J[row][cols[k]] += coef * d[k]; u[row] += coef * s.  Idx maps (row, col)
// to a storage slot (negative: structurally absent, the write is dropped).
template <class Idx, class R, class JS>
CHAD_HD void jadd(JS Jm, int row, int col, R v) {
  const int s = Idx::at(row, col);
  if (s >= 0) Jm[s] += v;
}
template <class Idx, class R, class JS, int NC>
CHAD_HD void scat(JS Jm, R* u, int row, R coef, const int (&cols)[NC], const R (&d)[NC], R s) {
#pragma unroll
  for (int k = 0; k < NC; ++k) jadd<Idx>(Jm, row, cols[k], coef * d[k]);
  u[row] += coef * s;
}
template <class Idx, class R, class JS, int NC>
CHAD_HD void scat(JS Jm, int row, R coef, const int (&cols)[NC], const R (&d)[NC]) {
#pragma unroll
  for (int k = 0; k < NC; ++k) jadd<Idx>(Jm, row, cols[k], coef * d[k]);
}

// Analytic Jacobian (row-major NS x NS) from the rate partials.  The S_H
// dependence enters as the rank-1 term u v^T, u = df/dS_H (at fixed y),
// v = dS_H/dy = -(dE/dy) / (dE/dS_H) from Eq. 7.
// With u_out == nullptr the full J = J_d + u v^T is assembled; otherwise only
// the direct part J_d (S_H held fixed) goes into Jm and u = df/dS_H into
// u_out, for the Sherman-Morrison solve of W = W_d - g u v^T.
// The sums start from -0, the identity of IEEE addition, so that the first
// term of each slot costs no addition (0 + v would: it turns -0 into 0).
// UNIT > 0: diagonal slots below UNIT start from 1 instead (with partials
// and D scaled by -g the slots below UNIT then hold W_d = I - g J_d).
template <class Idx, class R, int UNIT = 0, class JS, class DC, class PQ>
CHAD_HD void jacobian(const DC& c, const PQ& q, const R* y, R D, const AcidBase& ab,
                      const Rates<R>& o, JS Jm, R* u_out = nullptr) {
  R u[NS];
#pragma unroll
  for (int i = 0; i < Idx::size; ++i) Jm[i] = R(-0.0);
#pragma unroll
  for (int i = 0; i < NS; ++i) u[i] = R(-0.0);
#pragma unroll
  for (int i = 0; i < NS; ++i)
    if (Idx::at(i, i) < UNIT) Jm[Idx::at(i, i)] = R(1);
#pragma unroll
  for (int i = 0; i < 26; ++i) jadd<Idx>(Jm, i, i, -D);
  const R one = R(1), mone = R(-1);
  const R cIC12 = R(c.cIC[12]), nIN12 = R(c.nIN[12]);
  {  // rho1 disintegration
    const int cols[1] = {iX_c};
    const R d[1] = {o.d1};
    scat<Idx>(Jm, iX_c, mone, cols, d);
    scat<Idx>(Jm, iS_I, R(c.f_sI), cols, d);
    scat<Idx>(Jm, iX_ch, R(c.f_ch), cols, d);
    scat<Idx>(Jm, iX_pr, R(c.f_pr), cols, d);
    scat<Idx>(Jm, iX_li, R(c.f_li), cols, d);
    scat<Idx>(Jm, iX_I, R(c.f_xI), cols, d);
    scat<Idx>(Jm, iS_IC, R(c.cIC[0]), cols, d);
    scat<Idx>(Jm, iS_IN, R(c.nIN[0]), cols, d);
  }
  {  // rho2-4 hydrolysis
    const int c2[1] = {iX_ch}, c3[1] = {iX_pr}, c4[1] = {iX_li};
    const R d2[1] = {o.d2}, d3[1] = {o.d3}, d4[1] = {o.d4};
    scat<Idx>(Jm, iX_ch, mone, c2, d2);
    scat<Idx>(Jm, iS_su, one, c2, d2);
    scat<Idx>(Jm, iS_IC, R(c.cIC[1]), c2, d2);
    scat<Idx>(Jm, iX_pr, mone, c3, d3);
    scat<Idx>(Jm, iS_aa, one, c3, d3);
    scat<Idx>(Jm, iS_IC, R(c.cIC[2]), c3, d3);
    scat<Idx>(Jm, iX_li, mone, c4, d4);
    scat<Idx>(Jm, iS_su, R(c.c_su_li), c4, d4);
    scat<Idx>(Jm, iS_fa, R(c.f_fa_li), c4, d4);
    scat<Idx>(Jm, iS_IC, R(c.cIC[3]), c4, d4);
  }
  {  // rho5 sugars
    const int cols[3] = {iS_su, iX_su, iS_IN};
    scat<Idx>(Jm, u, iS_su, mone, cols, o.d5, o.s5);
    scat<Idx>(Jm, u, iS_bu, R(c.su_bu), cols, o.d5, o.s5);
    scat<Idx>(Jm, u, iS_pro, R(c.su_pro), cols, o.d5, o.s5);
    scat<Idx>(Jm, u, iS_ac, R(c.su_ac), cols, o.d5, o.s5);
    scat<Idx>(Jm, u, iS_h2, R(c.su_h2), cols, o.d5, o.s5);
    scat<Idx>(Jm, u, iX_su, R(c.Y_su), cols, o.d5, o.s5);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[4]), cols, o.d5, o.s5);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[4]), cols, o.d5, o.s5);
  }
  {  // rho6 amino acids
    const int cols[3] = {iS_aa, iX_aa, iS_IN};
    scat<Idx>(Jm, u, iS_aa, mone, cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iS_va, R(c.aa_va), cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iS_bu, R(c.aa_bu), cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iS_pro, R(c.aa_pro), cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iS_ac, R(c.aa_ac), cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iS_h2, R(c.aa_h2), cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iX_aa, R(c.Y_aa), cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[5]), cols, o.d6, o.s6);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[5]), cols, o.d6, o.s6);
  }
  {  // rho7 LCFA
    const int cols[4] = {iS_fa, iX_fa, iS_IN, iS_h2};
    scat<Idx>(Jm, u, iS_fa, mone, cols, o.d7, o.s7);
    scat<Idx>(Jm, u, iS_ac, R(c.fa_ac), cols, o.d7, o.s7);
    scat<Idx>(Jm, u, iS_h2, R(c.fa_h2), cols, o.d7, o.s7);
    scat<Idx>(Jm, u, iX_fa, R(c.Y_fa), cols, o.d7, o.s7);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[6]), cols, o.d7, o.s7);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[6]), cols, o.d7, o.s7);
  }
  {  // rho8 valerate
    const int cols[5] = {iS_va, iS_bu, iX_c4, iS_IN, iS_h2};
    scat<Idx>(Jm, u, iS_va, mone, cols, o.d8, o.s8);
    scat<Idx>(Jm, u, iS_pro, R(c.va_pro), cols, o.d8, o.s8);
    scat<Idx>(Jm, u, iS_ac, R(c.va_ac), cols, o.d8, o.s8);
    scat<Idx>(Jm, u, iS_h2, R(c.va_h2), cols, o.d8, o.s8);
    scat<Idx>(Jm, u, iX_c4, R(c.Y_c4), cols, o.d8, o.s8);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[7]), cols, o.d8, o.s8);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[7]), cols, o.d8, o.s8);
  }
  {  // rho9 butyrate
    const int cols[5] = {iS_va, iS_bu, iX_c4, iS_IN, iS_h2};
    scat<Idx>(Jm, u, iS_bu, mone, cols, o.d9, o.s9);
    scat<Idx>(Jm, u, iS_ac, R(c.bu_ac), cols, o.d9, o.s9);
    scat<Idx>(Jm, u, iS_h2, R(c.bu_h2), cols, o.d9, o.s9);
    scat<Idx>(Jm, u, iX_c4, R(c.Y_c4), cols, o.d9, o.s9);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[8]), cols, o.d9, o.s9);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[8]), cols, o.d9, o.s9);
  }
  {  // rho10 propionate
    const int cols[4] = {iS_pro, iX_pro, iS_IN, iS_h2};
    scat<Idx>(Jm, u, iS_pro, mone, cols, o.d10, o.s10);
    scat<Idx>(Jm, u, iS_ac, R(c.pro_ac), cols, o.d10, o.s10);
    scat<Idx>(Jm, u, iS_h2, R(c.pro_h2), cols, o.d10, o.s10);
    scat<Idx>(Jm, u, iX_pro, R(c.Y_pro), cols, o.d10, o.s10);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[9]), cols, o.d10, o.s10);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[9]), cols, o.d10, o.s10);
  }
  {  // rho11 acetate
    const int cols[3] = {iS_ac, iX_ac, iS_IN};
    scat<Idx>(Jm, u, iS_ac, mone, cols, o.d11, o.s11);
    scat<Idx>(Jm, u, iS_ch4, R(c.ac_ch4), cols, o.d11, o.s11);
    scat<Idx>(Jm, u, iX_ac, R(c.Y_ac), cols, o.d11, o.s11);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[10]), cols, o.d11, o.s11);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[10]), cols, o.d11, o.s11);
  }
  {  // rho12 hydrogen
    const int cols[3] = {iS_h2, iX_h2, iS_IN};
    scat<Idx>(Jm, u, iS_h2, mone, cols, o.d12, o.s12);
    scat<Idx>(Jm, u, iS_ch4, R(c.h2_ch4), cols, o.d12, o.s12);
    scat<Idx>(Jm, u, iX_h2, R(c.Y_h2), cols, o.d12, o.s12);
    scat<Idx>(Jm, u, iS_IC, R(c.cIC[11]), cols, o.d12, o.s12);
    scat<Idx>(Jm, u, iS_IN, R(c.nIN[11]), cols, o.d12, o.s12);
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) {  // rho13-19 decay
    const int col = iX_su + k;
    const R dk = o.ddec[k];
    jadd<Idx>(Jm, col, col, -dk);
    jadd<Idx>(Jm, (int)iX_c, col, dk);
    jadd<Idx>(Jm, (int)iS_IC, col, cIC12 * dk);
    jadd<Idx>(Jm, (int)iS_IN, col, nIN12 * dk);
  }
  const R vr = R(c.Vliq_over_Vgas);
  {  // transfers
    const int c8[2] = {iS_h2, iG_h2}, c9[2] = {iS_ch4, iG_ch4}, c10[2] = {iS_IC, iG_co2};
    scat<Idx>(Jm, iS_h2, mone, c8, o.dT8);
    scat<Idx>(Jm, iG_h2, vr, c8, o.dT8);
    scat<Idx>(Jm, iS_ch4, mone, c9, o.dT9);
    scat<Idx>(Jm, iG_ch4, vr, c9, o.dT9);
    scat<Idx>(Jm, u, iS_IC, mone, c10, o.dT10, o.sT10);
    scat<Idx>(Jm, u, iG_co2, vr, c10, o.dT10, o.sT10);
  }
  {  // gas outflow: f_G = -G q(P)
    const int g[3] = {iG_h2, iG_ch4, iG_co2};
    const R dP[3] = {o.P_h2, o.P_ch4, o.P_co2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      jadd<Idx>(Jm, g[a], g[a], -o.qvs);
      const R gq = y[g[a]] * o.dqv;
#pragma unroll
      for (int b = 0; b < 3; ++b) jadd<Idx>(Jm, g[a], g[b], -gq * dP[b]);
    }
  }
  if (u_out) {
#pragma unroll
    for (int i = 0; i < NS; ++i) u_out[i] = u[i];
    return;
  }
  // rank-1 S_H coupling: J += u v^T over the 8 states that enter Eq. 7
  const int hc[8] = {iS_va, iS_bu, iS_pro, iS_ac, iS_IC, iS_IN, iS_cat, iS_an};
  double vd[8];
  sh_tangent(c, q, ab, vd);
  R v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = R(vd[k]);
  const int ur[19] = {iS_su, iS_aa, iS_fa, iS_va, iS_bu, iS_pro, iS_ac, iS_h2, iS_ch4, iS_IC,
                      iS_IN, iX_su, iX_aa, iX_fa, iX_c4, iX_pro, iX_ac, iX_h2, iG_co2};
#pragma unroll
  for (int i = 0; i < 19; ++i)
#pragma unroll
    for (int k = 0; k < 8; ++k) jadd<Idx>(Jm, ur[i], hc[k], u[ur[i]] * v[k]);
}

}  // namespace chad
