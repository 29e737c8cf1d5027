// Device evaluation of the stationary-phase template (App. A, Eq. A1) in FP64.
//   Psi(f) = 2 pi f tc - phic - pi/4 + 3/(128 eta) g(v),  v = (pi M f)^(1/3),
//   g(v)   = sum_k alpha_k v^(k-5) + a5log ln(v / v_lso) + a6log v ln(4 v),
//   Psi'   = 2 pi t(f) (Eq. A2),  Psi'' = 2 pi t'(f).
#pragma once

#include <cmath>

#include "rf_internal.h"

namespace rf {

constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double kTwoPi = 6.28318530717958647692528676655900577;
constexpr double kSqrt6 = 2.44948974278317809819728407470589139;  // 1 / v_lso

__device__ __forceinline__ double tf2_series(const Tf2& p, double v) {
  const double iv = 1.0 / v;
  const double iv5 = iv * iv * iv * iv * iv;
  // sum_k a_k v^(k-5) = v^-5 (a0 + a1 v + ... + a7 v^7), Horner in v
  double poly = p.a[7];
#pragma unroll
  for (int k = 6; k >= 0; --k) poly = poly * v + p.a[k];
  double g = poly * iv5;
  if (p.a5log != 0.0) g += p.a5log * log(v * kSqrt6);
  if (p.a6log != 0.0) g += p.a6log * v * log(4.0 * v);
  return g;
}

// Phase in turns at bin k of a uniform grid f_k = k df, from tables of powers of k that do not
// depend on the template (or on df): u = k^(1/3), u5 = k^(-5/3), lu = ln(k) / 3.  With
// v = c u, c = (pi M df)^(1/3), every term of Psi / (2 pi) is a template coefficient times a power
// of u and possibly lu, so a bin costs about ten FP64 multiply-adds and no cube root, logarithm or
// division (the FP64 pipe has two lanes per SM: the direct evaluation took 127 us per template at
// n = 2^20).  The leading term is one product with a table entry instead of a fifth power, so
// its error is below the direct form's.  Phases add up: coefficients of two templates subtract.
struct Tf2Bins {
  double b0, b2, b3, b4, b7;  // u^-5, u^-3, u^-2, u^-1, u^2
  double l5, l6, m6;          // lu, u lu, u
  double d, e;                // k, 1
};

inline Tf2Bins make_tf2_bins(const Tf2& p, double df) {
  const double x = kPi * p.M * df;
  const double c = std::cbrt(x);
  const double s = p.pref / kTwoPi;
  const double cm5 = 1.0 / (x * c * c);
  Tf2Bins q;
  q.b0 = s * p.a[0] * cm5;
  q.b2 = s * p.a[2] / x;
  q.b3 = s * p.a[3] / (c * c);
  q.b4 = s * p.a[4] / c;
  q.b7 = s * p.a[7] * c * c;
  q.l5 = s * p.a5log;
  q.l6 = s * p.a6log * c;
  q.m6 = s * c * (p.a[6] + p.a6log * std::log(4.0 * c));
  q.d = df * p.tc;
  q.e = s * (p.a[5] + p.a5log * std::log(c * kSqrt6)) - p.phic / kTwoPi - 0.125;
  q.e -= std::rint(q.e);  // whole turns, exactly: a large phi_c costs the other terms no bits
  return q;
}

// a - b, times `unit` (a power of two: the phase in parts of a turn), whole turns of the constant
// term taken off
inline Tf2Bins tf2_bins_minus(const Tf2Bins& a, const Tf2Bins& b, double unit) {
  const double e = a.e - b.e;
  return Tf2Bins{unit * (a.b0 - b.b0), unit * (a.b2 - b.b2), unit * (a.b3 - b.b3), unit * (a.b4 - b.b4),
                 unit * (a.b7 - b.b7), unit * (a.l5 - b.l5), unit * (a.l6 - b.l6), unit * (a.m6 - b.m6),
                 unit * (a.d - b.d),   unit * (e - std::rint(e))};
}

// Bounds over the bins ka..kb >= 1 of the leading terms (u^-5 and k) and of the sum of the others.
struct Tf2Size {
  double lead, rest;
};
inline Tf2Size tf2_bins_size(const Tf2Bins& q, double ka, double kb) {
  const double ua = std::cbrt(ka), ub = std::cbrt(kb), l = std::log(kb) / 3.0;
  return Tf2Size{std::fabs(q.b0) / (ka * ua * ua) + std::fabs(q.d) * kb,
                 std::fabs(q.b2) / ka + std::fabs(q.b3) / (ua * ua) + std::fabs(q.b4) / ua +
                     std::fabs(q.b7) * ub * ub + std::fabs(q.l5) * l + std::fabs(q.l6) * ub * l +
                     std::fabs(q.m6) * ub + std::fabs(q.e)};
}

// The phase of bin k as a fraction of a turn in [-1/2, 1/2].
__device__ __forceinline__ double tf2_turn(const Tf2Bins& q, int64_t k, double u, double u5, double lu) {
  double t = fma(u, fma(q.l6, lu, fma(q.b7, u, q.m6)), fma(q.l5, lu, q.e));
  t = fma(u5, fma(u * u, fma(u, fma(u, q.b4, q.b3), q.b2), q.b0), t);
  if (q.d != 0.0) t = fma((double)k, q.d, t);
  // nearest whole number by the rounding of a large sum (|t| < 2^51)
  const double big = 6755399441055744.0;
  return t - ((t + big) - big);
}

// The same phase in FP32 pairs (value h + l, about 46 bits; the scheme of cdf.cuh for real numbers)
// for filters that are rounded to FP32 in the same kernel: 3e4 turns keep 5e-10 of a turn, below the
// rounding of the angle to FP32, and the FP32 pipes are 60 times as wide as the FP64 pipe.
struct Pair {
  float h, l;
};
__host__ __device__ __forceinline__ Pair make_pair_of(double x) {
  const float h = (float)x;
  return Pair{h, (float)(x - (double)h)};
}
struct Tf2Pairs {
  Pair b0, b2, b3, b4, b7, l5, l6, m6, e;  // no term in k: for t_c = 0
};
__host__ __device__ __forceinline__ Tf2Pairs make_tf2_pairs(const Tf2Bins& q) {
  return Tf2Pairs{make_pair_of(q.b0), make_pair_of(q.b2), make_pair_of(q.b3),
                  make_pair_of(q.b4), make_pair_of(q.b7), make_pair_of(q.l5),
                  make_pair_of(q.l6), make_pair_of(q.m6), make_pair_of(q.e)};
}
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  const float p = __fmul_rn(a.h, b.h);
  return Pair{p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)))};
}
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
  const float s = __fadd_rn(a.h, b.h), t = __fadd_rn(s, -a.h);
  const float e = __fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -t)), __fadd_rn(b.h, -t));
  return Pair{s, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ float tf2_turn(const Tf2Pairs& q, Pair u, Pair u5, Pair lu) {
  const Pair p = pair_add(pair_mul(u, pair_add(pair_mul(u, q.b4), q.b3)), q.b2);
  const Pair lead = pair_mul(u5, pair_add(pair_mul(pair_mul(u, u), p), q.b0));
  const Pair high = pair_mul(u, pair_add(pair_mul(q.l6, lu), pair_add(pair_mul(q.b7, u), q.m6)));
  const Pair t = pair_add(lead, pair_add(high, pair_add(pair_mul(q.l5, lu), q.e)));
  return __fadd_rn(__fadd_rn(t.h, -rintf(t.h)), t.l);
}

// Psi(f) in radians, f > 0.
__device__ __forceinline__ double tf2_phase(const Tf2& p, double f) {
  const double v = cbrt(kPi * p.M * f);
  return kTwoPi * f * p.tc - p.phic - 0.25 * kPi + p.pref * tf2_series(p, v);
}

// g'(v) and g''(v): sum_k a_k (k - 5) v^(k-6) and its derivative, Horner in v (sixteen calls of pow
// kept a single thread busy for 60 us)
__host__ __device__ __forceinline__ void tf2_series_d(const Tf2& p, double v, double& g1, double& g2) {
  double s1 = 2.0 * p.a[7], s2 = 2.0 * p.a[7];
#pragma unroll
  for (int k = 6; k >= 0; --k) {
    const double e = (double)(k - 5);
    s1 = s1 * v + e * p.a[k];
    s2 = s2 * v + e * (e - 1.0) * p.a[k];
  }
  const double iv = 1.0 / v, iv2 = iv * iv, iv6 = iv2 * iv2 * iv2;
  g1 = s1 * iv6;
  g2 = s2 * iv6 * iv;
  if (p.a5log != 0.0) {
    g1 += p.a5log / v;
    g2 -= p.a5log / (v * v);
  }
  if (p.a6log != 0.0) {
    g1 += p.a6log * (log(4.0 * v) + 1.0);
    g2 += p.a6log / v;
  }
}

// Psi'(f) = 2 pi tc + 3/(128 eta) g'(v) dv/df = 2 pi t(f) (Eq. A2)
__host__ __device__ __forceinline__ double tf2_dphase(const Tf2& p, double f) {
  const double v = cbrt(kPi * p.M * f);
  double g1, g2;
  tf2_series_d(p, v, g1, g2);
  return kTwoPi * p.tc + p.pref * g1 * (kPi * p.M / (3.0 * v * v));
}

// Psi''(f) = (pi M / (128 eta)) (g'' v^-2 - 2 g' v^-3) dv/df,  dv/df = pi M / (3 v^2)
__device__ __forceinline__ double tf2_d2phase(const Tf2& p, double f) {
  const double v = cbrt(kPi * p.M * f);
  double g1, g2;
  tf2_series_d(p, v, g1, g2);
  const double dv = kPi * p.M / (3.0 * v * v);
  return (kPi * p.M / (128.0 * p.eta)) * (g2 / (v * v) - 2.0 * g1 / (v * v * v)) * dv;
}

// B(f) = f^(-7/6)
__device__ __forceinline__ double tf2_amp(double f) { return exp(-7.0 / 6.0 * log(f)); }

// W(f) of Eq. (9)
__device__ __forceinline__ double window_w(double f, double f_low, double f_high, double dfl, double dfh) {
  if (f >= f_low && f <= f_high) return 1.0;
  if (f > f_low - dfl && f < f_low && dfl > 0.0) return 0.5 * (1.0 + cospi((f - f_low) / dfl));
  if (f > f_high && f < f_high + dfh && dfh > 0.0) return 0.5 * (1.0 - cospi((f - (f_high + dfh)) / dfh));
  return 0.0;
}

}  // namespace rf
