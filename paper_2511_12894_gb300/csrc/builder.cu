// Ratio-kernel builder (Sec. II.B-II.D; Eqs. 5, 7, 9, 10), FP64 (on FP32 grids the transforms in FP32
// pairs, below).
//
// Per neighbour j of the reference, on its build grid of n_b bins (f_k = k fs / n_b; n_b = n
// unless a coarser grid is asked for, Sec. II.D):
//   df_low_j = min(df_low_max, f_low / 2, 1 / sqrt(|dPsi''(f_low)| / (2 pi)))          (Eq. 10)
//   K~_j[k]  = (N_ref / N_j) R(f_k) W_j(f_k) exp(+i (Psi_j(f_k) - Psi_ref(f_k))) / n_b   (Eqs. 5, 7, 9)
//   rho_j    = unnormalised n_b-point inverse DFT of K~_j (zero for k > n_b/2)
//   kept     = { m : |rho_j[m]|^2 >= thr^2 a_j },  a_j = max |rho_j|^2 (relative) or 1
//   [m0, m0 + L) = shortest circular arc covering `kept`, ties to the smallest signed m0
//   taps c_j[l] = rho_j[(m0 + l) mod n_b]
// The automatic grid is the smallest power of two of at least four times the lag extent
// between the time offsets dt(f) = (Psi_j' - Psi_ref')(f) / (2 pi) (Eq. A2) at the window
// edges f_low - df_low_j and f_high + df_high, plus the taper spread 4 fs / df_low_j
// (capped at n); neighbours are processed grouped by grid.
// The templates share the amplitude law B = f^-7/6, so R = 1 and N_ref / N_j = 1;
// both factors are still formed from their definitions.
#include <algorithm>
#include <climits>
#include <cmath>
#include <memory>
#include <type_traits>
#include <utility>

#include "cdf.cuh"
#include "cplx.cuh"
#include "rf_internal.h"
#include "tf2.cuh"

namespace rf {

namespace {

// ---------------------------------------------------------------- FP32 grids: transforms in pairs
// The taps of an FP32 grid are rounded to FP32, and the transform that makes them cost 2.9 of the 7 ms
// of building 48 kernels on 2^19 bins, all of it on the FP64 pipe.  The same radix passes in FP32
// pairs (cdf.cuh) are bound by HBM: 171 us per radix-16 pass of those rows (754 MB, 65% of the
// copy rate; the first one, which forms the spectrum, 452 us, by the FP64 pipe), the whole build 1.83 ms.  The leading term of the phase stays FP64.
//
// Pairs serve where the result is the FP64 one:
// * A row's error is bounded by eps times its largest value: 2^-43 for the transform (2^-46.4 measured,
//   n = 2^14 .. 2^22) and what the phase loses, 2^-53 of its leading term and 2^-46 of the others.
// * A kernel is made in pairs when eps is at most 2^-23 of the truncation threshold, so that the smallest
//   kept tap is as good as its rounding to FP32 (thresholds from about 4e-6 for neighbours of one
//   bank); else, for absolute thresholds on |rho|^2 and for grids below 4096 bins, in FP64.  Each
//   kernel is judged by itself: what else is built in the call makes no difference.
// * A kernel whose span depends on a lag within eps of the cut (or, for analytic spans, on the last
//   bits of the largest value) is made again in FP64 before it is cut.
constexpr int64_t kPairMinGrid = 4096;
constexpr double kPairTransformErr = 1.0 / (double)(1ll << 43);
constexpr double kPairTapErr = 1.0 / (double)(1 << 23);

// A template's phase minus the reference's (for pairs in 4096ths of a turn) and, for pairs, eps.
struct RowPhase {
  Tf2Bins q;
  double eps;
};

__global__ void k_df_low(Tf2 ref, const Tf2* __restrict__ tg, int count, double f_low, double df_low_max,
                         double* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= count) return;
  const double d2 = tf2_d2phase(tg[j], f_low) - tf2_d2phase(ref, f_low);
  const double dtp = fabs(d2) / kTwoPi;  // |d t'(f_low)| = |d tau'(f_low)| for a common t_c
  double v = fmin(df_low_max, 0.5 * f_low);
  if (dtp > 0.0) v = fmin(v, 1.0 / sqrt(dtp));
  out[j] = v;
}

// Lag extent of each kernel for the automatic build grid (samples).
__global__ void k_grid_extent(Tf2 ref, const Tf2* __restrict__ tg, const double* __restrict__ dfl, int count,
                              double fs, double f_low, double f_high, double df_high, double* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= count) return;
  const double fa = f_low - dfl[j], fb = f_high + df_high;
  const double ta = (tf2_dphase(tg[j], fa) - tf2_dphase(ref, fa)) / kTwoPi;
  const double tb = (tf2_dphase(tg[j], fb) - tf2_dphase(ref, fb)) / kTwoPi;
  out[j] = fmax(fabs(ta), fabs(tb)) * fs + 4.0 * fs / dfl[j];
}

// Analytic truncation (Sec. II.D with the App. A expressions), one thread per template: the
// threshold amplitude A on |r| = 2 fs |rho| (N_ref / N_j = 1: one amplitude law) is thr times
// the kernel's peak (relative) or thr; each taper end f_e reaches d_e = (R / (4 pi df_e^2 A))^(1/3)
// on both sides of its lag time c_e = -dt(f_e); the kept lags run from floor(min(c_e - d_e) fs)
// to ceil(max(c_e + d_e) fs), at most the grid.
// (rfac: |r| = rfac fs |rho|, 2 for the complex kernel, 1 for the real form's taps 2 Re rho.)
// rp: null, or the rows' phases (kernels in pairs): a span that the error of the row's largest value
// could change, or taps kept down to a level that it disturbs, are marked by len = -len - 1.
__global__ void k_analytic_span(Tf2 ref, const Tf2* __restrict__ tg, const double* __restrict__ dfl,
                                const double* __restrict__ amax2, const RowPhase* __restrict__ rp, int count,
                                double thr, int relative, double rfac, int64_t nb, double fs, double f_low,
                                double f_high, double df_high, int* __restrict__ m0_out, int* __restrict__ len_out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= count) return;
  const double top = rfac * fs * sqrt(amax2[j]);
  const double amp = relative ? thr * top : thr;
  if (!(amp > 0.0)) {
    m0_out[j] = 0;
    len_out[j] = 0;
    return;
  }
  const double fe[4] = {f_low - dfl[j], f_low, f_high, f_high + df_high};
  const double dfe[4] = {dfl[j], dfl[j], df_high, df_high};
  double c[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) c[e] = -((tf2_dphase(tg[j], fe[e]) - tf2_dphase(ref, fe[e])) / kTwoPi);
  auto span = [&](double a, int& m0, int& len) {
    double lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const double R = tf2_amp(fe[e]) / tf2_amp(fe[e]);  // B_j / B_ref: one amplitude law
      const double d = cbrt(R / (4.0 * kPi * dfe[e] * dfe[e] * a));
      lo = fmin(lo, c[e] - d);
      hi = fmax(hi, c[e] + d);
    }
    // a span as long as the grid (a tiny amplitude, or a taper of width 0) keeps the whole
    // grid from lag 0; decided in double, before any integer conversion
    const double flo = floor(lo * fs), fhi = ceil(hi * fs);
    if (!(fhi - flo + 1.0 < (double)nb)) {
      m0 = 0;
      len = (int)nb;
      return;
    }
    const long long m_lo = (long long)flo, m_hi = (long long)fhi;
    long long m = m_lo & (nb - 1);
    if (m > nb / 2) m -= nb;
    m0 = (int)m;
    len = (int)(m_hi - m_lo + 1);
  };
  int m0, len;
  span(amp, m0, len);
  bool unsure = false;
  if (rp) {
    const double eps = rp[j].eps;
    unsure = !(eps * top <= kPairTapErr * amp);
    if (relative && !unsure) {
      int ma, la, mb, lb;
      span(amp * (1.0 - eps), ma, la);
      span(amp * (1.0 + eps), mb, lb);
      unsure = ma != mb || la != lb;
    }
  }
  m0_out[j] = m0;
  len_out[j] = unsure ? -len - 1 : len;
}

// Real-kernel form: rho -> 2 Re rho in place (imaginary parts zero).
__global__ void k_real_form(double2* __restrict__ rho, int64_t count) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    rho[i] = make_double2(2.0 * rho[i].x, 0.0);
}

__global__ void k_real_form(cdf* __restrict__ rho, int64_t count) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    rho[i] = cdf{make_float2(2.f * rho[i].h.x, 0.f), make_float2(2.f * rho[i].l.x, 0.f)};
}

// One row per template (grid.y): K~ over the full length-n buffer.  rp: the template's phase minus
// the reference's (tf2.cuh); [k0, k1]: the bins inside [f_low, f_high], where W = 1.  Bound by the
// FP64 pipe (two lanes per SM): the phase from the tables of bin powers is about ten multiply-adds
// a bin.
//
// K~ = (N_ref / N_j) W conj(h~_j / h~_ref) (Eq. 5 normalised as in Eq. 3).  Every template of the
// stationary-phase family has the amplitude law A f^-7/6 on the same band, so h~_j / h~_ref =
// (A_j / A_ref) e^{-i dPsi} and N_j / N_ref = A_j / A_ref: the two amplitude factors cancel exactly
// for any scales A, and |K~| = W.
__global__ void __launch_bounds__(256) k_kernel_spectrum(const RowPhase* __restrict__ rp,
                                                         const double* __restrict__ dfl, int64_t n, double df,
                                                         int64_t k0, int64_t k1, double f_low, double f_high,
                                                         double df_high, const double* __restrict__ pw,
                                                         int64_t stride, double2* __restrict__ K) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int j = blockIdx.y;
  double2 out = make_double2(0.0, 0.0);
  if (k > 0 && k <= n / 2) {
    const double inv_n = 1.0 / (double)n;  // n a power of two: exact
    const double a =
        k >= k0 && k <= k1 ? inv_n : inv_n * window_w((double)k * df, f_low, f_high, dfl[j], df_high);
    if (a > 0.0) {
      double s, c;
      sincospi(2.0 * tf2_turn(rp[j].q, k, pw[k], pw[stride + k], pw[2 * stride + k]), &s, &c);
      out = make_double2(a * c, a * s);
    }
  }
  K[(int64_t)j * n + k] = out;
}

// ---------------------------------------------------------------- pairs
// exp(-2 pi i m / nb) as pairs, from the FP64 table of n entries
__global__ void __launch_bounds__(256) k_split_roots(const double2* __restrict__ tw, int64_t stride, int64_t nb,
                                                     cdf* __restrict__ out) {
  const int64_t m = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (m >= nb) return;
  const double2 w = tw[m * stride];
  const float x = (float)w.x, y = (float)w.y;
  out[m] = cdf{make_float2(x, y), make_float2((float)(w.x - (double)x), (float)(w.y - (double)y))};
}

// exp(i (Psi_j - Psi_ref)) of bin k.  The phase is in 4096ths of a turn: the leading term, of up to
// 10^6 of them, in FP64, reduced to a whole number and a rest that leaves the FP64 pipe as a
// fixed-point number (its conversions to FP32 run at that pipe's rate); the others, fifty times smaller, in pairs
// (2^-46 of them is 10^-12 of a turn).  Then the nearest 4096th root of unity and the series of the rest,
// whose angle is below 7.7e-4 (relative errors of FP32 in its square and cube: 2e-14 and less).
struct PairPhase {
  double b0, d;
  Tf2Pairs q;
};
__device__ __forceinline__ cdf expi_phase(const PairPhase& f, int64_t k, double u5d, Pair u, Pair u5, Pair lu,
                                          const cdf* __restrict__ roots, int64_t root_step) {
  double t = u5d * f.b0;
  if (f.d != 0.0) t = fma((double)k, f.d, t);
  const double big = 6755399441055744.0;  // 1.5 2^52: the sum's low bits are the nearest whole number's
  const double r = t + big;
  const double rest = t - (r - big);
  constexpr double fix = 1536.0;  // 1.5 2^10: rest in units of 2^-42
  const long long i = __double_as_longlong(rest + fix) - 0x4098000000000000ll;
  const Pair p = pair_add(pair_mul(u, pair_add(pair_mul(u, f.q.b4), f.q.b3)), f.q.b2);
  const Pair low = pair_mul(pair_mul(u5, pair_mul(u, u)), p);
  const Pair high = pair_mul(u, pair_add(pair_mul(f.q.l6, lu), pair_add(pair_mul(f.q.b7, u), f.q.m6)));
  const Pair s = pair_add(low, pair_add(high, pair_add(pair_mul(f.q.l5, lu), f.q.e)));
  const float whole = rintf(s.h);
  // the rest's two halves are exact in FP32: 22 bits and sign, 20 bits
  const Pair fx{(float)(int)(i >> 20) * 2.384185791015625e-07f, (float)(int)(i & 0xfffff) * 2.2737367544323206e-13f};
  Pair d = pair_add(fx, Pair{__fadd_rn(s.h, -whole), s.l});
  const float m = rintf(d.h);
  const int idx = __double2loint(r) + (int)whole + (int)m;
  const float dh = __fadd_rn(__fadd_rn(d.h, -m), d.l);  // and what that sum loses
  const float dl = __fadd_rn(__fadd_rn(__fadd_rn(d.h, -m), -dh), d.l);
  constexpr double two_pi = 6.28318530717958647692528676655900577 / 4096.0;
  constexpr float ph = (float)two_pi, pl = (float)(two_pi - (double)ph);
  const float ah = __fmul_rn(dh, ph);
  const float al = __fmaf_rn(dh, ph, -ah) + (dh * pl + dl * ph);
  const float q = __fmaf_rn(ah, ah, 2.f * ah * al);
  const float c1 = q * __fmaf_rn(q, 1.f / 24.f, -0.5f);
  const float ch = __fadd_rn(1.f, c1);
  const cdf e{make_float2(ch, ah),
              make_float2(__fadd_rn(c1, -__fadd_rn(ch, -1.f)), al + ah * q * __fmaf_rn(q, 1.f / 120.f, -1.f / 6.f))};
  return cmul(e, cconj_pair(roots[(int64_t)(idx & 4095) * root_step]));
}

// First radix-16 pass of row blockIdx.y with K~ (as k_kernel_spectrum) formed on load: its bins above
// n/2 are zero, so half of the inputs are never formed and the spectrum never reaches memory.
__global__ void __launch_bounds__(128) k_pair_first(const RowPhase* __restrict__ rp, const double* __restrict__ dfl,
                                                    int64_t n, double df, int64_t k0, int64_t k1, double f_low,
                                                    double f_high, double df_high, const double* __restrict__ pw,
                                                    const float2* __restrict__ pw32, int64_t stride,
                                                    const cdf* __restrict__ roots, cdf* __restrict__ out) {
  const int64_t nq = n / 16;
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= nq) return;
  const int j = blockIdx.y;
  const Tf2Bins q = rp[j].q;  // in 4096ths of a turn
  const PairPhase f{q.b0, q.d,
                    make_tf2_pairs(q)};
  const float inv_n = 1.f / (float)n;  // n a power of two: exact
  const int64_t root_step = n / 4096;
  auto spectrum = [&](int64_t k) {
    cdf v{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    const bool in = k >= k0 && k <= k1;
    double w = 1.0;
    bool any = in;
    if (!in && k > 0) {
      w = window_w((double)k * df, f_low, f_high, dfl[j], df_high);
      any = w > 0.0;
    }
    if (any) {
      const float2 u = pw32[k], u5 = pw32[stride + k], lu = pw32[2 * stride + k];
      v = expi_phase(f, k, pw[stride + k], Pair{u.x, u.y}, Pair{u5.x, u5.y}, Pair{lu.x, lu.y}, roots, root_step);
      if (!in) {
        const float wh = (float)w, wl = (float)(w - (double)wh);
        v = cmul(v, cdf{make_float2(wh, 0.f), make_float2(wl, 0.f)});
      }
      v.h = make_float2(v.h.x * inv_n, v.h.y * inv_n);
      v.l = make_float2(v.l.x * inv_n, v.l.y * inv_n);
    }
    return v;
  };
  cdf a[16];
#pragma unroll 1
  for (int t = 0; t < 8; ++t) {
    const cdf v = spectrum(i + t * nq);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u == t) a[u] = v;  // one copy of the spectrum's code, registers indexed at compile time
  }
  const cdf zero{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  a[8] = i == 0 ? spectrum(n / 2) : zero;
#pragma unroll
  for (int t = 9; t < 16; ++t) a[t] = zero;
  cdf_dft<16>(a);
  cdf* o = out + (int64_t)j * n + i * 16;
#pragma unroll
  for (int t = 0; t < 16; ++t) o[t] = a[t];
}

// A later radix-R pass (fft.cu's scheme), sign +1.
template <int R>
__global__ void __launch_bounds__(128) k_pair_pass(const cdf* __restrict__ in, cdf* __restrict__ out, int64_t n,
                                                   int64_t Ns, const cdf* __restrict__ roots) {
  const int64_t nb = n / R;
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= nb) return;
  in += (int64_t)blockIdx.y * n;
  out += (int64_t)blockIdx.y * n;
  const int64_t k = i & (Ns - 1);
  const int64_t step = k * (n / (Ns * R));
  cdf a[R];
#pragma unroll
  for (int t = 0; t < R; ++t) a[t] = in[i + t * nb];
#pragma unroll
  for (int t = 1; t < R; ++t) a[t] = cmul(a[t], cconj_pair(roots[t * step]));
  cdf_dft<R>(a);
  const int64_t base = (i - k) * R + k;
#pragma unroll
  for (int t = 0; t < R; ++t) out[base + t * Ns] = a[t];
}

// The passes after the first; returns the buffer with the result.
cdf* pair_passes(cdf* cur, cdf* other, int64_t n, int batch, const cdf* roots, cudaStream_t s) {
  for (int64_t Ns = 16; Ns < n;) {
    const int64_t left = n / Ns;
    auto pass = [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      k_pair_pass<R><<<dim3((unsigned)((n / R + 127) / 128), (unsigned)batch), 128, 0, s>>>(cur, other, n, Ns, roots);
      RF_LAUNCHED();
      Ns *= R;
    };
    if (left >= 16) pass(std::integral_constant<int, 16>{});
    else if (left == 8) pass(std::integral_constant<int, 8>{});
    else if (left == 4) pass(std::integral_constant<int, 4>{});
    else pass(std::integral_constant<int, 2>{});
    std::swap(cur, other);
  }
  return cur;
}

__device__ __forceinline__ double mag2_rn(double2 v) { return __dadd_rn(__dmul_rn(v.x, v.x), __dmul_rn(v.y, v.y)); }

// The magnitudes are compared as integers (non-negative doubles order as their bits) and formed only
// where they can matter: a value whose parts are both below `floor_hi` (high words) has
// x^2 + y^2 below the bound that gave floor_hi, so the FP64 pipe (two lanes per SM) is left out of
// most of the rows.
__device__ __forceinline__ unsigned part_hi(double2 v) {
  return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
}
// High word below which both parts of a value with x^2 + y^2 >= m2 cannot lie: of sqrt(m2 / 2) (1 - 2^-19).
__device__ __forceinline__ unsigned floor_hi(double m2, double2) {
  return (unsigned)__double2hiint(sqrt(0.5 * m2) * (1.0 - 1.9073486328125e-06));
}
// The same for pairs, by the bits of h + l rounded to FP32 (2^-18 covers the rounding).  h alone will
// not do: the pairs are not renormalised, so after a cancellation l is of the size of the rounding of
// the terms that cancelled, up to a quarter of a value 1e-7 of the row's largest.
__device__ __forceinline__ double2 wide(cdf v) {
  return make_double2((double)v.h.x + (double)v.l.x, (double)v.h.y + (double)v.l.y);
}
__device__ __forceinline__ double mag2_rn(cdf v) { return mag2_rn(wide(v)); }
__device__ __forceinline__ unsigned part_hi(cdf v) {
  const float2 s = cadd(v.h, v.l);
  return max(__float_as_uint(s.x) & 0x7fffffffu, __float_as_uint(s.y) & 0x7fffffffu);
}
__device__ __forceinline__ unsigned floor_hi(double m2, cdf) {
  return __float_as_uint((float)(sqrt(0.5 * m2) * (1.0 - 3.814697265625e-06)));
}

// max |rho|^2 of a row's part (blockIdx.x of gridDim.x, row blockIdx.y) into amax2 (bits; 0 before).
// One block per row left most SMs idle: 612 us for 48 rows of 2^19 values.
template <typename V>
__global__ void __launch_bounds__(256) k_row_max2(const V* __restrict__ rho, int64_t n,
                                                  unsigned long long* __restrict__ amax2) {
  const V* r = rho + (int64_t)blockIdx.y * n;
  unsigned long long m = 0;
  unsigned lim = 0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const V v = r[i];
    if (part_hi(v) < lim) continue;
    asm volatile("" ::: "memory");  // no FP64 for the values left out
    const double a = mag2_rn(v);
    if (a > __longlong_as_double((long long)m)) {  // NaN never counts
      m = (unsigned long long)__double_as_longlong(a);
      lim = floor_hi(a, V{});
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0 && m) atomicMax(amax2 + blockIdx.y, m);
}

struct ArcBest {
  long long gap, m0;
};

__device__ __forceinline__ long long arc_key(long long m, long long n) { return m <= n / 2 ? m : m - n; }

__device__ __forceinline__ void arc_take(ArcBest& b, long long gap, long long m, long long n) {
  if (gap > b.gap || (gap == b.gap && arc_key(m, n) < arc_key(b.m0, n))) {
    b.gap = gap;
    b.m0 = m;
  }
}

// Kept lags of a contiguous range: first and last (-1: none), the widest gap between two
// consecutive ones with the lag after it, and whether some lag's value is too near the cut to say.
struct ArcPart {
  long long first, last;
  ArcBest best;
  int unsure;
};

// b followed by a later range c
__device__ __forceinline__ void arc_join(ArcPart& b, const ArcPart& c, long long n) {
  b.unsure |= c.unsure;
  if (c.first < 0) return;
  if (b.last >= 0) arc_take(b.best, c.first - b.last - 1, c.first, n);
  if (c.best.gap >= 0) arc_take(b.best, c.best.gap, c.best.m0, n);
  if (b.first < 0) b.first = c.first;
  b.last = c.last;
}

// Shortest covering arc of {m : |rho[m]|^2 >= cut2}, first step: a warp summarises `per` consecutive
// lags, 32 at a time by ballot.  (One block per row with a range per thread read its 2^19 values at a
// stride: 676 us for 48 rows.)  Pairs: lags whose |rho| is within eps of the row's largest of the cut
// are reported (rp).  The values are compared as integers, so that this costs no FP64.
template <typename V>
__global__ void __launch_bounds__(256) k_arc_parts(const V* __restrict__ rho, int64_t n, int per, int nparts,
                                                   const double* __restrict__ amax2,
                                                   const RowPhase* __restrict__ rp, double thr, int relative,
                                                   ArcPart* __restrict__ parts) {
  const int j = blockIdx.y;
  const int part = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (part >= nparts) return;
  const int lane = threadIdx.x & 31;
  const V* r = rho + (int64_t)j * n;
  const double cut2 = __dmul_rn(__dmul_rn(thr, thr), relative ? amax2[j] : 1.0);
  // (|rho| -+ eps max)^2 of cut2, the square of eps in the 2^-10
  const double band = std::is_same<V, cdf>::value ? (2.0 + 0x1p-10) * rp[j].eps * thr * amax2[j] : 0.0;
  const unsigned lim = floor_hi(fmax(0.0, cut2 - band), V{});
  using U64 = unsigned long long;
  const U64 cut_bits = (U64)__double_as_longlong(cut2), inf_bits = 0x7ff0000000000000ull;
  const U64 lo_bits = (U64)__double_as_longlong(fmax(0.0, cut2 - band));
  const U64 band_bits = (U64)__double_as_longlong(cut2 + band) - lo_bits;
  bool near = false;
  ArcPart b{-1, -1, {-1, 0}, 0};
  if (!relative || amax2[j] > 0.0) {
    const int64_t lo = (int64_t)part * per, hi = min(n, lo + per);
    // eight groups loaded ahead; FP64 is entered only where a warp has a candidate (the empty asm keeps
    // the compiler from evaluating it for every value, which took 333 to 700 us)
    constexpr int U = 8;
    unsigned masks[U];
    for (int64_t base = lo; base < hi; base += 32) {
      const int u = (int)((base - lo) / 32) % U;
      if (u == 0) {
        V v[U];
#pragma unroll
        for (int g = 0; g < U; ++g) {
          const int64_t m = base + 32 * g + lane;
          v[g] = m < hi ? r[m] : V{};
        }
        unsigned any = 0;
#pragma unroll
        for (int g = 0; g < U; ++g) {
          masks[g] = __ballot_sync(0xffffffffu, part_hi(v[g]) >= lim && base + 32 * g + lane < hi);
          any |= masks[g];
        }
        if (!any) {
          base += 32 * (U - 1);
          continue;
        }
#pragma unroll
        for (int g = 0; g < U; ++g)
          if (masks[g]) {
            asm volatile("" ::: "memory");
            const bool cand = (masks[g] >> lane) & 1u;
            const U64 m2 = cand ? (U64)__double_as_longlong(mag2_rn(v[g])) : ~0ull;
            masks[g] = __ballot_sync(0xffffffffu, m2 >= cut_bits && m2 <= inf_bits);
            if (std::is_same<V, cdf>::value) near |= m2 - lo_bits <= band_bits;
          }
      }
      unsigned mask = 0;
#pragma unroll
      for (int g = 0; g < U; ++g)
        if (g == u) mask = masks[g];
      if (!mask) continue;
      const int f = __ffs(mask) - 1;
      if (b.last >= 0) arc_take(b.best, base + f - b.last - 1, base + f, n);
      if (b.first < 0) b.first = base + f;
      // The lags after the first of the group.  Neighbouring lags are gaps of width 0, which matter only
      // while no wider gap is known: then the smallest signed lag of them, the first above n/2 or the
      // first.  (Taking every lag of a dense range in turn made its few warps the launch's tail.)
      unsigned rest = mask & (mask - 1);
      if (b.best.gap < 1) {
        const unsigned z = rest & (mask << 1);
        if (z) {
          arc_take(b.best, 0, base + __ffs(z) - 1, n);
          const int64_t s = n / 2 + 1 - base;  // lags from here on are negative ones
          const unsigned z2 = s <= 0 ? z : (s < 32 ? z >> s << s : 0u);
          if (z2) arc_take(b.best, 0, base + __ffs(z2) - 1, n);
        }
      }
      rest &= ~(mask << 1);
      while (rest) {
        const int q = __ffs(rest) - 1;
        rest &= rest - 1;
        const int before = 31 - __clz(mask & ((1u << q) - 1u));
        arc_take(b.best, q - before - 1, base + q, n);
      }
      b.last = base + 31 - __clz(mask);
    }
  }
  if (std::is_same<V, cdf>::value) b.unsure = __any_sync(0xffffffffu, near);
  if (lane == 0) parts[(int64_t)j * nparts + part] = b;
}

// Second step, a warp per row: the ranges joined in order, then the circle closed.  A row with a lag
// too near the cut has len = -len - 1.
__global__ void __launch_bounds__(32) k_arc_join(const ArcPart* __restrict__ parts, int nparts, int64_t n,
                                                 int* __restrict__ m0_out, int* __restrict__ len_out) {
  const int j = blockIdx.x, lane = threadIdx.x;
  const int ch = (nparts + 31) / 32;
  ArcPart b{-1, -1, {-1, 0}, 0};
  for (int q = lane * ch; q < min(nparts, (lane + 1) * ch); ++q) arc_join(b, parts[(int64_t)j * nparts + q], n);
  ArcPart g{-1, -1, {-1, 0}, 0};
  for (int l = 0; l < 32; ++l) {
    ArcPart c;
    c.first = __shfl_sync(0xffffffffu, b.first, l);
    c.last = __shfl_sync(0xffffffffu, b.last, l);
    c.best.gap = __shfl_sync(0xffffffffu, b.best.gap, l);
    c.best.m0 = __shfl_sync(0xffffffffu, b.best.m0, l);
    c.unsure = __shfl_sync(0xffffffffu, b.unsure, l);
    arc_join(g, c, n);
  }
  if (lane) return;
  int m0 = 0, len = 0;
  if (g.first >= 0) {
    arc_take(g.best, g.first + n - g.last - 1, g.first, n);
    m0 = (int)arc_key(g.best.m0, n);
    len = (int)(n - g.best.gap);
  }
  m0_out[j] = m0;
  len_out[j] = g.unsure ? -len - 1 : len;
}

// Row at[blockIdx.y] of pairs from row blockIdx.y in FP64.
__global__ void __launch_bounds__(256) k_rows_to_pairs(const double2* __restrict__ in, const int* __restrict__ at,
                                                       int64_t n, cdf* __restrict__ out) {
  in += (int64_t)blockIdx.y * n;
  out += (int64_t)at[blockIdx.y] * n;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const double2 v = in[i];
    const float2 h = make_float2((float)v.x, (float)v.y);
    out[i] = cdf{h, make_float2((float)(v.x - (double)h.x), (float)(v.y - (double)h.y))};
  }
}

template <typename R>
__device__ __forceinline__ R tap_x(double2 v) { return (R)v.x; }
template <typename R>
__device__ __forceinline__ R tap_y(double2 v) { return (R)v.y; }
template <typename R>
__device__ __forceinline__ R tap_x(cdf v) { return (R)(v.h.x + v.l.x); }
template <typename R>
__device__ __forceinline__ R tap_y(cdf v) { return (R)(v.h.y + v.l.y); }

template <typename V, typename W>
__global__ void __launch_bounds__(256) k_pack(const W* __restrict__ rho, int64_t n, const int* __restrict__ m0,
                                              const int* __restrict__ len, const int64_t* __restrict__ off,
                                              V* __restrict__ taps) {
  using R = typename real_of<V>::type;
  const int j = blockIdx.y;
  const int L = len[j];
  const int64_t mask = n - 1;
  for (int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; l < L; l += (int64_t)gridDim.x * blockDim.x) {
    const W v = rho[(int64_t)j * n + ((m0[j] + l) & mask)];
    taps[off[j] + l] = cmake<V>(tap_x<R>(v), tap_y<R>(v));
  }
}

// Real-kernel form: the real parts only (the imaginary parts are zero after k_real_form).
template <typename R, typename W>
__global__ void __launch_bounds__(256) k_pack_real(const W* __restrict__ rho, int64_t n,
                                                   const int* __restrict__ m0, const int* __restrict__ len,
                                                   const int64_t* __restrict__ off, R* __restrict__ taps) {
  const int j = blockIdx.y;
  const int L = len[j];
  const int64_t mask = n - 1;
  for (int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; l < L; l += (int64_t)gridDim.x * blockDim.x)
    taps[off[j] + l] = tap_x<R>(rho[(int64_t)j * n + ((m0[j] + l) & mask)]);
}

}  // namespace

rf_kernels* build_impl(rf_ctx* c, const rf_template& ref, const rf_template* nbrs, int32_t k, const double* inv_psd,
                       double thr, int relative, int64_t n_build, cudaStream_t s) {
  const int64_t n = c->n;
  const bool f64 = c->g.dtype == RF_F64;
  const bool real_form = (relative & RF_KERNEL_REAL) != 0;

  std::unique_ptr<rf_kernels> owner(new rf_kernels());
  rf_kernels* kern = owner.get();
  kern->k = k;
  kern->n = n;
  kern->real = real_form;
  kern->dtype = c->g.dtype;
  const size_t esz = tap_bytes(kern);
  kern->len.assign(k, 0);
  kern->lag0.assign(k, 0);
  kern->offset.assign((size_t)k + 1, 0);
  kern->df_low.assign(k, 0.0);
  kern->grid.assign(k, n);
  if (k == 0) {
    kern->taps.ensure(16);
    kern->len_d.ensure(16);
    kern->lag0_d.ensure(16);
    kern->off_d.ensure(16);
    RF_CUDA(cudaMemsetAsync(kern->off_d.p, 0, sizeof(int64_t), s));
    RF_CUDA(cudaStreamSynchronize(s));
    return owner.release();
  }

  // device scratch: [Tf2 k][dfl k][extent k][Tf2 k, grid order][dfl k, grid order]
  // [phase differences][amax2][m0][len]
  const int64_t kmax_chunk = std::min<int64_t>(k, 4096);
  const size_t meta_bytes = 2 * sizeof(Tf2) * (size_t)k + sizeof(double) * (3 * (size_t)k + 8 + kmax_chunk) +
                            (sizeof(RowPhase) + 2 * sizeof(int)) * (size_t)kmax_chunk + 8192;
  StreamBuf meta(c, meta_bytes, s);
  char* mp = meta.need().as<char>();
  auto carve = [&](size_t bytes) {
    char* r = mp;
    mp += (bytes + 255) & ~(size_t)255;
    return r;
  };
  Tf2* d_tg = reinterpret_cast<Tf2*>(carve(sizeof(Tf2) * k));
  double* d_dfl = reinterpret_cast<double*>(carve(sizeof(double) * k));
  double* d_ext = reinterpret_cast<double*>(carve(sizeof(double) * k));
  Tf2* d_tgs = reinterpret_cast<Tf2*>(carve(sizeof(Tf2) * k));
  double* d_dfls = reinterpret_cast<double*>(carve(sizeof(double) * k));
  RowPhase* d_rp = reinterpret_cast<RowPhase*>(carve(sizeof(RowPhase) * kmax_chunk));
  double* d_amax = reinterpret_cast<double*>(carve(sizeof(double) * kmax_chunk));
  int* d_m0 = reinterpret_cast<int*>(carve(sizeof(int) * kmax_chunk));
  int* d_len = reinterpret_cast<int*>(carve(sizeof(int) * kmax_chunk));
  RF_REQUIRE((size_t)(mp - meta.as<char>()) <= meta_bytes, "builder: scratch layout");

  std::vector<Tf2> tg(k);
  for (int j = 0; j < k; ++j) tg[j] = make_tf2(nbrs[j], c->g.pn_order);
  RF_CUDA(cudaMemcpyAsync(d_tg, tg.data(), sizeof(Tf2) * k, cudaMemcpyHostToDevice, s));
  const Tf2 pr = make_tf2(ref, c->g.pn_order);
  k_df_low<<<(k + 127) / 128, 128, 0, s>>>(pr, d_tg, k, c->g.f_low, c->g.df_low_max, d_dfl);
  RF_LAUNCHED();
  RF_CUDA(cudaMemcpyAsync(kern->df_low.data(), d_dfl, sizeof(double) * k, cudaMemcpyDeviceToHost, s));
  // build grid per neighbour
  if (n_build < 0) {
    std::vector<double> ext(k);
    k_grid_extent<<<(k + 127) / 128, 128, 0, s>>>(pr, d_tg, d_dfl, k, c->g.fs, c->g.f_low, c->g.f_high, c->g.df_high,
                                                  d_ext);
    RF_LAUNCHED();
    RF_CUDA(cudaMemcpyAsync(ext.data(), d_ext, sizeof(double) * k, cudaMemcpyDeviceToHost, s));
    RF_CUDA(cudaStreamSynchronize(s));
    for (int j = 0; j < k; ++j) {
      int64_t nb = 16;
      while ((double)nb < 4.0 * ext[j] && nb < n) nb *= 2;
      kern->grid[j] = std::min<int64_t>(nb, n);
    }
  } else if (n_build > 0) {
    for (int j = 0; j < k; ++j) kern->grid[j] = n_build;
  }
  RF_CUDA(cudaStreamSynchronize(s));  // df_low is on the host
  // which kernels are made in pairs (eps > 0; the rule above)
  const bool rel = relative & RF_TRUNC_RELATIVE, analytic = relative & RF_TRUNC_ANALYTIC;
  auto phase_of = [&](int j, double unit) {
    const double dfb = c->g.fs / (double)kern->grid[j];
    return tf2_bins_minus(make_tf2_bins(tg[j], dfb), make_tf2_bins(pr, dfb), unit);
  };
  std::vector<double> eps(k, 0.0);
  if (!f64 && (rel || analytic))
    for (int j = 0; j < k; ++j) {
      const int64_t nb = kern->grid[j];
      if (nb < kPairMinGrid) continue;
      const double dfb = c->g.fs / (double)nb;
      const double ka = std::max(1.0, std::floor((c->g.f_low - kern->df_low[j]) / dfb));
      const double kb = std::max(ka, std::min(0.5 * (double)nb, std::ceil((c->g.f_high + c->g.df_high) / dfb)));
      const Tf2Size size = tf2_bins_size(phase_of(j, 1.0), ka, kb);
      const double e = kPairTransformErr + kTwoPi * (size.lead * 0x1p-53 + size.rest * 0x1p-46);
      // (an absolute analytic amplitude shows its level only beside the largest value: k_analytic_span;
      // below 2^-30 of the phase every term also fits the integers of expi_phase)
      if (e <= (rel ? std::min(kPairTapErr * thr, 0x1p-30) : 0x1p-30)) eps[j] = e;
    }
  // neighbours in grid order (stable), FP64 before pairs; chunks of one grid and kind
  std::vector<int> order(k);
  for (int j = 0; j < k; ++j) order[j] = j;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return kern->grid[a] != kern->grid[b] ? kern->grid[a] < kern->grid[b] : (eps[a] > 0.0) < (eps[b] > 0.0);
  });
  bool identity = true;
  for (int q = 0; q < k && identity; ++q) identity = order[q] == q;
  if (identity) {
    d_tgs = d_tg;
    d_dfls = d_dfl;
  } else {
    std::vector<Tf2> tgs(k);
    std::vector<double> dfls(k);
    for (int q = 0; q < k; ++q) {
      tgs[q] = tg[order[q]];
      dfls[q] = kern->df_low[order[q]];
    }
    RF_CUDA(cudaMemcpyAsync(d_tgs, tgs.data(), sizeof(Tf2) * k, cudaMemcpyHostToDevice, s));
    RF_CUDA(cudaMemcpyAsync(d_dfls, dfls.data(), sizeof(double) * k, cudaMemcpyHostToDevice, s));
    RF_CUDA(cudaStreamSynchronize(s));  // the host vectors go out of scope
  }

  // per kernel: its taps in a part buffer (one per chunk) and its place there; a build of a single
  // chunk packs straight into the kernel set
  std::vector<std::unique_ptr<StreamBuf>> parts;
  std::vector<int> part_of(k);
  std::vector<int64_t> at_in_part(k);
  std::vector<int> hm0(kmax_chunk), hlen(kmax_chunk);
  std::vector<RowPhase> rp;
  std::vector<std::vector<int64_t>> off_host;
  // templates per chunk: three complex128 rows of nb per template (two of pairs), about 1.5 GB in total
  auto chunk_at = [&](int q0) {
    const int64_t nb = kern->grid[order[q0]];
    const int64_t per = 3 * nb * (int64_t)sizeof(double2);
    const int64_t most = std::min<int64_t>(kmax_chunk, std::max<int64_t>(1, ((int64_t)1536 << 20) / per));
    int cnt = 0;
    while (q0 + cnt < k && cnt < most && kern->grid[order[q0 + cnt]] == nb &&
           (eps[order[q0 + cnt]] > 0.0) == (eps[order[q0]] > 0.0))
      ++cnt;
    return cnt;
  };
  size_t rows_bytes = 0;
  for (int q0 = 0; q0 < k;) {
    const int cnt = chunk_at(q0);
    rows_bytes = std::max(rows_bytes, (size_t)3 * cnt * kern->grid[order[q0]] * sizeof(double2));
    q0 += cnt;
  }
  StreamBuf rows(c, rows_bytes, s);
  rows.need();
  int64_t roots_n = 0;
  for (int j = 0; j < k; ++j)
    if (eps[j] > 0.0) roots_n = std::max(roots_n, kern->grid[j]);
  StreamBuf roots(c, sizeof(cdf) * (size_t)roots_n, s);
  if (roots_n) roots.need();
  int64_t roots_of = 0;
  constexpr int kArcParts = 256;  // warps per row at most
  StreamBuf arcs(c, sizeof(ArcPart) * kArcParts * (size_t)kmax_chunk, s);
  arcs.need();
  const bool one_chunk = identity && chunk_at(0) == k;
  for (int q0 = 0; q0 < k;) {
    const int64_t nb = kern->grid[order[q0]];
    const int cnt = chunk_at(q0);
    const double dfb = c->g.fs / (double)nb;
    rf_grid gb = c->g;
    gb.n = nb;
    int64_t k0, k1;
    band_bins(gb, &k0, &k1);
    const bool pairs = eps[order[q0]] > 0.0;
    rp.resize(cnt);  // read by the copy until the chunk's synchronisation below
    // (for pairs in 4096ths of a turn, an exact scaling)
    for (int q = 0; q < cnt; ++q)
      rp[q] = RowPhase{phase_of(order[q0 + q], pairs ? 4096.0 : 1.0), eps[order[q0 + q]]};
    RF_CUDA(cudaMemcpyAsync(d_rp, rp.data(), sizeof(RowPhase) * cnt, cudaMemcpyHostToDevice, s));
    // rho of m rows: in FP64 (three rows of workspace each), and in the real form
    auto real_rows = [&](auto* R, int m) {
      if (!real_form) return;
      k_real_form<<<(unsigned)std::min<int64_t>(4096, (m * nb + 255) / 256), 256, 0, s>>>(R, m * nb);
      RF_LAUNCHED();
    };
    auto rows64 = [&](const RowPhase* d_p, const double* d_l, int m, double2* bufK) {
      double2* bufR = bufK + m * nb;
      double2* bufT = bufR + m * nb;
      k_kernel_spectrum<<<dim3((unsigned)((nb + 255) / 256), (unsigned)m), 256, 0, s>>>(
          d_p, d_l, nb, dfb, k0, k1, c->g.f_low, c->g.f_high, c->g.df_high, c->pw.as<double>(), c->pw_stride, bufK);
      RF_LAUNCHED();
      fft_c2c_f64(bufK, bufR, bufT, nb, m, +1, c->tw64.as<double2>(), n, s);
      real_rows(bufR, m);
      return bufR;
    };
    // the kept spans of m rows: first lags into d_s, lengths into d_n
    auto spans = [&](auto* R, const Tf2* d_t, const double* d_l, const RowPhase* d_p, int m, double* d_a, int* d_s,
                     int* d_n) {
      using V = std::remove_pointer_t<decltype(R)>;
      RF_CUDA(cudaMemsetAsync(d_a, 0, sizeof(double) * m, s));
      const unsigned mx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nb / 2048, (8LL * c->nsm + m - 1) / m));
      k_row_max2<V><<<dim3(mx, (unsigned)m), 256, 0, s>>>(R, nb, reinterpret_cast<unsigned long long*>(d_a));
      RF_LAUNCHED();
      if (analytic) {
        k_analytic_span<<<(m + 63) / 64, 64, 0, s>>>(pr, d_t, d_l, d_a, std::is_same<V, cdf>::value ? d_p : nullptr,
                                                     m, thr, rel, real_form ? 1.0 : 2.0, nb, c->g.fs, c->g.f_low,
                                                     c->g.f_high, c->g.df_high, d_s, d_n);
      } else {
        const int per = (int)std::max<int64_t>(32, nb / kArcParts);
        const int np = (int)((nb + per - 1) / per);
        k_arc_parts<V><<<dim3((unsigned)((np + 7) / 8), (unsigned)m), 256, 0, s>>>(R, nb, per, np, d_a, d_p, thr, rel,
                                                                                   arcs.as<ArcPart>());
        RF_LAUNCHED();
        k_arc_join<<<m, 32, 0, s>>>(arcs.as<ArcPart>(), np, nb, d_s, d_n);
      }
      RF_LAUNCHED();
    };
    double2* bufR = nullptr;
    cdf* bufP = nullptr;
    if (pairs) {
      if (roots_of != nb) {
        k_split_roots<<<(unsigned)((nb + 255) / 256), 256, 0, s>>>(c->tw64.as<double2>(), n / nb, nb, roots.as<cdf>());
        RF_LAUNCHED();
        roots_of = nb;
      }
      cdf* a = rows.as<cdf>();
      cdf* b = a + cnt * nb;
      k_pair_first<<<dim3((unsigned)((nb / 16 + 127) / 128), (unsigned)cnt), 128, 0, s>>>(
          d_rp, d_dfls + q0, nb, dfb, k0, k1, c->g.f_low, c->g.f_high, c->g.df_high, c->pw.as<double>(),
          c->pw32.as<float2>(), c->pw_stride, roots.as<cdf>(), a);
      RF_LAUNCHED();
      bufP = pair_passes(a, b, nb, cnt, roots.as<cdf>(), s);
      real_rows(bufP, cnt);
      spans(bufP, d_tgs + q0, d_dfls + q0, d_rp, cnt, d_amax, d_m0, d_len);
    } else {
      bufR = rows64(d_rp, d_dfls + q0, cnt, rows.as<double2>());
      spans(bufR, d_tgs + q0, d_dfls + q0, d_rp, cnt, d_amax, d_m0, d_len);
    }
    RF_CUDA(cudaMemcpyAsync(hm0.data(), d_m0, sizeof(int) * cnt, cudaMemcpyDeviceToHost, s));
    RF_CUDA(cudaMemcpyAsync(hlen.data(), d_len, sizeof(int) * cnt, cudaMemcpyDeviceToHost, s));
    RF_CUDA(cudaStreamSynchronize(s));
    // kernels in pairs whose span their error could change: again in FP64
    std::vector<int> redo;
    for (int q = 0; q < cnt; ++q)
      if (hlen[q] < 0) redo.push_back(q);
    for (size_t r0 = 0; r0 < redo.size();) {
      const int64_t per = 3 * nb * (int64_t)sizeof(double2);
      const int m = (int)std::min<int64_t>((int64_t)(redo.size() - r0),
                                           std::max<int64_t>(1, ((int64_t)512 << 20) / per));
      StreamBuf work(c, (size_t)(per * m), s);
      std::vector<Tf2> ht(m);
      std::vector<RowPhase> hp(m);
      std::vector<double> hl(m);
      std::vector<int> hs(m), hn(m);
      for (int i = 0; i < m; ++i) {
        const int j = order[q0 + redo[r0 + i]];
        ht[i] = tg[j];
        hp[i] = RowPhase{phase_of(j, 1.0), 0.0};
        hl[i] = kern->df_low[j];
      }
      StreamBuf bt(c, sizeof(Tf2) * m, s), bp(c, sizeof(RowPhase) * m, s), bl(c, 2 * sizeof(double) * m, s),
          bi(c, 3 * sizeof(int) * m, s);
      RF_CUDA(cudaMemcpyAsync(bt.need().p, ht.data(), sizeof(Tf2) * m, cudaMemcpyHostToDevice, s));
      RF_CUDA(cudaMemcpyAsync(bp.need().p, hp.data(), sizeof(RowPhase) * m, cudaMemcpyHostToDevice, s));
      RF_CUDA(cudaMemcpyAsync(bl.need().p, hl.data(), sizeof(double) * m, cudaMemcpyHostToDevice, s));
      RF_CUDA(cudaMemcpyAsync(bi.need().p, &redo[r0], sizeof(int) * m, cudaMemcpyHostToDevice, s));
      double2* R = rows64(bp.as<RowPhase>(), bl.as<double>(), m, work.need().as<double2>());
      spans(R, bt.as<Tf2>(), bl.as<double>(), bp.as<RowPhase>(), m, bl.as<double>() + m, bi.as<int>() + m,
            bi.as<int>() + 2 * m);
      k_rows_to_pairs<<<dim3((unsigned)std::min<int64_t>(1024, (nb + 255) / 256), (unsigned)m), 256, 0, s>>>(
          R, bi.as<int>(), nb, bufP);
      RF_LAUNCHED();
      RF_CUDA(cudaMemcpyAsync(hs.data(), bi.as<int>() + m, sizeof(int) * m, cudaMemcpyDeviceToHost, s));
      RF_CUDA(cudaMemcpyAsync(hn.data(), bi.as<int>() + 2 * m, sizeof(int) * m, cudaMemcpyDeviceToHost, s));
      RF_CUDA(cudaStreamSynchronize(s));
      for (int i = 0; i < m; ++i) {
        hm0[redo[r0 + i]] = hs[i];
        hlen[redo[r0 + i]] = hn[i];
      }
      r0 += m;
    }
    if (!redo.empty()) {
      RF_CUDA(cudaMemcpyAsync(d_m0, hm0.data(), sizeof(int) * cnt, cudaMemcpyHostToDevice, s));
      RF_CUDA(cudaMemcpyAsync(d_len, hlen.data(), sizeof(int) * cnt, cudaMemcpyHostToDevice, s));
      RF_CUDA(cudaStreamSynchronize(s));
    }
    std::vector<int64_t> off(cnt + 1, 0);
    for (int q = 0; q < cnt; ++q) {
      const int j = order[q0 + q];
      kern->lag0[j] = hm0[q];
      kern->len[j] = hlen[q];
      part_of[j] = (int)parts.size();
      at_in_part[j] = off[q];
      off[q + 1] = off[q] + hlen[q];
    }
    void* dst;
    if (one_chunk) {
      kern->taps.ensure(std::max<size_t>(16, (size_t)off[cnt] * esz));
      dst = kern->taps.p;
    } else {
      parts.emplace_back(new StreamBuf(c, (size_t)off[cnt] * esz, s));
      dst = parts.back()->need().p;
    }
    StreamBuf offd(c, sizeof(int64_t) * (cnt + 1), s);
    RF_CUDA(cudaMemcpyAsync(offd.need().p, off.data(), sizeof(int64_t) * (cnt + 1), cudaMemcpyHostToDevice, s));
    dim3 g2(64, (unsigned)cnt);
    const int64_t* od = offd.as<int64_t>();
    auto pack = [&](auto* src) {
      using S = std::remove_pointer_t<decltype(src)>;
      if (real_form && f64)
        k_pack_real<double, S><<<g2, 256, 0, s>>>(src, nb, d_m0, d_len, od, static_cast<double*>(dst));
      else if (real_form)
        k_pack_real<float, S><<<g2, 256, 0, s>>>(src, nb, d_m0, d_len, od, static_cast<float*>(dst));
      else if (f64)
        k_pack<double2, S><<<g2, 256, 0, s>>>(src, nb, d_m0, d_len, od, static_cast<double2*>(dst));
      else
        k_pack<float2, S><<<g2, 256, 0, s>>>(src, nb, d_m0, d_len, od, static_cast<float2*>(dst));
    };
    if (pairs) pack(bufP);
    else pack(bufR);
    RF_LAUNCHED();
    off_host.push_back(std::move(off));  // read by the copy above
    q0 += cnt;
  }
  for (int j = 0; j < k; ++j) kern->offset[j + 1] = kern->offset[j] + kern->len[j];
  const int64_t total = kern->offset[k];
  // taps in neighbour order: one copy per part when the order is unchanged, else one per kernel
  if (one_chunk) {
  } else if (kern->taps.ensure(std::max<size_t>(16, (size_t)total * esz)), identity) {
    int64_t at = 0;
    for (size_t pi = 0; pi < parts.size(); ++pi) {
      int64_t elems = 0;
      for (int j = 0; j < k; ++j)
        if (part_of[j] == (int)pi) elems += kern->len[j];
      if (elems)
        RF_CUDA(cudaMemcpyAsync(static_cast<char*>(kern->taps.p) + at * esz, parts[pi]->p, elems * esz,
                                cudaMemcpyDeviceToDevice, s));
      at += elems;
    }
  } else {
    for (int j = 0; j < k; ++j)
      if (kern->len[j])
        RF_CUDA(cudaMemcpyAsync(static_cast<char*>(kern->taps.p) + kern->offset[j] * esz,
                                static_cast<char*>(parts[part_of[j]]->p) + at_in_part[j] * esz,
                                (size_t)kern->len[j] * esz, cudaMemcpyDeviceToDevice, s));
  }
  kern->max_len = *std::max_element(kern->len.begin(), kern->len.end());
  kern->len_d.ensure(sizeof(int32_t) * k);
  kern->lag0_d.ensure(sizeof(int32_t) * k);
  kern->off_d.ensure(sizeof(int64_t) * (k + 1));
  RF_CUDA(cudaMemcpyAsync(kern->len_d.p, kern->len.data(), sizeof(int32_t) * k, cudaMemcpyHostToDevice, s));
  RF_CUDA(cudaMemcpyAsync(kern->lag0_d.p, kern->lag0.data(), sizeof(int32_t) * k, cudaMemcpyHostToDevice, s));
  RF_CUDA(cudaMemcpyAsync(kern->off_d.p, kern->offset.data(), sizeof(int64_t) * (k + 1), cudaMemcpyHostToDevice, s));
  RF_CUDA(cudaStreamSynchronize(s));
  return owner.release();
}

rf_kernels* import_impl(rf_ctx* c, int32_t k, const int32_t* lag0, const int32_t* len, const void* taps, bool real) {
  std::unique_ptr<rf_kernels> owner(new rf_kernels());
  rf_kernels* kern = owner.get();
  kern->k = k;
  kern->n = c->n;
  kern->dtype = c->g.dtype;
  kern->real = real;
  const size_t esz = tap_bytes(kern);
  kern->grid.assign(k, c->n);
  kern->len.assign(len, len + k);
  kern->lag0.assign(lag0, lag0 + k);
  kern->offset.assign((size_t)k + 1, 0);
  kern->df_low.assign(k, std::nan(""));
  for (int j = 0; j < k; ++j) kern->offset[j + 1] = kern->offset[j] + len[j];
  kern->max_len = k ? *std::max_element(kern->len.begin(), kern->len.end()) : 0;
  const int64_t total = kern->offset[k];
  kern->taps.ensure(std::max<size_t>(16, (size_t)total * esz));
  kern->len_d.ensure(std::max<size_t>(16, sizeof(int32_t) * k));
  kern->lag0_d.ensure(std::max<size_t>(16, sizeof(int32_t) * k));
  kern->off_d.ensure(sizeof(int64_t) * (k + 1));
  if (total) RF_CUDA(cudaMemcpy(kern->taps.p, taps, (size_t)total * esz, cudaMemcpyHostToDevice));
  if (k) {
    RF_CUDA(cudaMemcpy(kern->len_d.p, len, sizeof(int32_t) * k, cudaMemcpyHostToDevice));
    RF_CUDA(cudaMemcpy(kern->lag0_d.p, lag0, sizeof(int32_t) * k, cudaMemcpyHostToDevice));
  }
  RF_CUDA(cudaMemcpy(kern->off_d.p, kern->offset.data(), sizeof(int64_t) * (k + 1), cudaMemcpyHostToDevice));
  return owner.release();
}

}  // namespace rf
