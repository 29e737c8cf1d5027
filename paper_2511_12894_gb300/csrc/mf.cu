// Reference matched filter (Sec. II.A, Eqs. 2-4 and 6) and template spectra.
#include <algorithm>
#include <cmath>
#include <mutex>

#include <cuda.h>

#include "cplx.cuh"
#include "rf_internal.h"
#include "tf2.cuh"

namespace rf {

Tf2 make_tf2(const rf_template& t, int pn_order) {
  // Non-spinning TaylorF2 coefficients (Buonanno, Iyer, Ochsner, Pan & Sathyaprakash 2009),
  // truncated at v^pn_order.
  const double msun_s = 4.925491025543576e-6;
  const double pi = kPi;
  const double gamma_e = 0.57721566490153286061;
  Tf2 p{};
  const double mt = t.m1 + t.m2;
  p.M = mt * msun_s;
  p.eta = t.m1 * t.m2 / (mt * mt);
  p.tc = t.tc;
  p.phic = t.phic;
  p.pref = 3.0 / (128.0 * p.eta);
  const double e = p.eta;
  for (double& a : p.a) a = 0.0;
  p.a[0] = 1.0;
  if (pn_order >= 2) p.a[2] = 3715.0 / 756.0 + 55.0 / 9.0 * e;
  if (pn_order >= 3) p.a[3] = -16.0 * pi;
  if (pn_order >= 4) p.a[4] = 15293365.0 / 508032.0 + 27145.0 / 504.0 * e + 3085.0 / 72.0 * e * e;
  if (pn_order >= 5) {
    const double a5 = pi * (38645.0 / 756.0 - 65.0 / 9.0 * e);
    p.a[5] = a5;
    p.a5log = 3.0 * a5;
  }
  if (pn_order >= 6) {
    p.a[6] = 11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * pi * pi - 6848.0 / 21.0 * gamma_e +
             (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * pi * pi) * e + 76055.0 / 1728.0 * e * e -
             127825.0 / 1296.0 * e * e * e;
    p.a6log = -6848.0 / 21.0;
  }
  if (pn_order >= 7) p.a[7] = pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * e - 74045.0 / 756.0 * e * e);
  return p;
}

// The bins of the band: the k with f_low <= k df <= f_high, as compared in FP64 (k >= 1).
void band_bins(const rf_grid& g, int64_t* k0, int64_t* k1) {
  const double df = g.fs / (double)g.n;
  int64_t a = (int64_t)std::ceil(g.f_low / df), b = (int64_t)std::floor(g.f_high / df);
  while (a > 1 && (double)(a - 1) * df >= g.f_low) --a;
  while ((double)a * df < g.f_low) ++a;
  while ((double)(b + 1) * df <= g.f_high) ++b;
  while (b > 0 && (double)b * df > g.f_high) --b;
  *k0 = std::max<int64_t>(1, a);
  *k1 = std::min<int64_t>(g.n / 2, b);
}

namespace {

constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 512;
// Complex values of the four-step inverse transforms launched together (their intermediate).  Larger
// launches leave a smaller share of their last wave of blocks empty, which is worth more than an
// intermediate that fits L2 (the passes reach 20-40% of the HBM rate): 2^23, 2^24 and 2^25 values
// take 251, 243 and 232 us for 24 references of 2^20 samples, 694, 640 and 624 us for 6 of 2^23
// (with their window peaks).
constexpr int64_t kF4Chunk = int64_t(1) << 25;

// Tables of powers of the bin index k = 0..n/2 (rows of `stride`): k^(1/3), k^(-5/3), ln(k)/3 and
// k^(-7/6), 0 at k = 0.  The cube root is corrected by its exact residual, so the first two are good
// to about half an ulp.
// pw32 (if not null): the first three as FP32 pairs.
__global__ void __launch_bounds__(256) k_bin_powers(int64_t nbins, int64_t stride, double* __restrict__ pw,
                                                    float2* __restrict__ pw32) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nbins) return;
  double u = 0.0, u5 = 0.0, lu = 0.0, ua = 0.0;
  if (i > 0) {
    const double k = (double)i;
    const double r = rcbrt(k);
    // e = 1 - k r^3 from r^2 = r2 + r2l and r^3 = r3 + r3l (exact products): k^(-1/3) = r (1 + e / 3)
    const double r2 = r * r, r2l = fma(r, r, -r2);
    const double r3 = r2 * r, r3l = fma(r2, r, -r3) + r2l * r;
    const double kr = k * r3;
    const double e = (1.0 - kr) - (fma(k, r3, -kr) + k * r3l);
    const double c2 = r2l + r2 * (2.0 / 3.0) * e;  // k^(-2/3) = r2 + c2
    u = k * r2;
    u += fma(k, r2, -u) + k * c2;
    u5 = r2 / k;
    u5 += (fma(-u5, k, r2) + c2) / k;
    lu = log(k) / 3.0;
    ua = rsqrt(k) * (r2 + c2);
  }
  pw[i] = u;
  pw[stride + i] = u5;
  pw[2 * stride + i] = lu;
  pw[3 * stride + i] = ua;
  if (pw32) {
    const double t[3] = {u, u5, lu};
    for (int q = 0; q < 3; ++q) {
      const float h = (float)t[q];
      pw32[q * stride + i] = make_float2(h, (float)(t[q] - (double)h));
    }
  }
}

// Partial sums of 4 df B(f_k)^2 inv_psd[k] over the bins k0..k1 of the band, one partial per
// block; ua[k] = k^(-7/6), amp2 = 4 df df^(-7/3).
__global__ void __launch_bounds__(kRedThreads) k_sigma2_bins(const double* __restrict__ ip,
                                                             const double* __restrict__ ua, int64_t k0, int64_t k1,
                                                             double amp2, double* __restrict__ part) {
  double acc = 0.0;
  for (int64_t k = k0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k <= k1;
       k += (int64_t)gridDim.x * blockDim.x)
    acc = fma(ua[k] * ua[k], ip[k], acc);
  __shared__ double sh[kRedThreads];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = amp2 * sh[0];
}

// sigma^2 from the partials, by the first warp of a block in one fixed order (the same value in every
// block), and from it the filter scale 4 / (n sqrt(sigma^2)) df^(-7/6), for every thread.  A kernel of its
// own for this took 5.8 us of latency between the partials and the filters.
struct SigmaArgs {
  const double* part;
  int count;
  double n, amp;      // amp = df^(-7/6)
  double* sigma_out;  // null, or `nref` places for sigma (every template of the family has the same N)
  int nref;
};
__device__ __forceinline__ double sigma_scale(const SigmaArgs& a) {
  __shared__ double sh;
  if (threadIdx.x < 32) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < a.count; i += 32) acc += a.part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const double sg = sqrt(acc);
    if (threadIdx.x == 0) sh = 4.0 / (a.n * sg) * a.amp;
    if (blockIdx.x == 0 && a.sigma_out)
      for (int r = threadIdx.x; r < a.nref; r += 32) a.sigma_out[r] = sg;
  }
  __syncthreads();
  return sh;
}

constexpr int kFiltRefs = 8;  // references of one filter launch (their coefficients are arguments)
struct FiltRefs {
  Tf2Bins q[kFiltRefs];
};

// Filters F_r[k] = (4 / (n N)) conj(h~_r,k) inv_psd[k], k = 0..n/2, of `cnt` references; 0 outside
// the bins k0..k1 of the band.  With X the unnormalised DFT of the data, X[k] F_r[k] is the
// integrand of Eq. 2 (4 df dt = 4 / n).  One thread per bin: the tables and inv_psd are read once
// for all references.  PREC: phase, amplitude and product in FP64, rounded once (stored filters,
// FP64 grids); else (filters made and used within one call on an FP32 grid) the FP64 phase is reduced
// to a fraction of a turn before the FP32 sine and cosine.
template <typename V, bool PREC>
__global__ void __launch_bounds__(256) k_ref_filters(const double* __restrict__ ip, const double* __restrict__ pw,
                                                     int64_t stride, SigmaArgs sig, FiltRefs refs,
                                                     int cnt, int64_t nbins, int64_t k0, int64_t k1,
                                                     V* __restrict__ F, int64_t fstride) {
  using R = typename real_of<V>::type;
  const double scale = sigma_scale(sig);
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nbins) return;
  if (k < k0 || k > k1) {
    for (int r = 0; r < cnt; ++r) F[r * fstride + k] = cmake<V>((R)0, (R)0);
    return;
  }
  const double u = pw[k], u5 = pw[stride + k], lu = pw[2 * stride + k];
  const double a = scale * pw[3 * stride + k] * ip[k];
  for (int r = 0; r < cnt; ++r) {
    const double t = tf2_turn(refs.q[r], k, u, u5, lu);
    if constexpr (PREC) {
      double s, c;
      sincospi(2.0 * t, &s, &c);
      F[r * fstride + k] = cmake<V>((R)(a * c), (R)(a * s));  // conj(h~) = B exp(+i Psi)
    } else {
      float s, c;
      sincospif(2.0f * (float)t, &s, &c);
      F[r * fstride + k] = cmake<V>((R)a * c, (R)a * s);
    }
  }
}

// The same for FP32 grids with the phase in FP32 pairs, for templates with t_c = 0 whose phase stays
// below kPairTurns in the band.  Three references at n = 2^20: the FP64 phase took 49 us of the FP64
// pipe, this 12.5 us.  A pair keeps about 2^-46 of the phase; 2^18 turns of it (two bodies of 0.3 solar
// masses from 5 Hz, 1.0 from 2.4 Hz) leave 2^-28 of a turn, an eighth of the rounding of the angle to
// FP32 that follows in either form.  Bodies of 0.01 solar masses, 7e7 turns from 5 Hz, lost 1e-5 rad.
constexpr double kPairTurns = 262144.0;
struct FiltPairs {
  Tf2Pairs q[kFiltRefs];
};
__global__ void __launch_bounds__(256) k_ref_filters_pairs(const double* __restrict__ ip,
                                                           const double* __restrict__ ua,
                                                           const float2* __restrict__ pw32, int64_t stride,
                                                           SigmaArgs sig, FiltPairs refs, int cnt, int64_t nbins,
                                                           int64_t k0, int64_t k1,
                                                           float2* __restrict__ F, int64_t fstride) {
  const double scale = sigma_scale(sig);
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nbins) return;
  if (k < k0 || k > k1) {
    for (int r = 0; r < cnt; ++r) F[r * fstride + k] = make_float2(0.f, 0.f);
    return;
  }
  const float2 u = pw32[k], u5 = pw32[stride + k], lu = pw32[2 * stride + k];
  const float a = (float)(scale * ua[k] * ip[k]);
  for (int r = 0; r < cnt; ++r) {
    float s, c;
    sincospif(2.0f * tf2_turn(refs.q[r], Pair{u.x, u.y}, Pair{u5.x, u5.y}, Pair{lu.x, lu.y}), &s, &c);
    F[r * fstride + k] = make_float2(a * c, a * s);
  }
}

template <typename V>
__global__ void __launch_bounds__(256) k_template_fd(Tf2Bins q, const double* __restrict__ pw, int64_t stride,
                                                     double amp, int64_t nbins, V* __restrict__ h) {
  using R = typename real_of<V>::type;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nbins) return;
  V out = cmake<V>((R)0, (R)0);
  if (k > 0) {
    double s, c;
    sincospi(2.0 * tf2_turn(q, k, pw[k], pw[stride + k], pw[2 * stride + k]), &s, &c);
    const double a = amp * pw[3 * stride + k];
    out = cmake<V>((R)(a * c), (R)(-a * s));
  }
  h[k] = out;
}

// df^(-7/6)
double amp_scale(double df) { return 1.0 / (df * std::cbrt(std::sqrt(df))); }

// The partial sums of sigma^2; the filters finish them (and write sigma to sigma_out[nref], or null).
SigmaArgs launch_sigma2(rf_ctx* c, const double* inv_psd, double* sigma_out, int nref, cudaStream_t s) {
  const double df = c->g.fs / (double)c->n;
  int64_t k0, k1;
  band_bins(c->g, &k0, &k1);
  const double amp = amp_scale(df);
  double* part = c->red.as<double>();
  // two blocks per SM at most, so that the one-warp sum of the partials stays short
  const int blocks = (int)std::max<int64_t>(
      1, std::min<int64_t>(std::min(kRedBlocks, 2 * c->nsm), (k1 - k0 + 1) / (2 * kRedThreads)));
  k_sigma2_bins<<<blocks, kRedThreads, 0, s>>>(inv_psd, c->pw.as<double>() + 3 * c->pw_stride, k0, k1,
                                               4.0 * df * amp * amp, part);
  RF_LAUNCHED();
  return SigmaArgs{part, blocks, (double)c->n, amp, sigma_out, nref};
}

template <typename V, bool PREC>
void launch_filters(rf_ctx* c, const double* inv_psd, SigmaArgs sig, int cnt, const rf_template* refs, V* F,
                    int64_t fstride, cudaStream_t s) {
  const int64_t nbins = c->n / 2 + 1;
  const double df = c->g.fs / (double)c->n;
  int64_t k0, k1;
  band_bins(c->g, &k0, &k1);
  // Each reference in the form its own phase asks for, whatever else is in the call: launches of runs of
  // one kind (places beside the coefficients would mix kinds in a launch: 71 -> 73 us for three references at 2^20).
  const unsigned grid = (unsigned)((nbins + 255) / 256);
  FiltRefs fr;
  FiltPairs fp;
  for (int r0 = 0, m; r0 < cnt; r0 += m) {
    bool pairs = false;
    for (m = 0; m < kFiltRefs && r0 + m < cnt; ++m) {
      const Tf2Bins q = make_tf2_bins(make_tf2(refs[r0 + m], c->g.pn_order), df);
      const Tf2Size size = tf2_bins_size(q, (double)k0, (double)std::max(k0, k1));
      const bool p = !PREC && q.d == 0.0 && size.lead + size.rest <= kPairTurns;
      if (m > 0 && p != pairs) break;
      pairs = p;
      if (p) fp.q[m] = make_tf2_pairs(q);
      else fr.q[m] = q;
    }
    V* Fr = F + (int64_t)r0 * fstride;
    bool done = false;
    if constexpr (!PREC) {
      if (pairs) {
        k_ref_filters_pairs<<<grid, 256, 0, s>>>(inv_psd, c->pw.as<double>() + 3 * c->pw_stride, c->pw32.as<float2>(),
                                                 c->pw_stride, sig, fp, m, nbins, k0, k1, Fr, fstride);
        done = true;
      }
    }
    if (!done)
      k_ref_filters<V, PREC><<<grid, 256, 0, s>>>(inv_psd, c->pw.as<double>(), c->pw_stride, sig, fr, m, nbins, k0, k1,
                                                  Fr, fstride);
    RF_LAUNCHED();
    sig.sigma_out = nullptr;  // written once
  }
}

}  // namespace

void mf_create(rf_ctx* c) {
  const int64_t nbins = c->n / 2 + 1;
  c->pw_stride = (nbins + 15) & ~(int64_t)15;
  // Whole 2 MB pages: what is left of shared pages stays for the small buffers of later first calls
  // (a first tensor-core call of 16 neighbours at n = 2^16: 303 us without, 254 with this, mean of several).
  auto pages = [](size_t b) { return b > ((size_t)1 << 19) ? (b + ((size_t)1 << 21) - 1) >> 21 << 21 : b; };
  c->pw.ensure(pages(sizeof(double) * 4 * (size_t)c->pw_stride));
  const bool f32 = c->g.dtype == RF_F32;
  if (f32) c->pw32.ensure(pages(sizeof(float2) * 3 * (size_t)c->pw_stride));
  k_bin_powers<<<(unsigned)((nbins + 255) / 256), 256>>>(nbins, c->pw_stride, c->pw.as<double>(),
                                                         f32 ? c->pw32.as<float2>() : nullptr);
  RF_LAUNCHED();
  RF_CUDA(cudaStreamSynchronize(nullptr));
  // up to 8 references, 2^22 intermediate values in all (above that one reference fills the GPU)
  c->mf_batch = (int)std::max<int64_t>(1, std::min<int64_t>(8, ((int64_t)1 << 22) / c->n));
  const size_t esz = c->g.dtype == RF_F64 ? sizeof(double2) : sizeof(float2);
  if (c->mf_batch > 1) c->mf_ref.ensure(pages(esz * (size_t)c->mf_batch * (size_t)(c->n + nbins + 15)));
}

namespace {

// The context's transforms: two-pass four-step where n allows, else radix passes.
void forward_real(rf_ctx* c, const float* x, float2* X, float2* tmp, cudaStream_t s) {
  if (fft4_forward_supported(c->n, false)) fft4_forward_real(c, x, X, tmp, s);
  else fft_r2c_f32(x, X, tmp, c->n, c->tw32.as<float2>(), c->n, s);
}
void forward_real(rf_ctx* c, const double* x, double2* X, double2* tmp, cudaStream_t s) {
  if (fft4_forward_supported(c->n, true)) fft4_forward_real(c, x, X, tmp, s);
  else fft_r2c_f64(x, X, tmp, c->n, c->tw64.as<double2>(), c->n, s);
}
void inverse_product(rf_ctx* c, const float2* X, const float2* F, int64_t fstride, float2* z, float2* tmp, int cnt,
                     cudaStream_t s) {
  if (fft4_inverse_supported(c->n, false)) fft4_inverse_product(c, X, F, fstride, z, tmp, cnt, s);
  else ifft_product_f32(X, F, fstride, z, tmp, c->n, cnt, c->tw32.as<float2>(), c->n, s);
}
void inverse_product(rf_ctx* c, const double2* X, const double2* F, int64_t fstride, double2* z, double2* tmp, int cnt,
                     cudaStream_t s) {
  if (fft4_inverse_supported(c->n, true)) fft4_inverse_product(c, X, F, fstride, z, tmp, cnt, s);
  else ifft_product_f64(X, F, fstride, z, tmp, c->n, cnt, c->tw64.as<double2>(), c->n, s);
}

// The one-launch form reads the data and the filters in every block, after other blocks may have
// written their rows: inputs that the caller's output overlaps are copied first.
bool overlap(const void* a, size_t na, const void* b, size_t nb) {
  const char* p = static_cast<const char*>(a);
  const char* q = static_cast<const char*>(b);
  return p < q + nb && q < p + na;
}
const float* data_apart(rf_ctx* c, int nref, const void* x, const void* z, cudaStream_t s) {
  const size_t xb = sizeof(float) * (size_t)c->n;
  if (!overlap(x, xb, z, sizeof(float2) * (size_t)nref * (size_t)c->n)) return static_cast<const float*>(x);
  RF_CUDA(cudaMemcpyAsync(c->xf.p, x, xb, cudaMemcpyDeviceToDevice, s));
  return c->xf.as<float>();
}

// Filters of a batch, then one product inverse for the batch.
template <typename V, typename Inverse>
void mf_batches(rf_ctx* c, const double* inv_psd, SigmaArgs sig, int32_t nref, const rf_template* refs,
                V* z_out, Inverse&& inverse, cudaStream_t s) {
  constexpr bool PREC = sizeof(V) == sizeof(double2);
  const int64_t n = c->n, nbins = n / 2 + 1;
  const int64_t fstride = (nbins + 1) & ~(int64_t)1;
  const int batch = std::min<int>(c->mf_batch, nref);
  V* tmp = batch > 1 ? c->mf_ref.as<V>() : c->fb.as<V>();
  V* F = batch > 1 ? tmp + (int64_t)c->mf_batch * n : c->fa.as<V>();
  for (int r0 = 0; r0 < nref; r0 += batch) {
    const int cnt = std::min(batch, nref - r0);
    launch_filters<V, PREC>(c, inv_psd, sig, cnt, refs + r0, F, fstride, s);
    sig.sigma_out = nullptr;
    inverse(F, fstride, z_out + (int64_t)r0 * n, tmp, cnt);
  }
}

}  // namespace

void mf_reference_impl(rf_ctx* c, const void* x, const double* inv_psd, int32_t nref, const rf_template* refs,
                       void* z_out, double* sigma_out, cudaStream_t s) {
  const SigmaArgs sig = launch_sigma2(c, inv_psd, sigma_out, nref, s);
  if (c->g.dtype == RF_F64) {
    forward_real(c, static_cast<const double*>(x), c->xf.as<double2>(), c->fb.as<double2>(), s);
    mf_batches(c, inv_psd, sig, nref, refs, static_cast<double2*>(z_out),
               [&](const double2* F, int64_t fs, double2* z, double2* tmp, int cnt) {
                 inverse_product(c, c->xf.as<double2>(), F, fs, z, tmp, cnt, s);
               }, s);
  } else if (block_mf_supported(c, nref)) {
    const float* xa = data_apart(c, nref, x, z_out, s);
    mf_batches(c, inv_psd, sig, nref, refs, static_cast<float2*>(z_out),
               [&](const float2* F, int64_t fs, float2* z, float2*, int cnt) { block_mf(c, xa, F, fs, z, cnt, s); }, s);
  } else {
    forward_real(c, static_cast<const float*>(x), c->xf.as<float2>(), c->fb.as<float2>(), s);
    mf_batches(c, inv_psd, sig, nref, refs, static_cast<float2*>(z_out),
               [&](const float2* F, int64_t fs, float2* z, float2* tmp, int cnt) {
                 inverse_product(c, c->xf.as<float2>(), F, fs, z, tmp, cnt, s);
               }, s);
  }
}

void reference_filters_impl(rf_ctx* c, const double* inv_psd, int32_t nref, const rf_template* refs, void* filt,
                            double* sigma_out, cudaStream_t s) {
  const int64_t nb = c->n / 2 + 1;
  const SigmaArgs sig = launch_sigma2(c, inv_psd, sigma_out, nref, s);
  if (c->g.dtype == RF_F64)
    launch_filters<double2, true>(c, inv_psd, sig, nref, refs, static_cast<double2*>(filt), nb, s);
  else
    launch_filters<float2, true>(c, inv_psd, sig, nref, refs, static_cast<float2*>(filt), nb, s);
}

void mf_filtered_impl(rf_ctx* c, const void* x, int32_t nref, const void* filt, void* z_out, cudaStream_t s) {
  const int64_t n = c->n;
  const int64_t nb = n / 2 + 1;
  if (block_mf_supported(c, nref)) {
    const float* xa = data_apart(c, nref, x, z_out, s);
    const float2* F = static_cast<const float2*>(filt);
    const size_t fb = sizeof(float2) * (size_t)nref * (size_t)nb;
    if (overlap(filt, fb, z_out, sizeof(float2) * (size_t)nref * (size_t)n)) {
      void* copy = c->mf_tmp.ensure(fb);
      RF_CUDA(cudaMemcpyAsync(copy, filt, fb, cudaMemcpyDeviceToDevice, s));
      F = static_cast<const float2*>(copy);
    }
    block_mf(c, xa, F, nb, static_cast<float2*>(z_out), nref, s);
    return;
  }
  auto run = [&](auto vtag) {
    using V = decltype(vtag);
    using T = typename real_of<V>::type;
    // references per launch, bounded by the temporary buffer
    const int64_t most = fft4_inverse_supported(n, sizeof(T) == 8) ? std::max<int64_t>(1, kF4Chunk / n)
                                                           : std::min<int64_t>(65535, ((int64_t)1 << 27) / n);
    const int chunk = (int)std::max<int64_t>(1, std::min<int64_t>(nref, most));
    V* tmp = static_cast<V*>(c->mf_tmp.ensure(sizeof(V) * (size_t)chunk * n));
    forward_real(c, static_cast<const T*>(x), c->xf.as<V>(), tmp, s);
    for (int r0 = 0; r0 < nref; r0 += chunk) {
      const int cnt = std::min(chunk, nref - r0);
      inverse_product(c, c->xf.as<V>(), static_cast<const V*>(filt) + (int64_t)r0 * nb, nb,
                      static_cast<V*>(z_out) + (int64_t)r0 * n, tmp, cnt, s);
    }
  };
  if (c->g.dtype == RF_F64) run(double2{});
  else run(float2{});
}

void template_fd_impl(rf_ctx* c, const rf_template& t, void* h_out, cudaStream_t s) {
  const int64_t nbins = c->n / 2 + 1;
  const double df = c->g.fs / (double)c->n;
  const Tf2Bins q = make_tf2_bins(make_tf2(t, c->g.pn_order), df);
  const unsigned grid = (unsigned)((nbins + 255) / 256);
  if (c->g.dtype == RF_F64)
    k_template_fd<double2><<<grid, 256, 0, s>>>(q, c->pw.as<double>(), c->pw_stride, amp_scale(df), nbins,
                                                static_cast<double2*>(h_out));
  else
    k_template_fd<float2><<<grid, 256, 0, s>>>(q, c->pw.as<double>(), c->pw_stride, amp_scale(df), nbins,
                                               static_cast<float2*>(h_out));
  RF_LAUNCHED();
}

// ---------------------------------------------------------------- allocation-free variant
// rf_mf_reference_noalloc: the reference matched filter for callers that may not
// allocate device memory.  Its workspace is the file-scope array below (about
// 4 MiB, reserved in every GPU that loads the library, until the process exits).

namespace {

constexpr int64_t kNoAllocMaxN = int64_t(1) << 16;
constexpr size_t kNoAllocSlot = (size_t)kNoAllocMaxN * sizeof(double2);  // one complex128 row of kNoAllocMaxN
constexpr size_t kNoAllocRed = 8192;                                      // FP64 partial sums + sigma^2
constexpr size_t kNoAllocBytes = 4 * kNoAllocSlot + kNoAllocRed;
// The array has its own device address in every CUDA context that loads the module (the
// runtime's primary context of each device, or a context a host application created with
// the driver API), so the addresses are remembered per context, keyed by the context's
// process-unique ID (a handle value can be reused by a later context; the ID is not).
constexpr int kNoAllocCacheSlots = 64;
struct NoAllocSlot {
  unsigned long long ctx_id;
  void* addr;
};
std::mutex g_noalloc_mu;
NoAllocSlot g_noalloc_cache[kNoAllocCacheSlots] = {};
int g_noalloc_used = 0;
int g_noalloc_next = 0;

// The allocation-free form has no room for tables of bin powers and evaluates the template at
// every bin.

// Partial sums of 4 df B(f_k)^2 inv_psd[k] over the band, one partial per block.
__global__ void __launch_bounds__(kRedThreads) k_sigma2_partial(const double* __restrict__ ip, int64_t nbins,
                                                                double df, double f_low, double f_high,
                                                                double* __restrict__ part) {
  double acc = 0.0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nbins;
       k += (int64_t)gridDim.x * blockDim.x) {
    const double f = (double)k * df;
    if (f >= f_low && f <= f_high && k > 0) acc += exp(-7.0 / 3.0 * log(f)) * ip[k];
  }
  __shared__ double sh[kRedThreads];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = 4.0 * df * sh[0];
}

__global__ void k_sum_partials(const double* __restrict__ part, int count, double* __restrict__ out) {
  __shared__ double sh[kRedThreads];
  double acc = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) acc += part[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = sh[0];
}

// Z~[k] = (4 / (n N)) X[k] conj(h~_k) inv_psd[k] on the band, 0 elsewhere and for k > n/2.
// X is the unnormalised DFT of the data (x~ = dt X), so 4 df dt = 4 / n.
template <typename V>
__global__ void __launch_bounds__(256) k_mf_pointwise(const V* __restrict__ X, const double* __restrict__ ip,
                                                      const double* __restrict__ sigma2, Tf2 p, int64_t n,
                                                      double df, double f_low, double f_high, V* __restrict__ Z,
                                                      double* __restrict__ sigma_out) {
  using R = typename real_of<V>::type;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0 && sigma_out) sigma_out[0] = sqrt(sigma2[0]);
  if (k >= n) return;
  const double f = (double)k * df;
  V out = cmake<V>((R)0, (R)0);
  if (k <= n / 2 && k > 0 && f >= f_low && f <= f_high) {
    const double psi = tf2_phase(p, f);
    const double scale = 4.0 / ((double)n * sqrt(sigma2[0]));
    if constexpr (sizeof(R) == 8) {
      double s, c;
      sincos(psi, &s, &c);
      const double a = scale * tf2_amp(f) * ip[k];
      // conj(h~) = B exp(+i Psi)
      out = cmul(X[k], cmake<V>(a * c, a * s));
    } else {
      // reduce the FP64 phase to (-pi, pi] before the FP32 sine/cosine
      const double red = psi - kTwoPi * rint(psi * (1.0 / kTwoPi));
      float s, c;
      sincosf((float)red, &s, &c);
      const float a = (float)(scale * ip[k]) * powf((float)f, -7.0f / 6.0f);
      out = cmul(X[k], cmake<V>(a * c, a * s));
    }
  }
  Z[k] = out;
}

// exp(-2 pi i m / n), m < n, into the workspace (rebuilt on every call).
template <typename V>
__global__ void __launch_bounds__(256) k_noalloc_twiddles(V* __restrict__ tw, int64_t n) {
  using R = typename real_of<V>::type;
  const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n) return;
  double s, c;
  sincospi(2.0 * (double)m / (double)n, &s, &c);
  tw[m] = cmake<V>((R)c, (R)(-s));
}

}  // namespace

}  // namespace rf

// The workspace.  Host code must not use this name as an address: it is a host-side
// stand-in.  The device address comes from cudaGetSymbolAddress, once per device.
static __device__ __align__(256) unsigned char rf_noalloc_scratch[rf::kNoAllocBytes];

namespace rf {
namespace {

// Driver entry points for the current context and its ID, looked up once through the
// runtime (no link against the driver library).
using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

struct CtxFns {
  CtxGetCurrentFn get_current;
  CtxGetIdFn get_id;
};

const CtxFns& ctx_fns() {
  static const CtxFns fns = [] {
    CtxFns f{nullptr, nullptr};
    void* a = nullptr;
    void* b = nullptr;
    cudaDriverEntryPointQueryResult qa{}, qb{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 4000, cudaEnableDefault, &qa) == cudaSuccess &&
        qa == cudaDriverEntryPointSuccess)
      f.get_current = reinterpret_cast<CtxGetCurrentFn>(a);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb) == cudaSuccess &&
        qb == cudaDriverEntryPointSuccess)
      f.get_id = reinterpret_cast<CtxGetIdFn>(b);
    (void)cudaGetLastError();
    return f;
  }();
  return fns;
}

// Process-unique ID of the calling thread's current context, or 0 when none is current.
unsigned long long current_context_id() {
  const CtxFns& f = ctx_fns();
  RF_REQUIRE(f.get_current != nullptr && f.get_id != nullptr,
             "the driver does not provide cuCtxGetCurrent / cuCtxGetId");
  CUcontext ctx = nullptr;
  if (f.get_current(&ctx) != CUDA_SUCCESS || ctx == nullptr) return 0;
  unsigned long long id = 0;
  RF_REQUIRE(f.get_id(ctx, &id) == CUDA_SUCCESS, "cuCtxGetId failed on the current context");
  return id;
}

void* lookup_scratch_symbol() {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, rf_noalloc_scratch);
  if (e != cudaSuccess || p == nullptr) {
    (void)cudaGetLastError();
    set_error("cudaGetSymbolAddress of the static workspace failed: %s", cudaGetErrorString(e));
    throw Fail{RF_ECUDA};
  }
  return p;
}

// Device address of rf_noalloc_scratch in the calling thread's current context.  The
// set-up (cudaGetSymbolAddress) runs on the first call made in a context and its result is
// remembered for that context; a thread with no current context gets the runtime's
// primary context of its current device, which that first runtime call binds.
unsigned char* noalloc_scratch_address() {
  unsigned long long id = current_context_id();
  void* fresh = nullptr;
  if (id == 0) {
    fresh = lookup_scratch_symbol();  // binds the primary context
    id = current_context_id();
    RF_REQUIRE(id != 0, "no CUDA context is current after the workspace lookup");
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  for (int i = 0; i < g_noalloc_used; ++i)
    if (g_noalloc_cache[i].ctx_id == id) return static_cast<unsigned char*>(g_noalloc_cache[i].addr);
  if (!fresh) fresh = lookup_scratch_symbol();
  // remember it; with every slot taken, the oldest entry makes room
  int slot;
  if (g_noalloc_used < kNoAllocCacheSlots) {
    slot = g_noalloc_used++;
  } else {
    slot = g_noalloc_next;
    g_noalloc_next = (g_noalloc_next + 1) % kNoAllocCacheSlots;
  }
  g_noalloc_cache[slot] = NoAllocSlot{id, fresh};
  return static_cast<unsigned char*>(fresh);
}

void noalloc_check_dev(const void* p, const char* name, bool allow_null) {
  if (!p) {
    RF_REQUIRE(allow_null, "%s is NULL", name);
    return;
  }
  RF_REQUIRE(((uintptr_t)p & 15u) == 0, "%s is not 16-byte aligned", name);
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    (void)cudaGetLastError();
    RF_REQUIRE(false, "%s is not a CUDA device pointer", name);
  }
  RF_REQUIRE(at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged, "%s is not device memory", name);
}

void mf_reference_noalloc_impl(const rf_grid& g, const void* x, const double* inv_psd, const rf_template& ref,
                               void* z_out, double* sigma_out, cudaStream_t s) {
  RF_REQUIRE(g.n >= 256 && (g.n & (g.n - 1)) == 0, "n=%lld must be a power of two >= 256", (long long)g.n);
  RF_REQUIRE(g.n <= kNoAllocMaxN, "n=%lld exceeds the static workspace limit n <= %lld of rf_mf_reference_noalloc",
             (long long)g.n, (long long)kNoAllocMaxN);
  RF_REQUIRE(std::isfinite(g.fs) && g.fs > 0, "fs must be positive");
  RF_REQUIRE(std::isfinite(g.f_low) && std::isfinite(g.f_high) && g.f_low > 0 && g.f_low < g.f_high,
             "need 0 < f_low < f_high");
  RF_REQUIRE(g.f_high + g.df_high <= 0.5 * g.fs * (1 + 1e-12) && g.df_high >= 0,
             "f_high + df_high must not exceed fs/2");
  RF_REQUIRE(g.pn_order >= 0 && g.pn_order <= 7, "pn_order must be 0..7");
  RF_REQUIRE(g.dtype == RF_F64 || g.dtype == RF_F32, "dtype must be RF_F64 or RF_F32");
  RF_REQUIRE(std::isfinite(ref.m1) && std::isfinite(ref.m2) && ref.m1 > 0 && ref.m2 > 0 && std::isfinite(ref.tc) &&
                 std::isfinite(ref.phic),
             "ref: masses must be positive and all fields finite");
  noalloc_check_dev(x, "x", false);
  noalloc_check_dev(inv_psd, "inv_psd", false);
  noalloc_check_dev(z_out, "z_out", false);
  noalloc_check_dev(sigma_out, "sigma_out", true);

  unsigned char* ws = noalloc_scratch_address();
  const int64_t n = g.n;
  const double df = g.fs / (double)n;
  void* tw = ws;
  void* xf = ws + kNoAllocSlot;
  void* fa = ws + 2 * kNoAllocSlot;
  void* fb = ws + 3 * kNoAllocSlot;
  double* part = reinterpret_cast<double*>(ws + 4 * kNoAllocSlot);
  double* sig2 = part + kRedBlocks;
  static_assert((kRedBlocks + 1) * sizeof(double) <= kNoAllocRed, "reduction slots");
  // Every region is fully rewritten below before it is read (twiddles, spectra, partial
  // sums), so nothing left by an earlier call leaks into this one.
  const unsigned grid = (unsigned)((n + 255) / 256);
  k_sigma2_partial<<<kRedBlocks, kRedThreads, 0, s>>>(inv_psd, n / 2 + 1, df, g.f_low, g.f_high, part);
  RF_LAUNCHED();
  k_sum_partials<<<1, kRedThreads, 0, s>>>(part, kRedBlocks, sig2);
  RF_LAUNCHED();
  const Tf2 p = make_tf2(ref, g.pn_order);
  if (g.dtype == RF_F64) {
    k_noalloc_twiddles<double2><<<grid, 256, 0, s>>>(static_cast<double2*>(tw), n);
    RF_LAUNCHED();
    fft_r2c_f64(static_cast<const double*>(x), static_cast<double2*>(xf), static_cast<double2*>(fb), n,
                static_cast<double2*>(tw), n, s);
    k_mf_pointwise<double2><<<grid, 256, 0, s>>>(static_cast<double2*>(xf), inv_psd, sig2, p, n, df, g.f_low,
                                                 g.f_high, static_cast<double2*>(fa), sigma_out);
    RF_LAUNCHED();
    fft_c2c_f64(static_cast<double2*>(fa), static_cast<double2*>(z_out), static_cast<double2*>(fb), n, 1, +1,
                static_cast<double2*>(tw), n, s);
  } else {
    k_noalloc_twiddles<float2><<<grid, 256, 0, s>>>(static_cast<float2*>(tw), n);
    RF_LAUNCHED();
    fft_r2c_f32(static_cast<const float*>(x), static_cast<float2*>(xf), static_cast<float2*>(fb), n,
                static_cast<float2*>(tw), n, s);
    k_mf_pointwise<float2><<<grid, 256, 0, s>>>(static_cast<float2*>(xf), inv_psd, sig2, p, n, df, g.f_low,
                                                g.f_high, static_cast<float2*>(fa), sigma_out);
    RF_LAUNCHED();
    fft_c2c_f32(static_cast<float2*>(fa), static_cast<float2*>(z_out), static_cast<float2*>(fb), n, 1, +1,
                static_cast<float2*>(tw), n, s);
  }
}

}  // namespace
}  // namespace rf

extern "C" rf_status rf_mf_reference_noalloc(const rf_grid* grid, const void* x, const double* inv_psd,
                                             const rf_template* ref, void* z_out, double* sigma_out,
                                             rf_stream stream) {
  rf::clear_error();
  try {
    RF_REQUIRE(grid != nullptr && ref != nullptr, "grid and ref must be non-NULL");
    rf::mf_reference_noalloc_impl(*grid, x, inv_psd, *ref, z_out, sigma_out, (cudaStream_t)stream);
    return RF_OK;
  } catch (const rf::Fail& e) {
    return e.st;
  } catch (...) {
    rf::set_error("unexpected internal error");
    return RF_EINVAL;
  }
}
