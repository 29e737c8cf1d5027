// Complex numbers in pairs of FP32 values (value = h + l, about 46 bits), for the FP64 transforms whose
// results are rounded to FP32.
//
// The FP64 pipe has two lanes per SM, the FP32 pipes 128: a pair addition is eight FP32 operations
// (the exact error of h + h by Knuth's two-sum, the low parts added to it), a product four plus the
// sum, each done for the real and the imaginary part at once by the paired FP32 instructions, and is
// five to seven times faster than its FP64 counterpart.  The pairs are not renormalised: l collects
// the rounding errors of h, and the neglected terms are of the order of 2^-46 of the operands.  Both
// are relative to the operands: where a sum cancels, l can be as large as h.  Divisions of labour: the phase of a template stays FP64; sums of the transform and
// products with roots of unity are pairs; magnitudes that decide a threshold are formed in FP64 from
// h + l.
#pragma once

#include "cplx.cuh"

namespace rf {

struct __align__(16) cdf {
  float2 h, l;
};

// Paired FP32 operations, rounded to nearest and never contracted.
__device__ __forceinline__ float2 pmul(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ float2 pneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 pdup(float a) { return make_float2(a, a); }

// s + e = a + b exactly
__device__ __forceinline__ float2 two_sum(float2 a, float2 b, float2& e) {
  const float2 s = cadd(a, b);
  const float2 bb = csub(s, a);
  e = cadd(csub(a, csub(s, bb)), csub(b, bb));
  return s;
}

__device__ __forceinline__ cdf cadd(cdf a, cdf b) {
  cdf r;
  float2 e;
  r.h = two_sum(a.h, b.h, e);
  r.l = cadd(e, cadd(a.l, b.l));
  return r;
}
__device__ __forceinline__ cdf csub(cdf a, cdf b) {
  cdf r;
  float2 e;
  r.h = two_sum(a.h, pneg(b.h), e);
  r.l = cadd(e, csub(a.l, b.l));
  return r;
}
// SIGN i a
template <int SIGN>
__device__ __forceinline__ cdf cturn(cdf a) {
  return cdf{make_float2(-SIGN * a.h.y, SIGN * a.h.x), make_float2(-SIGN * a.l.y, SIGN * a.l.x)};
}
__device__ __forceinline__ cdf cmul(cdf a, cdf w) {
  const float2 rh = pdup(w.h.x), rl = pdup(w.l.x), ih = pdup(w.h.y), il = pdup(w.l.y);
  const cdf t = cturn<1>(a);
  const float2 p = pmul(a.h, rh), q = pmul(t.h, ih);
  float2 ep = pfma(a.h, rh, pneg(p)), eq = pfma(t.h, ih, pneg(q));
  ep = pfma(a.h, rl, pfma(a.l, rh, ep));
  eq = pfma(t.h, il, pfma(t.l, ih, eq));
  cdf r;
  float2 e;
  r.h = two_sum(p, q, e);
  r.l = cadd(e, cadd(ep, eq));
  return r;
}
__device__ __forceinline__ cdf cconj_pair(cdf a) {
  return cdf{make_float2(a.h.x, -a.h.y), make_float2(a.l.x, -a.l.y)};
}

// a exp(+2 pi i Q / 16): constants as pairs of the correctly rounded cos and sin of k pi / 8
template <int Q>
__device__ __forceinline__ cdf crot16(cdf a) {
  constexpr int q = Q & 15;
  if constexpr (q == 0) return a;
  else if constexpr (q == 4) return cturn<1>(a);
  else if constexpr (q == 8) return cdf{pneg(a.h), pneg(a.l)};
  else if constexpr (q == 12) return cturn<-1>(a);
  else {
    constexpr double C1 = 0.92387953251128675613, S1 = 0.38268343236508977173, R = 0.70710678118654752440;
    constexpr double cs[16] = {1, C1, R, S1, 0, -S1, -R, -C1, -1, -C1, -R, -S1, 0, S1, R, C1};
    constexpr double sn[16] = {0, S1, R, C1, 1, C1, R, S1, 0, -S1, -R, -C1, -1, -C1, -R, -S1};
    constexpr float ch = (float)cs[q], sh = (float)sn[q];
    constexpr float cl = (float)(cs[q] - (double)ch), sl = (float)(sn[q] - (double)sh);
    return cmul(a, cdf{make_float2(ch, sh), make_float2(cl, sl)});
  }
}

// Inverse (sign +1) DFTs in natural order, as dft<> of cplx.cuh.
__device__ __forceinline__ void cdf_dft4(cdf& a0, cdf& a1, cdf& a2, cdf& a3) {
  const cdf t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), d = cturn<1>(csub(a1, a3));
  a0 = cadd(t0, t2);
  a2 = csub(t0, t2);
  a1 = cadd(t1, d);
  a3 = csub(t1, d);
}

// R = R1 R2, n = n1 + R1 n2, k = k2 + R2 k1 (R2 = R / 4 inner, radix 4 outer for 16; 2 x 4 for 8)
template <int R>
__device__ __forceinline__ void cdf_dft(cdf* a) {
  if constexpr (R == 2) {
    const cdf t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
  } else if constexpr (R == 4) {
    cdf_dft4(a[0], a[1], a[2], a[3]);
  } else if constexpr (R == 8) {
    static_for<0, 2>([&](auto n1c) {
      constexpr int n1 = decltype(n1c)::value;
      cdf_dft4(a[n1], a[n1 + 2], a[n1 + 4], a[n1 + 6]);
    });
    // bin k2 of column n1 sits at a[n1 + 2 k2]
    static_for<1, 4>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      a[1 + 2 * k] = crot16<2 * k>(a[1 + 2 * k]);
    });
    cdf b[8];
    static_for<0, 4>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      b[k] = cadd(a[2 * k], a[2 * k + 1]);
      b[k + 4] = csub(a[2 * k], a[2 * k + 1]);
    });
#pragma unroll
    for (int t = 0; t < 8; ++t) a[t] = b[t];
  } else {
    static_assert(R == 16, "radix");
    static_for<0, 4>([&](auto n1c) {
      constexpr int n1 = decltype(n1c)::value;
      cdf_dft4(a[n1], a[n1 + 4], a[n1 + 8], a[n1 + 12]);
    });
    // bin k2 of column n1 sits at a[n1 + 4 k2]; the outer transforms run over n1
    static_for<0, 4>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      static_for<1, 4>([&](auto n1c) {
        constexpr int n1 = decltype(n1c)::value;
        a[n1 + 4 * k] = crot16<n1 * k>(a[n1 + 4 * k]);
      });
      cdf_dft4(a[4 * k], a[4 * k + 1], a[4 * k + 2], a[4 * k + 3]);
    });
    // bin k2 + 4 k1 sits at a[k1 + 4 k2]
    static_for<0, 4>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      static_for<k + 1, 4>([&](auto mc) {
        constexpr int m = decltype(mc)::value;
        const cdf t = a[m + 4 * k];
        a[m + 4 * k] = a[k + 4 * m];
        a[k + 4 * m] = t;
      });
    });
  }
}

}  // namespace rf
