// Float-float arithmetic (an unevaluated sum h + l of two FP32 numbers, about
// 48 significant bits) and the ENO-type interpolations on it (WENO5-Z, WENO5-JS,
// TENO5, TENO6).
//
// Why: one SM of GB300 retires two FP64 operations per clock and 128 FP32
// ones, so an FP64 instruction costs the time of 64 FP32 instructions, while
// a float-float addition takes 11 and a product 4 to 7 of them.  The nonlinear
// weights of WENO5-Z are most of the FP64 operations of a face, and they act
// only on differences of the stencil's values: in
//   L = w_2 + C_r / 6 + sum_k a_k (C_k - C_r) / (6 sum_k a_k)
// (C_k / 6 the three candidates as deviations from the cell's value, a_k the
// weights, r the candidate of the largest weight) everything that carries the
// value itself is FP64, and the last term, a correction that vanishes with
// the candidates' disagreement, is float-float.  Its error, 2^-47 of that
// correction, stays below the rounding that the all-FP64 form makes in its
// numerator (six terms of up to 18/6 of the value).
//
// Host-compilable (without contraction of a*b+c) so that a host test can
// compare it with the interpolation in extended precision.
#pragma once
#include <cstdint>
#include <cstring>

#include "mpmc_narrow.h"

#ifdef __CUDACC__
#define MPMC_FF __host__ __device__ __forceinline__
#else
#include <cmath>
#define MPMC_FF inline
#endif

namespace mpmc {

struct ff {
  float h, l;
};

// FP32 operations that the compiler may not contract or reorder
MPMC_FF float fadd(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
MPMC_FF float fmul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
MPMC_FF float ffma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fmaf(a, b, c);
#endif
}
// an FP32 reciprocal within about an ulp, for 2^-126 <= |a| <= 2^126
MPMC_FF float frcp(float a) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return __fmaf_rn(r, __fmaf_rn(-a, r, 1.f), r);
#else
  return 1.f / a;
#endif
}
MPMC_FF uint32_t fbits(float a) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(a);
#else
  uint32_t u;
  std::memcpy(&u, &a, 4);
  return u;
#endif
}
MPMC_FF float ffloat(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float a;
  std::memcpy(&a, &u, 4);
  return a;
#endif
}
MPMC_FF uint32_t dhi(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2hiint(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return (uint32_t)(b >> 32);
#endif
}
MPMC_FF uint32_t dlo(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2loint(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return (uint32_t)b;
#endif
}
MPMC_FF double dmake(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
MPMC_FF double dfma(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return __fma_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}
MPMC_FF int imax(int a, int b) { return a > b ? a : b; }
MPMC_FF int imin(int a, int b) { return a < b ? a : b; }

// |a| >= |b| assumed: the sum and its rounding error (Dekker)
MPMC_FF ff ff_fast(float a, float b) {
  const float s = fadd(a, b);
  return {s, fadd(b, -fadd(s, -a))};
}
// a + b exactly (Knuth)
MPMC_FF ff ff_two(float a, float b) {
  const float s = fadd(a, b), t = fadd(s, -a);
  return {s, fadd(fadd(a, -fadd(s, -t)), fadd(b, -t))};
}
// a + b, renormalized (after cancellation the low part may exceed the high one)
MPMC_FF ff ff_add(ff a, ff b) {
  const ff s = ff_two(a.h, b.h);
  return ff_fast(s.h, fadd(s.l, fadd(a.l, b.l)));
}
MPMC_FF ff ff_sub(ff a, ff b) { return ff_add(a, ff{-b.h, -b.l}); }
// a + b without renormalization, for terms of one sign
MPMC_FF ff ff_addp(ff a, ff b) {
  const ff s = ff_two(a.h, b.h);
  return {s.h, fadd(s.l, fadd(a.l, b.l))};
}
// a b, the low part left at up to 2^-22 of the high one
MPMC_FF ff ff_mul(ff a, ff b) {
  const float p = fmul(a.h, b.h);
  float e = ffma(a.h, b.h, -p);
  e = ffma(a.h, b.l, e);
  return {p, ffma(a.l, b.h, e)};
}
MPMC_FF ff ff_sqr(ff a) {
  const float p = fmul(a.h, a.h);
  return {p, ffma(fadd(a.h, a.h), a.l, ffma(a.h, a.h, -p))};
}
MPMC_FF ff ff_mulf(ff a, float c) {
  const float p = fmul(a.h, c);
  return {p, ffma(a.l, c, ffma(a.h, c, -p))};
}
// 1 / b: one Newton step in its second-order form from the FP32 reciprocal
MPMC_FF ff ff_rcp(ff b) {
  const float r = frcp(b.h);
  const float e = ffma(-b.l, r, ffma(-b.h, r, 1.f));
  return {r, fmul(r, ffma(e, e, e))};
}
// 2^k, -126 <= k <= 127
MPMC_FF float fpow2(int k) { return ffloat((uint32_t)(k + 127) << 23); }

// x 2^-(E - 1023) as float-float from the bits, on the integer pipes (a
// hardware conversion issues on the FP64 pipe).  E: an exponent field no
// smaller than x's.  Values below 2^-126 after scaling become zero.
MPMC_FF ff ff_scaled(double x, int E) {
  const uint32_t H = dhi(x), L = dlo(x);
  const int e = (int)((H >> 20) & 0x7ffu) - E + 127;
  // the 23 leading fraction bits of x under the new exponent, rounded up
  // where the next bit is set (a carry into the exponent is the next binade)
  const uint32_t m = ((H << 3) | (L >> 29)) & 0x007fffffu, s = H & 0x80000000u;
  const uint32_t hb = e >= 1 ? (s | (((uint32_t)e << 23) + m + ((L >> 28) & 1u)) ) : s;
  // what is left of the 29 low bits, signed, at 2^(e - 127 - 52)
  const float sc = ffloat(s | ((uint32_t)imax(e - 52, 0) << 23));
  const int low = (int)(L << 3) >> 3;
#ifdef __CUDA_ARCH__
  const float lf = __int2float_rn(low);
#else
  const float lf = (float)low;
#endif
  return {ffloat(hb), fmul(lf, sc)};
}

// the FP32 number f times 2^(E - 1023) as FP64, from the bits; f normal or
// zero, and the result normal (subnormal f gives zero)
MPMC_FF double ff_widen(float f, int E) {
  const uint32_t b = fbits(f), e = (b >> 23) & 0xffu;
  const uint32_t hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((uint32_t)(E - 127) << 20));
  return e ? dmake(hi, b << 29) : 0.0;
}

// sum_d (a_d - b_d) of FP32 numbers to FP64 rounding: the differences are exact
// as pairs, their high parts are summed exactly, and what that leaves is summed
// as a pair (within 2^-64 of the differences' magnitudes).  One rounding of the
// sum follows, where FP64 differences and sums take 2 D - 1.
// ok: false where a part leaves FP32's normal range; the caller takes FP64.
template <int D>
MPMC_FF double ff_diff_sum(const float* a, const float* b, bool& ok) {
  ff s = ff_two(a[0], -b[0]);
  if (D == 1) {
    ok = ok && widens(s.h) && widens(s.l);
    return widen(s.h) + widen(s.l);
  }
  ff r = {s.l, 0.f};
#pragma unroll
  for (int d = 1; d < D; ++d) {
    const ff t = ff_two(a[d], -b[d]);
    s = ff_two(s.h, t.h);
    ff q = ff_two(r.h, s.l);
    r = ff{q.h, fadd(r.l, q.l)};
    q = ff_two(r.h, t.l);
    r = ff{q.h, fadd(r.l, q.l)};
  }
  ok = ok && widens(s.h) && widens(r.h) && widens(r.l);
  return widen(s.h) + (widen(r.h) + widen(r.l));
}

// ---------------------------------------------------------------------------
// The interpolations of one side, as a correction to a leading candidate.
// B: 4 x the indicators + 4 eps of the left, central and right three-cell
// stencils, X0 = C_0 - C_1, X2 = C_2 - C_1.

// sum_k a_k (C_k - C_r) / (6 sum_k a_k); r: the candidate of the largest weight
MPMC_FF ff eno_corr(ff a0, ff a1, ff a2, ff X0, ff X2, int& r) {
  const ff s01 = ff_addp(a0, a1), s12 = ff_addp(a1, a2), S = ff_addp(s01, a2);
  const bool lead0 = a0.h > a1.h && a0.h > a2.h, lead2 = a2.h > a1.h && !lead0;
  r = lead0 ? 0 : (lead2 ? 2 : 1);
  // r = 1: a_0 X0 + a_2 X2;  r = 0: a_2 X2 - (a_1 + a_2) X0;
  // r = 2: a_0 X0 - (a_0 + a_1) X2
  const ff p = {lead0 ? -s12.h : a0.h, lead0 ? -s12.l : a0.l};
  const ff q = {lead2 ? -s01.h : a2.h, lead2 ? -s01.l : a2.l};
  const ff N = ff_add(ff_mul(p, X0), ff_mul(q, X2));
  return ff_mul(N, ff_rcp(ff_mulf(S, 6.f)));
}

// WENO5-Z: a_k = d_k (1 + tau / B_k), d = 1, 6, 3, all times 2^-20 so that
// tau / B_k stays in range down to B_k = 2^-122
MPMC_FF ff weno5z_corr(ff B0, ff B1, ff B2, ff X0, ff X2, int& r) {
  constexpr float U = 1.f / 1048576.f;
  ff tau = ff_sub(B0, B2);
  const float sg = tau.h < 0.f ? -U : U;
  tau.h = fmul(tau.h, sg);
  tau.l = fmul(tau.l, sg);
  const ff r0 = ff_mul(tau, ff_rcp(B0));
  const ff r1 = ff_mul(ff_mulf(tau, 6.f), ff_rcp(B1));
  const ff r2 = ff_mul(ff_mulf(tau, 3.f), ff_rcp(B2));
  ff a0 = ff_two(U, r0.h), a1 = ff_two(6.f * U, r1.h), a2 = ff_two(3.f * U, r2.h);
  a0.l = fadd(a0.l, r0.l);
  a1.l = fadd(a1.l, r1.l);
  a2.l = fadd(a2.l, r2.l);
  return eno_corr(a0, a1, a2, X0, X2, r);
}

// WENO5-JS: a_k = d_k / B_k^2, taken relative to the smallest B
MPMC_FF ff weno5js_corr(ff B0, ff B1, ff B2, ff X0, ff X2, int& r) {
  const float m01 = B0.h < B1.h ? B0.h : B1.h, m = m01 < B2.h ? m01 : B2.h;
  const ff a0 = ff_sqr(ff_mulf(ff_rcp(B0), m));
  const ff a1 = ff_mulf(ff_sqr(ff_mulf(ff_rcp(B1), m)), 6.f);
  const ff a2 = ff_mulf(ff_sqr(ff_mulf(ff_rcp(B2), m)), 3.f);
  return eno_corr(a0, a1, a2, X0, X2, r);
}

// TENO: the kept candidates (bit k clear where r_k^6 < CT sum r^6,
// r_k = 1 + tau / B_k).  First in FP32 with a margin far above its rounding
// (r_k is exact to ~1e-6: tau's cancellation is done in float-float), in
// float-float where a candidate is that close to the cut.
template <int K>
MPMC_FF unsigned teno_mask(const ff* B, ff tau, float CT) {
  if (tau.h < 0.f) tau = ff{-tau.h, -tau.l};
  constexpr float U = 1.f / 1048576.f;   // r_k 2^-20, as in weno5z_corr
  float r[K], m = 0.f, g[K], gs = 0.f;
  for (int k = 0; k < K; ++k) {
    r[k] = U + fmul(tau.h, U) * frcp(B[k].h);
    m = r[k] > m ? r[k] : m;
  }
  const float im = frcp(m);
  for (int k = 0; k < K; ++k) {
    const float x = r[k] * im, x2 = x * x;
    g[k] = x2 * x2 * x2;
    gs += g[k];
  }
  unsigned kept = 0u;
  bool close = false;
  for (int k = 0; k < K; ++k) {
    const float c = CT * gs;
    if (!(g[k] < c)) kept |= 1u << k;
    close = close || (g[k] < 1.001f * c && g[k] > 0.999f * c);
  }
  if (close) {
    ff rk[K], q[K], qs = {0.f, 0.f};
    for (int k = 0; k < K; ++k) {
      const ff t = ff_mul(ff{fmul(tau.h, U), fmul(tau.l, U)}, ff_rcp(B[k]));
      const ff u = ff_two(U, t.h);
      rk[k] = ff{u.h, fadd(u.l, t.l)};
    }
    for (int k = 0; k < K; ++k) {
      const ff x = ff_mulf(rk[k], im), x2 = ff_sqr(x);
      q[k] = ff_mul(ff_sqr(x2), x2);
      qs = ff_addp(qs, q[k]);
    }
    kept = 0u;
    // (CT as float-float: 1e-5 and 1e-7)
    const ff c = ff_mul(qs, CT == 1e-5f ? ff{1.e-05f, 2.5262125e-13f} : ff{1.e-07f, -1.1686097e-15f});
    for (int k = 0; k < K; ++k)
      if (!(ff_sub(q[k], c).h < 0.f)) kept |= 1u << k;
  }
  return kept;
}

// TENO6's selection for one side: the four-cell candidate's indicator b4 and
// tau = |b6 - (b_l + b_r + 4 b_c) / 6| (all times 4) as squares of zero-sum
// combinations of the differences (mpmc_device.cuh's teno6_kept on d_j)
MPMC_FF unsigned teno6_mask(ff d0, ff d1, ff d2, ff d3, ff d4, ff B0, ff B1, ff B2, ff ep) {
  // b4 = s^2 / 36 + (13/12) t^2 + (781/720) u^2
  const ff s = ff_add(ff_add(ff_mulf(d2, 11.f), ff_mulf(d3, -7.f)), ff_add(d4, d4));
  const ff t = ff_add(ff_add(ff_mulf(d2, -2.f), ff_mulf(d3, 3.f)), ff{-d4.h, -d4.l});
  const ff u = ff_add(ff_sub(d2, ff_add(d3, d3)), d4);
  const ff K = ff{4.3333335e+00f, -1.5894572e-07f}, K9 = ff{1.1111111e-01f, -8.278423e-10f}, KU = ff{4.338889e+00f, -2.3312039e-07f};
  const ff b4 = ff_addp(ff_addp(ff_mul(K9, ff_sqr(s)), ff_mul(K, ff_sqr(t))), ff_addp(ff_mul(KU, ff_sqr(u)), ep));
  // b6 from its five combinations
  const ff c1 = ff_add(ff_add(ff_add(ff_mulf(d0, -3.f), ff_mulf(d1, 27.f)), ff_add(ff_mulf(d2, 47.f), ff_mulf(d3, -13.f))),
                       ff_add(d4, d4));
  const ff c2 = ff_add(ff_mulf(ff_sub(d0, d3), 11.f), ff_mulf(ff_sub(d2, d1), 163.f));
  const ff c3 = ff_add(ff_add(ff_add(ff_mulf(d0, 16315.f), ff_mulf(d1, 33146.f)),
                              ff_add(ff_mulf(d2, -131724.f), ff_mulf(d3, 98750.f))),
                       ff_mulf(d4, -16487.f));
  const ff c4 = ff_add(ff_sub(d3, d0), ff_mulf(ff_sub(d1, d2), 3.f));
  const ff c5 = ff_add(ff_add(ff_add(d0, d4), ff_mulf(ff_add(d1, d3), -4.f)), ff_mulf(d2, 6.f));
  const ff G1 = ff{1.1111111e-03f, -2.6904874e-11f}, G2 = ff{2.5641025e-04f, 9.462476e-12f}, G3 = ff{1.0081331e-09f, 1.6934418e-18f}, G4 = ff{4.339014e+00f, -1.1830685e-08f}, G5 = ff{4.339017e+00f, 1.0037913e-07f};
  ff b6 = ff_addp(ff_mul(G1, ff_sqr(c1)), ff_mul(G2, ff_sqr(c2)));
  b6 = ff_addp(b6, ff_addp(ff_mul(G3, ff_sqr(c3)), ff_mul(G4, ff_sqr(c4))));
  b6 = ff_addp(b6, ff_mul(G5, ff_sqr(c5)));
  // (B_l + B_r + 4 B_c) / 6 carries one 4 eps
  const ff sx = ff{1.6666667e-01f, -4.967054e-09f};
  const ff m = ff_mul(ff_addp(ff_addp(B0, B2), ff_mulf(B1, 4.f)), sx);
  const ff tau = ff_sub(ff_addp(b6, ep), m);
  const ff b[4] = {B0, B1, B2, b4};
  return teno_mask<4>(b, tau, 1e-7f);
}

// 4 eps of an interpolation: mantissa in [1, 2) and exponent
struct WenoEps {
  float h, l;
  int e;
};
// the fixed epsilons of TENO (1e-40) and WENO5-JS (1e-6), times 4
MPMC_FF WenoEps teno_eps4(int e) { return WenoEps{1.0889035e+00f, 2.7813691e-08f, e - 131}; }
MPMC_FF WenoEps js_eps4(int e) { return WenoEps{1.048576e+00f, 2.6473999e-09f, e - 18}; }

// value from the kept TENO candidates, with their optimal weights
// renormalized: sum_k w_k C_k / (6 sum_k w_k) on the differences
// d0 .. d4 (d4: TENO6's fourth candidate, (9 d2 - 4 d3 + d4) / 2)
template <int KIND>
MPMC_FF double teno_value(unsigned kept, double d0, double d1, double d2, double d3, double d4) {
  const bool k0 = kept & 1u, k1 = kept & 2u, k2 = kept & 4u, k3 = kept & 8u;
  // weights in twentieths: TENO5 (2, 12, 6), TENO6 (1, 9, 6, 4); every
  // coefficient below is a small integer, the one rounding is the quotient's
  const float w0 = k0 ? (KIND == 3 ? 1.f : 2.f) : 0.f, w1 = k1 ? (KIND == 3 ? 9.f : 12.f) : 0.f, w2 = k2 ? 6.f : 0.f,
              w3 = KIND == 3 && k3 ? 4.f : 0.f;
  const float W = 12.f * (w0 + w1 + w2 + w3);
  const float a0 = -4.f * w0, a1 = 10.f * w0 + 2.f * w1, a2 = 4.f * w1 + 8.f * w2 + 9.f * w3, a3 = -2.f * w2 - 4.f * w3;
  double s = ff_widen(a1, 1023) * d1;
  s = dfma(ff_widen(a0, 1023), d0, s);
  s = dfma(ff_widen(a3, 1023), d3, s);
  if (KIND == 3) s = dfma(ff_widen(w3, 1023), d4, s);
  s = dfma(ff_widen(a2, 1023), d2, s);
  // 1 / W to FP64 rounding, W = 12 .. 240
  const double Wd = ff_widen(W, 1023), r0 = ff_widen(frcp(W), 1023);
  double e = dfma(-Wd, r0, 1.0);
  e = dfma(e, e, e);
  return s * dfma(r0, e, r0);
}

// Both sides of a face from the six cells w[0..5]: L of w[0..4] (TENO6:
// w[0..5]), R of w[5..1] (w[5..0]).  KIND: 0 WENO5-Z, 1 WENO5-JS, 2 TENO5,
// 3 TENO6.  eps: 4 eps of that interpolation.  False (nothing written) where
// a difference of the stencil is not finite or beyond 2^900: the caller takes
// the FP64 form.
template <int KIND>
MPMC_FF bool eno_lr_ff(const double* w, const WenoEps eps, double& L, double& R) {
  const double d0 = w[1] - w[0], d1 = w[2] - w[1], d2 = w[3] - w[2], d3 = w[4] - w[3], d4 = w[5] - w[4];
  const uint32_t A = 0x7fffffffu;
  const int e0 = (int)(dhi(d0) & A), e1 = (int)(dhi(d1) & A), e2 = (int)(dhi(d2) & A), e3 = (int)(dhi(d3) & A),
            e4 = (int)(dhi(d4) & A);
  int E = imax(imax(imax(e0, e1), imax(e2, e3)), e4) >> 20;
  if (E > 1923) return false;
  E = imax(E, 400);   // differences below 2^-622 count as 2^-622 ones: no correction
  const ff D0 = ff_scaled(d0, E), D1 = ff_scaled(d1, E), D2 = ff_scaled(d2, E), D3 = ff_scaled(d3, E),
           D4 = ff_scaled(d4, E);
  // 4 eps at the differences' scale, at least 2^-122
  const int ke = eps.e - 2 * (E - 1023);
  const float es = fpow2(imax(imin(ke, 100), -122));
  const ff ep = {fmul(eps.h, es), fmul(eps.l, es)};
  // second differences t, their (13/3) t^2 (4 beta = (13/3) t^2 + s^2)
  const ff t0 = ff_sub(D1, D0), t1 = ff_sub(D2, D1), t2 = ff_sub(D3, D2), t3 = ff_sub(D4, D3);
  const ff K = ff{4.3333335e+00f, -1.5894572e-07f};
  const ff q0 = ff_addp(ff_mul(K, ff_sqr(t0)), ep), q1 = ff_addp(ff_mul(K, ff_sqr(t1)), ep),
           q2 = ff_addp(ff_mul(K, ff_sqr(t2)), ep), q3 = ff_addp(ff_mul(K, ff_sqr(t3)), ep);
  const ff D1d = {D1.h + D1.h, D1.l + D1.l}, D2d = {D2.h + D2.h, D2.l + D2.l}, D3d = {D3.h + D3.h, D3.l + D3.l};
  // left: s = 3 d1 - d0, d1 + d2, d3 - 3 d2; right: d4 - 3 d3, d2 + d3, 3 d2 - d1
  const ff BL0 = ff_addp(q0, ff_sqr(ff_add(t0, D1d))), BL1 = ff_addp(q1, ff_sqr(ff_add(D1, D2))),
           BL2 = ff_addp(q2, ff_sqr(ff_sub(t2, D2d)));
  const ff BR0 = ff_addp(q3, ff_sqr(ff_sub(t3, D3d))), BR1 = ff_addp(q2, ff_sqr(ff_add(D2, D3))),
           BR2 = ff_addp(q1, ff_sqr(ff_add(t1, D2d)));
  if (KIND >= 2) {
    unsigned kl, kr;
    if (KIND == 2) {
      const ff bl[3] = {BL0, BL1, BL2}, br[3] = {BR0, BR1, BR2};
      kl = teno_mask<3>(bl, ff_sub(BL0, BL2), 1e-5f);
      kr = teno_mask<3>(br, ff_sub(BR0, BR2), 1e-5f);
    } else {
      kl = teno6_mask(D0, D1, D2, D3, D4, BL0, BL1, BL2, ep);
      kr = teno6_mask(ff{-D4.h, -D4.l}, ff{-D3.h, -D3.l}, ff{-D2.h, -D2.l}, ff{-D1.h, -D1.l}, ff{-D0.h, -D0.l}, BR0,
                      BR1, BR2, ep);
    }
    L = w[2] + teno_value<KIND>(kl, d0, d1, d2, d3, d4);
    R = w[3] - teno_value<KIND>(kr, d4, d3, d2, d1, d0);
    return true;
  }
  const ff f0 = ff_sub(t1, t0), f1 = ff_sub(t2, t1), f2 = ff_sub(t3, t2);
  int rl, rr;
  ff cl, cr;
  const ff XL0 = {-(f0.h + f0.h), -(f0.l + f0.l)}, XL2 = {-f1.h, -f1.l}, XR0 = {f2.h + f2.h, f2.l + f2.l};
  if (KIND == 0) {
    cl = weno5z_corr(BL0, BL1, BL2, XL0, XL2, rl);
    cr = weno5z_corr(BR0, BR1, BR2, XR0, f1, rr);
  } else {
    cl = weno5js_corr(BL0, BL1, BL2, XL0, XL2, rl);
    cr = weno5js_corr(BR0, BR1, BR2, XR0, f1, rr);
  }
  // C_r / 6 in FP64: left (5 d1 - 2 d0, d1 + 2 d2, 4 d2 - d3), right
  // -(5 d3 - 2 d4, d3 + 2 d2, 4 d2 - d1)
  const double c5 = 5.0 / 6.0, c4 = 4.0 / 6.0, c2 = 2.0 / 6.0, c1 = 1.0 / 6.0;
  {
    const double x = rl == 2 ? d2 : d1, p = rl == 0 ? c5 : (rl == 1 ? c1 : c4);
    const double y = rl == 0 ? d0 : (rl == 1 ? d2 : d3), q = rl == 0 ? -c2 : (rl == 1 ? c2 : -c1);
    L = w[2] + dfma(p, x, dfma(q, y, ff_widen(cl.h, E) + ff_widen(cl.l, E)));
  }
  {
    const double x = rr == 2 ? d2 : d3, p = rr == 0 ? -c5 : (rr == 1 ? -c1 : -c4);
    const double y = rr == 0 ? d4 : (rr == 1 ? d2 : d1), q = rr == 0 ? c2 : (rr == 1 ? -c2 : c1);
    R = w[3] + dfma(p, x, dfma(q, y, ff_widen(cr.h, E) + ff_widen(cr.l, E)));
  }
  return true;
}

}  // namespace mpmc
