// Float-float arithmetic (an unevaluated sum h + l of two FP32 numbers, about
// 48 significant bits) and the WENO5-Z interpolation on it.
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

// |a| >= |b| assumed: the sum and its rounding error
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

// ---------------------------------------------------------------------------
// WENO5-Z (exponent 1) of one side, as a correction to its leading candidate.
// B: 4 x the smoothness indicators + 4 eps, X0 = C_0 - C_1, X2 = C_2 - C_1.
// Returns sum_k a_k (C_k - C_r) / (6 sum_k a_k); r: the candidate of the largest weight.
MPMC_FF ff weno5z_corr(ff B0, ff B1, ff B2, ff X0, ff X2, int& r) {
  // a_k = d_k (1 + tau / B_k), d = 1, 6, 3, all times 2^-20 so that tau / B_k
  // stays in range down to B_k = 2^-122
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

// 4 eps of WENO5-Z for weno5z_lr_ff: mantissa in [1, 2) and exponent
struct WenoEps {
  float h, l;
  int e;
};

// Both sides of a face from the six cells w[0..5]: L of w[0..4], R of
// w[5..1].  False (nothing written) where a difference of the stencil is
// not finite or beyond 2^900: the caller takes the FP64 form.
MPMC_FF bool weno5z_lr_ff(const double* w, const WenoEps eps, double& L, double& R) {
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
  // second differences t, their (13/3) t^2 (4 beta = (13/3) t^2 + s^2), the
  // third differences f
  const ff t0 = ff_sub(D1, D0), t1 = ff_sub(D2, D1), t2 = ff_sub(D3, D2), t3 = ff_sub(D4, D3);
  const ff K = {4.3333335f, -1.5894572e-07f};
  const ff q0 = ff_addp(ff_mul(K, ff_sqr(t0)), ep), q1 = ff_addp(ff_mul(K, ff_sqr(t1)), ep),
           q2 = ff_addp(ff_mul(K, ff_sqr(t2)), ep), q3 = ff_addp(ff_mul(K, ff_sqr(t3)), ep);
  const ff f0 = ff_sub(t1, t0), f1 = ff_sub(t2, t1), f2 = ff_sub(t3, t2);
  const ff D1d = {D1.h + D1.h, D1.l + D1.l}, D2d = {D2.h + D2.h, D2.l + D2.l}, D3d = {D3.h + D3.h, D3.l + D3.l};
  int rl, rr;
  ff cl, cr;
  {
    // left: s = 3 d1 - d0, d1 + d2, d3 - 3 d2
    const ff B0 = ff_addp(q0, ff_sqr(ff_add(t0, D1d)));
    const ff B1 = ff_addp(q1, ff_sqr(ff_add(D1, D2)));
    const ff B2 = ff_addp(q2, ff_sqr(ff_sub(t2, D2d)));
    cl = weno5z_corr(B0, B1, B2, ff{-(f0.h + f0.h), -(f0.l + f0.l)}, ff{-f1.h, -f1.l}, rl);
  }
  {
    // right: s = d4 - 3 d3, d2 + d3, 3 d2 - d1
    const ff B0 = ff_addp(q3, ff_sqr(ff_sub(t3, D3d)));
    const ff B1 = ff_addp(q2, ff_sqr(ff_add(D2, D3)));
    const ff B2 = ff_addp(q1, ff_sqr(ff_add(t1, D2d)));
    cr = weno5z_corr(B0, B1, B2, ff{f2.h + f2.h, f2.l + f2.l}, f1, rr);
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
