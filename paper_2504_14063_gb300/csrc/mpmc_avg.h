// The scalars of a face's characteristic matrices (Appendix A): c = rho a and
// X of the equilibrium state of the two cells' arithmetic average, in
// float-float arithmetic (mpmc_ff.h; the reason for it stands there).
//
// X and c shape the projection only: an error in them reaches the face values
// times the difference that the interpolations of two fields leave, which is
// small against the field (zero where it is smooth).  So float-float's 2^-46
// suffices if it is relative to the cells' jump, not to a stiff liquid's
// energies (~ gamma Pinf): the average's p and T are solved as increments
// x = p - P_i, y = T - T_i on the two cells' own states.  With partial
// densities m_ki, m_kj, r_k = 1 / (p + Pinf_k), G_ki = T_i / (P_i + Pinf_k):
//   volume  sum_k R_k r_k B_k = 0,   B_k = M_k y - g_k x - h_k,
//   M_k = m_ki + m_kj,  g_k = m_ki G_ki + m_kj G_kj,
//   h_k = m_kj (dT - G_kj dP),  dP = P_j - P_i, dT = T_j - T_i;
//   energy  (sum cp_k M_k) y - (sum R_k g_k) x
//             = dT sum cv_k m_kj + sum R_k h_k + |du|^2 rho_i rho_j / (2 (rho_i + rho_j)),
// the second linear (the kinetic energy that the average loses appears as
// heat), so that y follows from x and the first is a rational function of x:
// Newton steps, first in FP32, then two or three in float-float.  At its root
//   X = T s_1 / sum cp_k M_k,  c^2 = (sum cp_k M_k) (sum M_k) / (T (s_2 sum cp_k M_k - s_1^2)),
//   s_q = sum R_k M_k r_k^q,
// which are Eq. SpeedOfSound and Appendix A's X with alpha and beta put in.
#pragma once
#include "mpmc_ff.h"

namespace mpmc {

// species constants as float-floats
struct SpeciesFF {
  ff R, cv, cp, pinf, q, b;
};

MPMC_FF ff ff_of(double x) { return ff_scaled(x, 1023); }
MPMC_FF double ff_double(ff a) { return ff_widen(a.h, 1023) + ff_widen(a.l, 1023); }
MPMC_FF float fabs_(float a) { return ffloat(fbits(a) & 0x7fffffffu); }
MPMC_FF float frsqrt_(float a) {
#ifdef __CUDA_ARCH__
  return rsqrtf(a);
#else
  return 1.f / std::sqrt(a);
#endif
}
// sqrt(a), a in the FP32 range
MPMC_FF ff ff_sqrt(ff a) {
  const float y = frsqrt_(a.h), s = fmul(a.h, y);
  const float e = fadd(ffma(-s, s, a.h), a.l);
  return ff_fast(s, fmul(e, fmul(0.5f, y)));
}

// X, c and 1 / c of the face between the cells i and j (mi, mj: partial
// densities; ui, uj: velocities as the face sees them).  False (nothing
// written) where the steps do not settle, where the jump's rounding would reach
// 2^-41 of c (strong jumps of a liquid with traces of gas, whose pressure is
// what they leave of it: FP64's own error is less there, elsewhere more or
// both are below it), or where a quantity leaves 2^-60..2^60: the caller takes
// the FP64 form.
template <int NS, int D>
MPMC_FF bool face_avg_ff(const SpeciesFF* sp, const double* mi, const double* mj, const double Pi, const double Pj,
                         const double Ti, const double Tj, const double* ui, const double* uj, double& X, double& c,
                         double& ic) {
  const uint32_t A = 0x7fffffffu, TOP = (1023u + 60u) << 20;
  uint32_t big = dhi(Pi) & A;
  big = big > (dhi(Pj) & A) ? big : (dhi(Pj) & A);
  big = big > (dhi(Ti) & A) ? big : (dhi(Ti) & A);
  big = big > (dhi(Tj) & A) ? big : (dhi(Tj) & A);
  const ff P0 = ff_of(Pi), P1 = ff_of(Pj), T0 = ff_of(Ti), T1 = ff_of(Tj);
  const ff dP = ff_of(Pj - Pi), dT = ff_of(Tj - Ti);
  ff al[NS], be[NS], M[NS];
  ff cpM = {0.f, 0.f}, gR = {0.f, 0.f}, c0 = {0.f, 0.f}, ri = {0.f, 0.f}, rj = {0.f, 0.f};
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const uint32_t hi = dhi(mi[k]) & A, hj = dhi(mj[k]) & A;
    big = big > hi ? big : hi;
    big = big > hj ? big : hj;
    const ff a = ff_of(mi[k]), b = ff_of(mj[k]);
    ri = ff_add(ri, a);
    rj = ff_add(rj, b);
    M[k] = ff_add(a, b);
    const ff Gi = ff_mul(T0, ff_rcp(ff_add(P0, sp[k].pinf))), Gj = ff_mul(T1, ff_rcp(ff_add(P1, sp[k].pinf)));
    // (an absent species: no term, whatever 1 / (P + Pinf) is)
    const bool on = M[k].h != 0.f;
    const ff g = ff_add(ff_mul(a, Gi), ff_mul(b, Gj)), h = ff_mul(b, ff_sub(dT, ff_mul(Gj, dP)));
    al[k] = on ? h : ff{0.f, 0.f};
    be[k] = on ? g : ff{0.f, 0.f};
    cpM = ff_add(cpM, ff_mul(sp[k].cp, M[k]));
    gR = ff_add(gR, ff_mul(sp[k].R, be[k]));
    c0 = ff_add(c0, ff_add(ff_mul(sp[k].cv, ff_mul(b, dT)), ff_mul(sp[k].R, al[k])));
  }
  if (big >= TOP) return false;
  ff u2 = {0.f, 0.f};
#pragma unroll
  for (int d = 0; d < D; ++d) u2 = ff_addp(u2, ff_sqr(ff_of(uj[d] - ui[d])));
  const ff Mt = ff_add(ri, rj);
  c0 = ff_add(c0, ff_mul(ff_mulf(u2, 0.5f), ff_mul(ff_mul(ri, rj), ff_rcp(Mt))));
  const ff inv = ff_rcp(cpM), y0 = ff_mul(c0, inv), y1 = ff_mul(gR, inv);
  float am[NS], bm[NS];   // magnitudes of al's and be's terms
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    am[k] = fabs_(sp[k].R.h) * (fabs_(M[k].h * y0.h) + fabs_(al[k].h));
    bm[k] = fabs_(sp[k].R.h) * (fabs_(M[k].h * y1.h) + fabs_(be[k].h));
    al[k] = ff_mul(sp[k].R, ff_sub(ff_mul(M[k], y0), al[k]));
    be[k] = ff_mul(sp[k].R, ff_sub(ff_mul(M[k], y1), be[k]));
  }
  // Newton from the mean pressure, in FP32
  float x = 0.5f * dP.h, pm = 3e38f;   // pm: the distance to the nearest pole
  for (int it = 0; it < 8; ++it) {
    float V = 0.f, dV = 0.f;
    pm = 3e38f;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const float q = (P0.h + x) + sp[k].pinf.h;
      const bool on = M[k].h != 0.f;
      const float r = on ? frcp(q) : 0.f, B = al[k].h + be[k].h * x;
      if (M[k].h > 0.f) pm = q < pm ? q : pm;
      V += B * r;
      dV += r * (be[k].h - r * B);
    }
    const float dx = -V * frcp(dV);
    x += dx;
    if (!(fabs_(dx) > 1.5e-5f * pm)) break;
  }
  // two steps with a float-float residual (derivative and step in FP32), a third
  // where the second was not yet small (trace gas in a liquid across a jump,
  // whose FP32 root is off by parts in a thousand), and the sums at the root
  ff xx = {x, 0.f}, s1, s2;
  float dx = 0.f, dV = 0.f;
  for (int it = 0; it < 3; ++it) {
    ff V = {0.f, 0.f};
    dV = 0.f;
    const ff p = ff_add(P0, xx);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const ff q = ff_add(p, sp[k].pinf);
      const bool on = M[k].h != 0.f;
      const ff r = on ? ff_rcp(q) : ff{0.f, 0.f};
      const ff B = ff_add(al[k], ff_mul(be[k], xx));
      V = ff_add(V, ff_mul(B, r));
      dV += r.h * (be[k].h - r.h * B.h);
    }
    dx = -V.h * frcp(dV);
    xx = ff_add(xx, ff{dx, 0.f});
    if (it > 0 && !(fabs_(dx) > 1e-10f * pm)) break;
  }
  pm = 3e38f;
  const ff p = ff_add(P0, xx), T = ff_add(T0, ff_add(y0, ff_mul(y1, xx)));
  s1 = {0.f, 0.f};
  s2 = {0.f, 0.f};
  float s3 = 0.f, mV = 0.f;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const ff q = ff_add(p, sp[k].pinf);
    if (M[k].h > 0.f) pm = q.h < pm ? q.h : pm;
    const ff r = M[k].h != 0.f ? ff_rcp(q) : ff{0.f, 0.f};
    const ff t = ff_mul(ff_mul(sp[k].R, M[k]), r);
    s1 = ff_add(s1, t);
    const ff tr = ff_mul(t, r);
    s2 = ff_add(s2, tr);
    s3 += fabs_(tr.h * r.h);
    mV += (am[k] + bm[k] * fabs_(xx.h)) * fabs_(r.h);
  }
  const ff Q = ff_mul(T, ff_sub(ff_mul(cpM, s2), ff_sqr(s1)));
  // what the terms' rounding (2^-46 of their magnitudes) leaves in p, times
  // d ln c / d p, in 2^-45
  const float rel = mV * s3 * fabs_(frcp(dV * s2.h));
  const ff Xf = ff_mul(ff_mul(T, s1), inv);
  const ff cf = ff_sqrt(ff_mul(ff_mul(cpM, Mt), ff_rcp(Q)));
  const float LO = 8.67e-19f, HI = 1.15e18f;   // 2^-60, 2^60
  const bool ok = rel <= 16.f && fabs_(dx) <= 1e-9f * pm && pm > LO && pm < HI && T.h > LO && T.h < HI && Mt.h > LO &&
                  cf.h > LO && cf.h < HI && fabs_(Xf.h) < HI && s2.h > 1e-30f;
  if (!ok) return false;
  X = ff_double(Xf);
  c = ff_double(cf);
  // 1 / c to FP64 rounding: the back-projection relies on c (1 / c) = 1
  const double r0 = ff_widen(frcp(cf.h), 1023);
  double e = dfma(-c, r0, 1.0);
  e = dfma(e, e, e);
  ic = dfma(r0, e, r0);
  return true;
}

// the sound speed at (P, T, Y) and specific volume v: a = c v with
// c^2 = cp / (T (cp S_2 - S_1^2)), S_q = sum Y_k R_k / (P + Pinf_k)^q.
// False beyond 2^-60..2^60: the caller takes the FP64 form.
template <int NS>
MPMC_FF bool sound_speed_ff(const SpeciesFF* sp, const double* Y, const double p, const double T, const double v,
                            double& a) {
  const uint32_t A = 0x7fffffffu, TOP = (1023u + 60u) << 20, BOT = (1023u - 60u) << 20;
  const uint32_t hp = dhi(p) & A, hT = dhi(T), hv = dhi(v);
  if (hp >= TOP || hT - BOT >= TOP - BOT || hv - BOT >= TOP - BOT) return false;
  const ff P0 = ff_of(p), T0 = ff_of(T);
  ff cp = {0.f, 0.f}, s1 = {0.f, 0.f}, s2 = {0.f, 0.f};
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const ff y = ff_of(Y[k]);
    const ff r = y.h != 0.f ? ff_rcp(ff_add(P0, sp[k].pinf)) : ff{0.f, 0.f};
    const ff z = ff_mul(ff_mul(y, sp[k].R), r);
    cp = ff_add(cp, ff_mul(y, sp[k].cp));
    s1 = ff_add(s1, z);
    s2 = ff_add(s2, ff_mul(z, r));
  }
  const ff Q = ff_mul(T0, ff_sub(ff_mul(cp, s2), ff_sqr(s1)));
  if (!(Q.h > 1e-30f && s2.h > 1e-30f && cp.h > 8.67e-19f && cp.h < 1.15e18f)) return false;
  a = ff_double(ff_mul(ff_sqrt(ff_mul(cp, ff_rcp(Q))), ff_of(v)));
  return true;
}

}  // namespace mpmc
