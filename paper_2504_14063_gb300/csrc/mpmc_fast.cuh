// The forward FP64 face pass (arXiv 2504.14063): mpmc_kernels.cuh's k_face
// with the parts of its arithmetic that act on the cells' differences only
// moved from the FP64 pipe (2 operations per clock and SM on GB300) to
// float-float on the FP32 pipe (mpmc_ff.h says what that rests on).  Face
// passes of one SSP-RK3 step, all FP64 and so: shock-bubble 1024 x 512 8.70 ->
// 2.88 ms, droplet field 128^3 79.7 -> 26.0 ms.  Of the plain form's FP64
// instructions about 590 per face are left (3D, four species, CDI and diffusion);
// the pipe is 70 % busy with them (86 % before) at 25 % of the warps, the rest
// latency of the FP32 chains and of instruction fetches.
// The right-hand sides' error against extended precision is 0.5 to 1.0 of the
// FP64 form's (four workloads, every field; tests/test_gpu_forward_accuracy.py).
//
// Steps and right-hand sides run these kernels, unless they return limiter
// flags for a reverse pass.  Those, the recording calls of the discrete adjoint
// (mpmc_rk_step_record, mpmc_rk_step_replay) and what mpmc_rk_step_adjoint and
// mpmc_rhs_adjoint recompute run mpmc_kernels.cuh's: the reverse sweep
// evaluates the faces in that form, and the derivative it takes is
// discontinuous in the states' rounding (the mass-fraction limiter acts
// unless sum Y is one to 1e-15, a stencil of rounding noise has weights of
// its own), so the states it linearizes at keep that form's rounding.
#pragma once
#include "mpmc_kernels.cuh"

namespace mpmc {
namespace fast {

// the FP64 form of both sides, for stencils outside the range of the
// float-float one (differences that are not finite or beyond 2^900); out of
// line, so that it costs the callers no registers
template <int RC>
__device__ __noinline__ double2 eno_lr_fp64(double w0, double w1, double w2, double w3, double w4, double w5,
                                            double eps) {
  const double w[6] = {w0, w1, w2, w3, w4, w5};
  double L, R;
  mpmc::recon_lr<RC>(w, eps, L, R);
  return make_double2(L, R);
}

// Out of line: a face interpolates nine fields (3D, four species), and the code
// of all of them inlined (17,000 instructions of a face) does not fit the
// instruction caches; the pass then waited for instructions three times as
// long as it issued them (droplet field 128^3, faces of a step: 46.4 ms
// inlined, 39.3 ms with this function called, 33.8 ms with the face states
// and the limiter's tests called too).
// two: twice the method's field (eps, compared with its square, then counts
// four times).  (In the FP64 form of TENO and WENO5-JS, whose eps is fixed,
// the doubled field is halved and its values doubled.)
template <int RC>
__device__ __noinline__ double2 eno_lr(double w0, double w1, double w2, double w3, double w4, double w5, float eh,
                                       float el, int ee, int two) {
  const double w[6] = {w0, w1, w2, w3, w4, w5};
  WenoEps e = {eh, el, ee + 2 * two};
  if constexpr (RC == RC_WENO5JS) e = js_eps4(2 * two);
  if constexpr (RC == RC_TENO5 || RC == RC_TENO6) e = teno_eps4(2 * two);
  double L, R;
  if (eno_lr_ff<RC>(w, e, L, R)) return make_double2(L, R);
  const double h = two ? 0.5 : 1.0, g = two ? 2.0 : 1.0;
  double2 v = eno_lr_fp64<RC>(h * w0, h * w1, h * w2, h * w3, h * w4, h * w5,
                              0.25 * scalbn((double)eh + (double)el, ee));
  v.x *= g;
  v.y *= g;
  return v;
}

// both face values of one field from the cells y[0..5] = i-2..i+3 around
// the face i+1/2, in float-float (mpmc_ff.h).  TWICE: the field is twice the
// method's.
template <int RC, bool TWICE = false>
__device__ __forceinline__ void recon_lr(const KParams& P, const double* y, double& L, double& R) {
  const double2 v = eno_lr<RC>(y[0], y[1], y[2], y[3], y[4], y[5], P.weno_eps4.h, P.weno_eps4.l, P.weno_eps4.e,
                               TWICE ? 1 : 0);
  L = v.x;
  R = v.y;
}

// F(S) + s (U*_S - U_S): the HLLC flux on the side S of the contact the
// face lies on (s = min(0, s_L) for the left side, max(0, s_R) for the right,
// sS its wave speed, dS = sS - u_S, du = ss - u_S), collected around the two
// factors
//   m = u_S + s (f - 1),  w = s f du,  f = dS / (sS - ss),
// with f - 1 = du / (dS - du) formed without the difference
template <int NS, int D>
__device__ __forceinline__ void hllc_one(int d, const State<NS>& S, double s, double dS, double du, double ss,
                                          double* F) {
  const double q = du * drcp(dS - du);
  const double m = fma(s, q, S.u[d]), w = fma(s, q, s) * du;
#pragma unroll
  for (int k = 0; k < NS; ++k) F[k] = S.rhoY[k] * m;
#pragma unroll
  for (int j = 0; j < D; ++j) F[NS + j] = S.m[j] * m;
  F[NS + d] += fma(S.rho, w, S.p);
  F[NS + D] = fma(w, fma(S.rho, ss, S.p * drcp(dS)), fma(S.E, m, S.u[d] * S.p));
}

template <int NS, int D>
__device__ __forceinline__ void hllc_flux(int d, const State<NS>& L, const State<NS>& R, double* F) {
  const double ub = 0.5 * (L.u[d] + R.u[d]), ab = 0.5 * (L.a + R.a);
  const double sL = fmin(ub - ab, L.u[d] - L.a);
  const double sR = fmax(ub + ab, R.u[d] + R.a);
  const double sm = sel_neg(sL, sL, 0.0), sp = sel_neg(sR, 0.0, sR);
  const double dL = sL - L.u[d], dR = sR - R.u[d];
  // the contact speed as an increment on u_L (exactly u where P and u are
  // continuous): ss - u_L = (P_R - P_L - w_R (u_R - u_L)) / (w_L - w_R),
  // w_S = rho_S (s_S - u_S)
  const double wL = L.rho * dL, wR = R.rho * dR, Du = R.u[d] - L.u[d];
  const double duL = fma(-wR, Du, R.p - L.p) * drcp(wL - wR), duR = duL - Du;
  const double ss = L.u[d] + duL;
  // only the side of the contact the face lies on is evaluated; sign(0) = 0
  // takes both with weight 1/2
  if (positive(ss)) {
    hllc_one<NS, D>(d, L, sm, dL, duL, ss, F);
  } else if (negative(ss)) {
    hllc_one<NS, D>(d, R, sp, dR, duR, ss, F);
  } else {
    constexpr int NV = NS + D + 1;
    double FL[NV], FR[NV];
    hllc_one<NS, D>(d, L, sm, dL, duL, ss, FL);
    hllc_one<NS, D>(d, R, sp, dR, duR, ss, FR);
#pragma unroll
    for (int v = 0; v < NV; ++v) F[v] = 0.5 * FL[v] + 0.5 * FR[v];
  }
}

// the sound speed of eos_forward at (P, T, Y) in FP64, out of line: for
// states beyond the float-float one's range
template <int NS>
__device__ __noinline__ double sound_speed_fp64(const KParams& P, const double* Y, const double p, const double T) {
  double rho, e, a, al, be;
  eos_forward<NS>(P, Y, p, T, rho, e, a, al, be);
  return a;
}

// face-side state from reconstructed (Y, u, P, T) (steps 4-5 of Sec. 3.1.3).
// With z_k = Y_k R_k / (P + Pinf_k): v = T sum z_k + sum Y_k b_k and
// e = T (sum Y_k cv_k + sum Pinf_k z_k) + sum Y_k q_k.  The sound speed only
// sets HLLC's wave speeds, which act on the two sides' difference: it is
// float-float (as X and c of the projection).
template <int NS>
__device__ __noinline__ void face_state(const KParams& P, const double* Y, const double* u, double p,
                                                     double T, State<NS>& s) {
  double vs = 0.0, eb = 0.0, vb = 0.0, eq = 0.0, rg = 0.0;
  bool have_rg = false;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    if (nonzero(Y[k])) {
      // ideal-gas species share 1/P
      double r;
      if (!nonzero(P.pinf[k])) {
        if (!have_rg) {
          rg = drcp(p);
          have_rg = true;
        }
        r = rg;
      } else {
        r = drcp(p + P.pinf[k]);
      }
      const double z = (Y[k] * P.Rk[k]) * r;
      vs += z;
      eb = fma(Y[k], P.cv[k], eb);
      if (nonzero(P.pinf[k])) eb = fma(P.pinf[k], z, eb);
      if (P.has_b) vb = fma(Y[k], P.b[k], vb);
      if (P.has_q) eq = fma(Y[k], P.q[k], eq);
    }
  }
  const double v = fma(T, vs, vb), e = fma(T, eb, eq);
  s.rho = drcp(v);
  double ke = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    s.u[d] = u[d];
    s.m[d] = s.rho * u[d];
    ke = fma(u[d], u[d], ke);
  }
#pragma unroll
  for (int k = 0; k < NS; ++k) s.rhoY[k] = s.rho * Y[k];
  s.p = p;
  s.E = s.rho * fma(0.5, ke, e);
  if (!sound_speed_ff<NS>(P.sff, Y, p, T, v, s.a)) {
    double Yc[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) Yc[k] = Y[k];
    s.a = sound_speed_fp64<NS>(P, Yc, p, T);
  }
}

// mass-fraction limiter of Sec. 3.3.1 on one face side (Yc: cell values), as
// y_limiter with its comparisons on the bits and dd from the sign of Yc - Y
// (the same values as min(Y, Yc) - Y and max(Y, Yc) - Y)
template <int NS>
__device__ __forceinline__ bool limit_Y(double* Y, const double* Yc) {
  bool active = false;
#pragma unroll
  for (int k = 0; k < NS; ++k)
    if (negative(Y[k])) {
      Y[k] = 0.0;
      active = true;
    }
  double sum = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) sum += Y[k];
  const double def = 1.0 - sum;
  // (NaN counts as within the tolerance, as in y_limiter)
  const unsigned long long db = (unsigned long long)__double_as_longlong(def) & 0x7fffffffffffffffull;
  if (db > (unsigned long long)__double_as_longlong(NS * YSUM_TOL) && db <= 0x7ff0000000000000ull) {
    const bool over = __double2hiint(def) < 0;
    double dd[NS], Sig = 0.0;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const double t = Yc[k] - Y[k];
      dd[k] = (__double2hiint(t) < 0) == over ? t : 0.0;
      Sig += dd[k];
    }
    if (nonzero(Sig)) {
      const double f = normal_(Sig) ? def * drcp(Sig) : def / Sig;
#pragma unroll
      for (int k = 0; k < NS; ++k) Y[k] = fma(f, dd[k], Y[k]);
      active = true;
    }
  }
  return active;
}

// p-T equilibrium of a cell with r_k = 1 / (P + Pinf_k), for the FP64
// primitive pass: pt_equilibrium<NS, true> in fewer FP64 operations.  The
// closed forms keep its order and its rounding (the pressure of a stiff
// liquid is a small difference); several distinct Pinf: the residual's root
// from FP32, then a float-float Halley step (to ~2^-46 of the residual's
// terms), then one Newton step whose residual is FP64; the general iteration
// where that step is above 5e-10 of the distance to the nearest pole (its
// derivative is FP32: 2^-21 of a step, 2^-52 of that distance at most).
template <int NS>
__device__ __forceinline__ int cell_pt(const KParams& P, const double* Y, double e, double v, double& p, double& T,
                                       double* r) {
  double Cv = 0.0, q = 0.0, b = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    Cv = add_(Cv, mul_(Y[k], P.cv[k]));
    if (P.has_q) q = add_(q, mul_(Y[k], P.q[k]));
    if (P.has_b) b = add_(b, mul_(Y[k], P.b[k]));
  }
  const double em = P.has_q ? sub_(e, q) : e, vm = P.has_b ? sub_(v, b) : v;
  int st = ST_OK;
  if (!positive(em) || !positive(vm)) st = ST_INADMISSIBLE;
  const double Ep = normal_(vm) ? ddiv(em, vm, drcp(vm)) : em / vm;
  double pl = -1.0, Rg = 0.0, Rl = 0.0;
  bool multi = false, gas = false;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    if (positive(Y[k])) {
      if (positive(P.pinf[k])) {
        if (negative(pl)) pl = P.pinf[k];
        else if (bits_of(P.pinf[k]) != bits_of(pl)) multi = true;
        Rl = add_(Rl, mul_(Y[k], P.Rk[k]));
      } else {
        gas = true;
        Rg = add_(Rg, mul_(Y[k], P.Rk[k]));
      }
    }
  }
  if (!multi) {
    double num, den = Cv;
    if (negative(pl)) {
      num = mul_(Ep, Rg);
    } else if (!gas) {
      num = sub_(sub_(mul_(Ep, Rl), mul_(pl, Cv)), mul_(pl, Rl));
    } else {
      const double a2 = sub_(sub_(mul_(Ep, add_(Rg, Rl)), mul_(pl, Cv)), mul_(pl, Rl));
      const double a3 = mul_(mul_(Ep, pl), Rg);
      const double sq = sqrt(add_(mul_(a2, a2), mul_(mul_(4.0, Cv), a3)));
      const double w = add_(fabs(a2), sq);
      const bool neg = negative(a2);
      num = neg ? mul_(2.0, a3) : w;
      den = neg ? w : mul_(2.0, Cv);
    }
    p = normal_(den) ? ddiv(num, den, drcp(den)) : num / den;
#pragma unroll
    for (int k = 0; k < NS; ++k) r[k] = qdiv(1.0, p + P.pinf[k]);
  } else {
    double w[NS], pmin = 1e300;
    int big = 0;   // the largest |w|'s high word
    ff wf[NS];
    const ff Cf = ff_of(Cv);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      if (positive(Y[k]) && bits_of(P.pinf[k]) < bits_of(pmin)) pmin = P.pinf[k];   // (Pinf >= 0)
      w[k] = nonzero(Y[k]) ? (Y[k] * P.Rk[k]) * (Ep - P.pinf[k]) : 0.0;
      wf[k] = ff_of(w[k]);
      big = max(big, __double2hiint(w[k]) & 0x7fffffff);
    }
    const double lo = -pmin;
    // the quadratic with the liquids merged into one, then the residual, in FP32
    float x;
    {
      float Rgf = 0.f, Rlf = 0.f, wl = 0.f;
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const float yr = narrow(Y[k]) * P.f32.Rk[k];
        if (P.f32.pinf[k] > 0.f) {
          Rlf += yr;
          wl += yr * P.f32.pinf[k];
        } else {
          Rgf += yr;
        }
      }
      const float Ef = narrow(Ep), pe = wl / Rlf;
      const float a2 = Ef * (Rgf + Rlf) - pe * Cf.h - pe * Rlf;
      const float sq = sqrtf(fmaxf(a2 * a2 + 4.f * Cf.h * (Ef * pe * Rgf), 0.f));
      x = a2 >= 0.f ? (a2 + sq) / (2.f * Cf.h) : 2.f * (Ef * pe * Rgf) / (sq - a2);
    }
    const float lof = narrow(lo);
    if (!(x > lof)) x = lof + fmaxf(fabsf(lof), 1.f);
    x = (float)pt_start_f32<NS>(P, Y, w, Cv, lo, (double)x);
    // float-float residual, its derivatives in FP32: a Halley step
    ff xx = {x, 0.f};
    float df = 0.f, d2 = 0.f;
    {
      ff f = {-Cf.h, -Cf.l};
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        if (nonzero(Y[k])) {
          const ff rk = ff_rcp(ff_add(xx, P.sff[k].pinf));
          const ff t = ff_mul(wf[k], rk);
          f = ff_add(f, t);
          df -= t.h * rk.h;
          d2 += 2.f * t.h * rk.h * rk.h;
        }
      }
      const float h = 1.f - 0.5f * f.h * d2 / (df * df);
      xx = ff_add(xx, ff{-f.h / (df * h), 0.f});
    }
    p = ff_double(xx);
    // Newton with the FP64 residual (its derivative in FP32); 1 / (p + Pinf)
    // follows the step to first order
    double fd = -Cv;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      r[k] = drcp(p + P.pinf[k]);
      if (nonzero(Y[k])) fd = fma(w[k], r[k], fd);
    }
    const float dxf = -narrow(fd) / df;
    if (big < (1023 + 100) << 20 && fabsf(dxf) <= 5e-10f * (xx.h - lof) && xx.h < 1e30f) {
      const double dx = ff_widen(dxf, 1023);
      p += dx;
#pragma unroll
      for (int k = 0; k < NS; ++k) r[k] = fma(-dx * r[k], r[k], r[k]);
    } else {
      double Tg;
      const int s2 = pt_equilibrium<NS>(P, Y, e, v, p, Tg);
      if (st == ST_OK) st = s2;
#pragma unroll
      for (int k = 0; k < NS; ++k) r[k] = 1.0 / (p + P.pinf[k]);
    }
  }
  double den = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k)
    if (nonzero(Y[k])) {
      const double c = Y[k] * P.cv[k];
      den = add_(den, nonzero(P.pinf[k]) ? ddiv(mul_(c, add_(p, mul_(P.gam[k], P.pinf[k]))), p + P.pinf[k], r[k]) : c);
    }
  T = normal_(den) ? ddiv(em, den, drcp(den)) : em / den;
  return st;
}

// ---------------------------------------------------------------------------
// the forward FP64 primitive pass: mpmc_kernels.cuh's k_prim with its divisions
// taken from shared reciprocals and the several-liquid p-T solve's iterations
// on the FP32 pipe (cell_pt)
template <int NS, int D>
__global__ void __launch_bounds__(CELL_THREADS)
    k_prim(const KParams P, const double* __restrict__ U, const double* __restrict__ Uin, double* __restrict__ Wc,
           unsigned long long* __restrict__ red, int* __restrict__ status) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double smax = 0.0, gmax = 0.0;
  if (c < P.ncell + P.nextra) {
    constexpr int NV = NS + D + 1;
    double Uc[NV];
    if (c >= P.ncell) {
      // the inflow state or a characteristic ghost, from U's ghost buffer
#pragma unroll
      for (int v = 0; v < NV; ++v) Uc[v] = Uin[(long long)v * P.gstride + (c - P.ncell)];
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) Uc[v] = U[(long long)v * P.ncell + c];
    }
    const long long ws = P.wstride;
    // decode in the oracle's order and rounding, the divisions by rho from one
    // reciprocal
    double rho = 0.0, Y[NS], u[3], e, irho, ke = 0.0;
#pragma unroll
    for (int k = 0; k < NS; ++k) rho = add_(rho, Uc[k]);
    if (normal_(rho)) {
      irho = drcp(rho);
      irho = fma(fma(-rho, irho, 1.0), irho, irho);
#pragma unroll
      for (int k = 0; k < NS; ++k) Y[k] = ddiv(Uc[k], rho, irho);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        u[d] = d < D ? ddiv(Uc[NS + d], rho, irho) : 0.0;
        if (d < D) ke = add_(ke, mul_(u[d], u[d]));
      }
      e = sub_(ddiv(Uc[NS + D], rho, irho), mul_(0.5, ke));
    } else {
      decode<NS, D>(Uc, rho, Y, u, e, irho);
    }
    int st = positive(rho) ? ST_OK : ST_INADMISSIBLE;
    if (!rhoY_admissible<NS>(Uc, rho)) st = ST_INADMISSIBLE;
    double p, T, r[NS];
    const int st2 = cell_pt<NS>(P, Y, e, irho, p, T, r);
    if (st == ST_OK) st = st2;
    // sound speed: a = c v, c^2 = cp / (T (cp S_2 - S_1^2)), S_q = sum Y_k R_k r_k^q
    double a, z[NS];
    {
      double cp = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        z[k] = nonzero(Y[k]) ? (Y[k] * P.Rk[k]) * r[k] : 0.0;
        cp = fma(Y[k], P.cp[k], cp);
        s1 += z[k];
        if (nonzero(Y[k])) s2 = fma(z[k], r[k], s2);
      }
      a = (cp * irho) * drsqrt(cp * (T * fma(cp, s2, -s1 * s1)));
    }
    Wc[P.wT * ws + c] = T;
    Wc[P.wP * ws + c] = p;
    Wc[P.wRho * ws + c] = rho;
    Wc[P.wA * ws + c] = a;
#pragma unroll
    for (int k = 0; k < NS; ++k) Wc[(P.wY + k) * ws + c] = Y[k];
#pragma unroll
    for (int d = 0; d < D; ++d) Wc[(P.wU + d) * ws + c] = u[d];

    double mu = 0.0, lam = 0.0;
    if (P.cdi || P.diffusion || P.viscous) {
      double phi[2], Yp[2];
#pragma unroll
      for (int ph = 0; ph < 2; ++ph) {
        // phi_p = sum U_k v_k, h_p rho_p phi_p = sum U_k h_k in the oracle's
        // order and rounding, the quotients corrected: the regularization flux is
        // the difference of phi against its sharpening, and with a rounding or two
        // more in phi the right-hand side's error in a liquid was 1.1 to 1.5 times
        // as large (bubble, shock onto a droplet)
        double f = 0.0, hr = 0.0, yp = 0.0;
#pragma unroll
        for (int k = 0; k < NS; ++k)
          if (P.phase[k] == ph) {
            yp += Y[k];
            if (nonzero(Uc[k])) {
              double vk = ddiv(mul_(P.Rk[k], T), add_(p, P.pinf[k]), r[k]), hk = mul_(P.cp[k], T);
              if (P.has_b) {
                vk = add_(vk, P.b[k]);
                hk = add_(hk, mul_(P.b[k], p));
              }
              if (P.has_q) hk = add_(hk, P.q[k]);
              f = add_(f, mul_(Uc[k], vk));
              hr = add_(hr, mul_(Uc[k], hk));
            }
          }
        phi[ph] = f;
        Yp[ph] = yp;
        if (P.cdi) {
          const bool present = yp >= ABSENT, norm = normal_(f);
          const double rf = norm ? drcp(f) : 0.0;
          Wc[(P.wHrho + ph) * ws + c] = present ? (norm ? ddiv(hr, f, rf) : hr / f) : 0.0;
#pragma unroll
          for (int k = 0; k < NS; ++k)
            if (P.phase[k] == ph)
              Wc[(P.wYrho + k) * ws + c] = present ? (norm ? ddiv(Uc[k], f, rf) : Uc[k] / f) : 0.0;
        }
      }
      if (P.cdi) {
        Wc[P.wPhi0 * ws + c] = phi[0];
        const double num = phi[0] + P.psi_delta, den = phi[1] + P.psi_delta;
        Wc[P.wPsi * ws + c] = P.cdi_eps * log(normal_(den) ? ddiv(num, den, drcp(den)) : num / den);
      }
      // phase viscosities: liquid constant, gas by Wilke's rule
      double mup[2] = {P.mu_liquid, 0.0};
      if (P.diffusion || P.viscous) {
        double num = 0.0;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
          if (P.phase[i] != 1) continue;
          double den = 0.0;
#pragma unroll
          for (int j = 0; j < NS; ++j)
            if (P.phase[j] == 1) den = fma(Y[j], P.wilke[i][j], den);
          if (positive(den)) num += qdiv(Y[i] * P.mu[i], den);
        }
        mup[1] = Yp[1] >= ABSENT ? num : 0.0;
        mu = phi[0] * mup[0] + phi[1] * mup[1];
      }
      if (P.viscous) {
        // heat conductivity: liquid constant, gas (mu_g / Pr) sum (Y^c/Y_g) Cp^c
        double cpY = 0.0;
#pragma unroll
        for (int k = 0; k < NS; ++k)
          if (P.phase[k] == 1) cpY += Y[k] * P.cp[k];
        const double lam_g = Yp[1] >= ABSENT ? mup[1] / P.prandtl * (cpY / Yp[1]) : 0.0;
        lam = phi[0] * P.lambda_liquid + phi[1] * lam_g;
        Wc[P.wMu * ws + c] = mu;
        Wc[P.wLam * ws + c] = lam;
      }
      if (P.diffusion) {
        // X^c/X_p = (Y^c/W^c) / sY, sY = sum_p Y/W;
        // W^c D^c / W_p = (W^c/Sc^c) (sY/Y_p) mu_p (phi_p/Y_p) / rho
#pragma unroll
        for (int ph = 0; ph < 2; ++ph) {
          double sY = 0.0, yw[NS];
#pragma unroll
          for (int j = 0; j < NS; ++j)
            if (P.phase[j] == ph) {
              yw[j] = Y[j] * P.iW[j];
              sY += yw[j];
            }
          const bool present = Yp[ph] >= ABSENT && sY >= ABSENT;
          const double ry = qdiv(1.0, Yp[ph]), rs = qdiv(1.0, sY);
          const double Bp = (sY * ry) * ((mup[ph] * irho) * (phi[ph] * ry));
#pragma unroll
          for (int k = 0; k < NS; ++k) {
            if (P.phase[k] != ph) continue;
            Wc[(P.wXr + k) * ws + c] = present ? yw[k] * rs : 0.0;
            Wc[(P.wB + k) * ws + c] = present ? P.WSc[k] * Bp : 0.0;
          }
        }
      }
    }
    if (st != ST_OK) atomicMax(status, st);
    if (c < P.ncell) {
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const double ud = fabs(u[d]);
        smax = fmax(smax, (ud + a) * P.inv_dx);
        gmax = fmax(gmax, ud);
      }
      if (P.diffusion || P.viscous) smax = fmax(smax, 4.0 * mu * irho * (P.inv_dx * P.inv_dx));
      if (P.viscous) {
        // conduction limit with the thermal diffusivity lambda / (rho cv)
        double cv = 0.0;
#pragma unroll
        for (int k = 0; k < NS; ++k) cv += Y[k] * P.cv[k];
        smax = fmax(smax, 4.0 * lam / (rho * cv) * (P.inv_dx * P.inv_dx));
      }
    }
  }
  if (red) block_max2(smax, gmax, red);
}

// ---------------------------------------------------------------------------
// y >= ABSENT (false for NaN) from the bits
__device__ __forceinline__ bool present_(double y) {
  const long long b = __double_as_longlong(y);
  return b >= __double_as_longlong(ABSENT) && b <= 0x7ff0000000000000ll;
}

// ---------------------------------------------------------------------------
// velocity component t of a mapped cell, negated where a wall mirrors it
__device__ __forceinline__ double uget(const KParams& P, const double* __restrict__ Wc, int t, CRef r) {
  return mirror(wget(P, Wc, P.wU + t, r), r.flip, t);
}

// ---------------------------------------------------------------------------
// partial densities of a mapped cell (as load_U)
template <int NS>
__device__ __forceinline__ void load_rhoY(const KParams& P, const double* __restrict__ U,
                                          const double* __restrict__ G, CRef r, double* out) {
  const bool ghost = r.idx >= P.ncell;
  const double* p = ghost ? G + (r.idx - P.ncell) : U + r.idx;
  const long long st = ghost ? P.gstride : P.ncell;
#pragma unroll
  for (int k = 0; k < NS; ++k) out[k] = p[(long long)k * st];
}

// X and c of the averaged state in FP64: the p-T equilibrium of the averaged
// conserved vector, for faces whose float-float solve (face_avg_ff) does not
// settle or leaves its range; out of line, so that it costs the face kernel
// no registers
template <int NS, int D>
__device__ __noinline__ double2 face_avg_fp64(const KParams& P, const double* Wc, const double* Uk, const double* Uin,
                                              const CRef ri, const CRef rj) {
  constexpr int NV = NS + D + 1;
  double Ui[NV], Uj[NV];
  load_U<NS, D>(P, Uk, Uin, ri, Ui);
  load_U<NS, D>(P, Uk, Uin, rj, Uj);
#pragma unroll
  for (int v = 0; v < NV; ++v) Ui[v] = 0.5 * (Ui[v] + Uj[v]);
  // these scalars only shape the projection: ordinary (contracted) arithmetic
  double rho, Y[NS], uu[3], e, vol, p, T, a, al, be;
  decode<NS, D, false>(Ui, rho, Y, uu, e, vol);
  // the Newton start of several stiffened liquids: the mean of the two
  // cells' pressures, close to the averaged state's
  pt_equilibrium<NS, false>(P, Y, e, vol, p, T, rho,
                            0.5 * (wget(P, Wc, P.wP, ri) + wget(P, Wc, P.wP, rj)));
  eos_char<NS>(P, Y, p, T, rho, a, al, be);
  return make_double2((rho * a * a * be - 1.0) / (al * a * a * rho), a * rho);
}

// ---------------------------------------------------------------------------
// DIR: the face direction, a template parameter so that every array indexed
// by it is indexed by a constant (registers, not the stack).  RC: the
// ENO-type interpolation (RC_WENO5Z, the method's, or one of Sec. 4.1's others)
// Four blocks per SM (128 registers): more warps hide the latencies of the
// FP64 and FP32 chains (three or two blocks, unbounded registers: 20 % slower;
// five and six, with spills: within 5 % either way).
// SPLIT: a block is 32 faces x one warp per interpolated field (in the order
// T, u_d + and -, Y_k, u_t): every warp forms X and c and interpolates its
// field, the second builds the right states beside the first's left ones, the
// first finishes the faces.  On a grid that leaves most warp slots empty the
// pass lasts as long as one thread's chain of operations, which this shortens:
// 100 and 400 cells in 1D, per pass 31 -> 24 and 27 -> 20 us (the same bits).
template <int NS, int D>
constexpr int SPLIT_WARPS = 3 + NS + (D - 1);

template <int NS, int D, int DIR, int RC, bool SPLIT = false>
__global__ void __launch_bounds__(SPLIT ? 32 * SPLIT_WARPS<NS, D> : FACE_THREADS, SPLIT ? 1 : 4)
    k_face(const __grid_constant__ KParams P, const double* __restrict__ Wc, const double* __restrict__ Un,
           const double* __restrict__ Uk, const double* __restrict__ Uin, const double* __restrict__ scal,
           const double rk0, const double rk1, const double rk2, double* __restrict__ F,
           unsigned long long* __restrict__ stats) {
  constexpr int NV = NS + D + 1;
  constexpr int d = DIR;
  const int f0 = P.n[0] + (d == 0), f1 = P.n[1] + (d == 1), f2 = P.n[2] + (d == 2);
  const long long nf = (long long)f0 * f1 * f2;
  const int role = SPLIT ? (int)threadIdx.x >> 5 : 0, lane = (int)threadIdx.x & 31;
  // (split: lanes beyond the last face repeat it, unstored)
  long long fid = SPLIT ? (long long)blockIdx.x * 32 + lane : (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = fid < nf;
  if (SPLIT) fid = live ? fid : nf - 1;
  else if (!live) return;
  int fc[3];
  unflatten(fid, f0, f1, fc);
  int ci[3] = {fc[0], fc[1], fc[2]};
  ci[d] -= 1;  // the cell on the low side of the face
  const double dt = scal[0], Gamma = scal[1];
  // FP32 roundings for the limiter's tests
  const float rk0f = lim_narrow(rk0), rk1f = lim_narrow(rk1), rk2f = lim_narrow(rk2),
              dtdx = lim_narrow(dt) * P.f32.inv_dx;

  CRef cr[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    int cc[3] = {ci[0], ci[1], ci[2]};
    cc[d] += j - 2;
    cr[j] = map_cell_m<1u << d>(P, cc[0], cc[1], cc[2]);
  }
  const CRef ri = cr[2], rj = cr[3];
  uint32_t fl = 0u;

  // step 1: the scalars of the characteristic matrices (Appendix A) at the
  // averaged conserved state
  double X, c, ic;
  {
    double mi[NS], mj[NS], ui[3] = {0.0, 0.0, 0.0}, uj[3] = {0.0, 0.0, 0.0};
    load_rhoY<NS>(P, Uk, Uin, ri, mi);
    load_rhoY<NS>(P, Uk, Uin, rj, mj);
#pragma unroll
    for (int t = 0; t < D; ++t) {
      ui[t] = uget(P, Wc, t, ri);
      uj[t] = uget(P, Wc, t, rj);
    }
    if (!face_avg_ff<NS, D>(P.sff, mi, mj, wget(P, Wc, P.wP, ri), wget(P, Wc, P.wP, rj), wget(P, Wc, P.wT, ri),
                            wget(P, Wc, P.wT, rj), ui, uj, X, c, ic)) {
      const double2 v = face_avg_fp64<NS, D>(P, Wc, Uk, Uin, ri, rj);
      X = v.x;
      c = v.y;
      ic = 1.0 / c;
    }
  }

  // steps 2-3: project, interpolate both sides (WENO5-Z unless RC says
  // otherwise), back to physical space
  double YL[NS], YR[NS], uL[3] = {0.0, 0.0, 0.0}, uR[3] = {0.0, 0.0, 0.0}, PL, PR, TL, TR;
  if constexpr (SPLIT) {
    constexpr int NFLD = SPLIT_WARPS<NS, D>;
    __shared__ double sh[2][NFLD][32];
    {
      double y[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        if (role < 3) {
          const double p = wget(P, Wc, P.wP, cr[j]);
          if (role == 0) y[j] = fma(-X, p, wget(P, Wc, P.wT, cr[j]));
          else y[j] = fma(role == 1 ? c : -c, uget(P, Wc, d, cr[j]), p);
        } else if (role < 3 + NS) {
          y[j] = wget(P, Wc, P.wY + role - 3, cr[j]);
        } else {
          // the tangential directions in increasing order
          const int q = role - 3 - NS, t = q < d ? q : q + 1;
          y[j] = uget(P, Wc, t, cr[j]);
        }
      }
      const double2 v = eno_lr<RC>(y[0], y[1], y[2], y[3], y[4], y[5], P.weno_eps4.h, P.weno_eps4.l, P.weno_eps4.e,
                                   role == 1 || role == 2 ? 1 : 0);
      sh[0][role][lane] = v.x;
      sh[1][role][lane] = v.y;
    }
    __syncthreads();
    PL = 0.5 * (sh[0][1][lane] + sh[0][2][lane]);
    PR = 0.5 * (sh[1][1][lane] + sh[1][2][lane]);
    TL = fma(X, PL, sh[0][0][lane]);
    TR = fma(X, PR, sh[1][0][lane]);
    uL[d] = (0.5 * ic) * (sh[0][1][lane] - sh[0][2][lane]);
    uR[d] = (0.5 * ic) * (sh[1][1][lane] - sh[1][2][lane]);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      YL[k] = sh[0][3 + k][lane];
      YR[k] = sh[1][3 + k][lane];
    }
#pragma unroll
    for (int t = 0; t < D; ++t) {
      if (t == d) continue;
      const int q = 3 + NS + (t < d ? t : t - 1);
      uL[t] = sh[0][q][lane];
      uR[t] = sh[1][q][lane];
    }
  } else {
  {
    double w1[6], w5[6], w6[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const double T = wget(P, Wc, P.wT, cr[j]);
      const double p = wget(P, Wc, P.wP, cr[j]);
      const double un = uget(P, Wc, d, cr[j]);
      // (twice Appendix A's w5 and w6: the halves are taken once, on the way back)
      w1[j] = fma(-X, p, T);
      w5[j] = fma(c, un, p);
      w6[j] = fma(-c, un, p);
    }
    double w1L, w1R, w5L, w5R, w6L, w6R;
    fast::recon_lr<RC>(P, w1, w1L, w1R);
    fast::recon_lr<RC, true>(P, w5, w5L, w5R);
    fast::recon_lr<RC, true>(P, w6, w6L, w6R);
    PL = 0.5 * (w5L + w6L);
    PR = 0.5 * (w5R + w6R);
    TL = fma(X, PL, w1L);
    TR = fma(X, PR, w1R);
    uL[d] = (0.5 * ic) * (w5L - w6L);
    uR[d] = (0.5 * ic) * (w5R - w6R);
  }
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    double y[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) y[j] = wget(P, Wc, P.wY + k, cr[j]);
    fast::recon_lr<RC>(P, y, YL[k], YR[k]);
  }
#pragma unroll
  for (int t = 0; t < D; ++t) {
    if (t == d) continue;
    double y[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) y[j] = uget(P, Wc, t, cr[j]);
    fast::recon_lr<RC>(P, y, uL[t], uR[t]);
  }

  }

  // cell values of the two face neighbours
  double Yi[NS], Yj[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    Yi[k] = wget(P, Wc, P.wY + k, ri);
    Yj[k] = wget(P, Wc, P.wY + k, rj);
  }
  const double Ti = wget(P, Wc, P.wT, ri), Tj = wget(P, Wc, P.wT, rj);
  const double Pi = wget(P, Wc, P.wP, ri), Pj = wget(P, Wc, P.wP, rj);

  // interpolation limiters (Sec. 3.3.1)
  if (P.pos_limiter) {
    if (limit_Y<NS>(YL, Yi)) fl |= F_YLIM_L;
    if (limit_Y<NS>(YR, Yj)) fl |= F_YLIM_R;
    if (!positive(TL)) { TL = Ti; fl |= F_THETA_T_L; }
    if (!positive(TR)) { TR = Tj; fl |= F_THETA_T_R; }
    bool okL = true, okR = true;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      if (positive(YL[k]) && !positive(PL + P.pinf[k])) okL = false;
      if (positive(YR[k]) && !positive(PR + P.pinf[k])) okR = false;
    }
    if (!okL) { PL = Pi; fl |= F_THETA_P_L; }
    if (!okR) { PR = Pj; fl |= F_THETA_P_R; }
  }

  // steps 4-6: face EOS, conserved face states, HLLC
  double Fx[NV];
  {
    State<NS> sL, sR;
    if constexpr (SPLIT) {
      // the second warp builds the right state; the others are done
      __shared__ State<NS> sh[32];
      if (role == 1) {
        face_state<NS>(P, YR, uR, PR, TR, sR);
        sh[lane] = sR;
      } else if (role == 0) {
        face_state<NS>(P, YL, uL, PL, TL, sL);
      }
      __syncthreads();
      if (role != 0 || !live) return;
      sR = sh[lane];
    } else {
      face_state<NS>(P, YL, uL, PL, TL, sL);
      face_state<NS>(P, YR, uR, PR, TR, sR);
    }
    hllc_flux<NS, D>(d, sL, sR, Fx);
  }

  // flux limiter (Sec. 3.3.2): pseudo-updates of both cells, tested on the
  // FP32 pipe with a margin and in FP64 where that cannot decide.  The up to
  // three tests of a face were a tenth of its FP64 operations.
  float Bi[NV], Bj[NV], Mi[NV], Mj[NV];
  const float lamf = (float)(2 * D) * (rk2f * dtdx);
  if (P.pos_limiter) {
    limiter_base<NS, D>(P, Un, Uk, Uin, ri, rk0f, rk1f, Bi, Mi);
    limiter_base<NS, D>(P, Un, Uk, Uin, rj, rk0f, rk1f, Bj, Mj);
  }
  auto passes = [&](const double* Ft) {
    float Ff[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Ff[v] = lim_narrow(Ft[v]);
    const int a = admissible_fp32<NS, D>(P, Bi, Mi, Ff, -lamf);
    if (a == 0) return false;
    const int b = admissible_fp32<NS, D>(P, Bj, Mj, Ff, lamf);
    if (b == 0) return false;
    if (a == 1 && b == 1) return true;
    const double lam = 2.0 * D * rk2 * dt * P.inv_dx;
    double tmp[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) tmp[v] = Ft[v];
    return admissible_fp64<NS, D>(P, Un, Uk, Uin, ri, tmp, rk0, rk1, -lam) &&
           admissible_fp64<NS, D>(P, Un, Uk, Uin, rj, tmp, rk0, rk1, lam);
  };
  if (P.pos_limiter && !passes(Fx)) {
    double Uki[NV], Ukj[NV];
    load_U<NS, D>(P, Uk, Uin, ri, Uki);
    load_U<NS, D>(P, Uk, Uin, rj, Ukj);
    State<NS> si, sj;
    si.rho = wget(P, Wc, P.wRho, ri);
    sj.rho = wget(P, Wc, P.wRho, rj);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      si.rhoY[k] = Uki[k];
      sj.rhoY[k] = Ukj[k];
    }
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      si.u[t] = t < D ? uget(P, Wc, t, ri) : 0.0;
      sj.u[t] = t < D ? uget(P, Wc, t, rj) : 0.0;
      si.m[t] = t < D ? Uki[NS + t] : 0.0;
      sj.m[t] = t < D ? Ukj[NS + t] : 0.0;
    }
    si.p = Pi;
    sj.p = Pj;
    si.E = Uki[NS + D];
    sj.E = Ukj[NS + D];
    si.a = wget(P, Wc, P.wA, ri);
    sj.a = wget(P, Wc, P.wA, rj);
    hllc_flux<NS, D>(d, si, sj, Fx);
    fl |= F_HLLC_FALLBACK;
  }

  // interface regularization (Sec. 3.2), KEEP split form, with its limiter
  if (P.cdi && P.two_phase) {
    bool pres_i[2] = {false, false}, pres_j[2] = {false, false};
    {
      // (branches on the phase rather than ypi[P.phase[k]]: an array indexed
      // at run time would live on the stack)
      double ypi[2] = {0.0, 0.0}, ypj[2] = {0.0, 0.0};
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        if (P.phase[k]) {
          ypi[1] += Yi[k];
          ypj[1] += Yj[k];
        } else {
          ypi[0] += Yi[k];
          ypj[0] += Yj[k];
        }
      }
#pragma unroll
      for (int ph = 0; ph < 2; ++ph) {
        pres_i[ph] = present_(ypi[ph]);
        pres_j[ph] = present_(ypj[ph]);
      }
    }
    if ((pres_i[0] || pres_j[0]) && (pres_i[1] || pres_j[1])) {
      const double psi_i = wget(P, Wc, P.wPsi, ri), psi_j = wget(P, Wc, P.wPsi, rj);
      const double dphi = wget(P, Wc, P.wPhi0, rj) - wget(P, Wc, P.wPhi0, ri);
      // the interface normal n_d = d_d psi / |grad psi| from 4 dx grad psi;
      // zero where |grad psi| < GTOL (the comparisons on the bits)
      double g[3] = {0.0, 0.0, 0.0};
      g[d] = 4.0 * (psi_j - psi_i);
#pragma unroll
      for (int t = 0; t < D; ++t) {
        if (t == d) continue;
        int a0[3] = {ci[0], ci[1], ci[2]}, a1[3] = {ci[0], ci[1], ci[2]};
        int b0[3] = {ci[0], ci[1], ci[2]}, b1[3] = {ci[0], ci[1], ci[2]};
        a0[t] += 1;
        a1[t] -= 1;
        b0[t] += 1;
        b1[t] -= 1;
        b0[d] += 1;
        b1[d] += 1;
        const double pip = wget(P, Wc, P.wPsi, map_cell_dt<d>(P, t, a0[0], a0[1], a0[2]));
        const double pim = wget(P, Wc, P.wPsi, map_cell_dt<d>(P, t, a1[0], a1[1], a1[2]));
        const double pjp = wget(P, Wc, P.wPsi, map_cell_dt<d>(P, t, b0[0], b0[1], b0[2]));
        const double pjm = wget(P, Wc, P.wPsi, map_cell_dt<d>(P, t, b1[0], b1[1], b1[2]));
        g[t] = (pip - pim) + (pjp - pjm);
      }
      const double g2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
      const unsigned long long gb = (unsigned long long)__double_as_longlong(g2),
                               g_lo = (unsigned long long)__double_as_longlong(P.gtol2),
                               g_hi = (unsigned long long)__double_as_longlong(1e300);
      double nd = 0.0;
      if (gb - g_lo < g_hi - g_lo) nd = g[d] * drsqrt(g2);
      else if (gb >= g_hi && g2 >= 1e300) nd = g[d] / sqrt(g2);
      // 1 - tanh^2(x) = sech^2(x) = 4 E / (1 + E)^2, E = exp(-2 |x|), x =
      // psi / (2 eps): no cancellation near the phi_min floor
      const double E = exp(-fabs((0.5 * (psi_i + psi_j)) * P.inv_cdi_eps));
      const double rE = drcp(1.0 + E);
      // (sech^2 - sharp0) / 4
      const double sh = fma(E * rE, rE, -0.25 * P.sharp0);
      const double ahat0 = Gamma * fma(P.cdi_eps_dx, dphi, -sh * nd);
      double Fdi[NV], Rtot = 0.0, hR = 0.0;
#pragma unroll
      for (int ph = 0; ph < 2; ++ph) {
        const bool pi = pres_i[ph], pj = pres_j[ph];
        // the cells' mean, or the value of the one that holds the phase: the
        // half goes into the velocity
        const double ah = pi && pj ? 0.5 * ahat0 : ahat0;
        const double ahat = ph == 0 ? ah : -ah;
        auto keep = [&](double a, double b) { return pi && pj ? a + b : (pi ? a : (pj ? b : 0.0)); };
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          if (P.phase[k] != ph) continue;
          const double R = -keep(wget(P, Wc, P.wYrho + k, ri), wget(P, Wc, P.wYrho + k, rj)) * ahat;
          Fdi[k] = R;
          Rtot += R;
        }
        hR -= keep(wget(P, Wc, P.wHrho + ph, ri), wget(P, Wc, P.wHrho + ph, rj)) * ahat;
      }
      double kb = 0.0;
#pragma unroll
      for (int t = 0; t < D; ++t) {
        const double ui = uget(P, Wc, t, ri);
        const double uj = uget(P, Wc, t, rj);
        kb += ui * uj;
        Fdi[NS + t] = 0.5 * (ui + uj) * Rtot;
      }
      Fdi[NS + D] = 0.5 * kb * Rtot + hR;
      double Ft[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) Ft[v] = Fx[v] + Fdi[v];
      if (P.pos_limiter && !passes(Ft)) {
        fl |= F_CDI_DROPPED;
      } else {
#pragma unroll
        for (int v = 0; v < NV; ++v) Fx[v] = Ft[v];
      }
    }
  }

  // diffusive flux F_nu: species diffusion (Eq. SpeciesMassDiffusion),
  // viscous stress and heat conduction.  It passes the same flux limiter as
  // the regularization flux: added to the admissible flux when both
  // pseudo-updates stay admissible, else not added at this face.
  double Fnu[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) Fnu[v] = 0.0;
  if (P.diffusion) {
    const double rb = 0.5 * (wget(P, Wc, P.wRho, ri) + wget(P, Wc, P.wRho, rj));
    // the face enthalpies cp_k T + b_k P + q_k at the two cells' mean P and T;
    // twice the averages of B and Y, their 1/4 in the common factor
    const double hrb = -0.25 * P.inv_dx * rb;
    double Jc = 0.0, Jb = 0.0, Jq = 0.0;
#pragma unroll
    for (int ph = 0; ph < 2; ++ph) {
      double Yp = 0.0, S = 0.0, Ys[NS], BG[NS];
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        if (P.phase[k] != ph) continue;
        Ys[k] = Yi[k] + Yj[k];
        Yp += Ys[k];
        BG[k] = (wget(P, Wc, P.wB + k, ri) + wget(P, Wc, P.wB + k, rj)) *
                (wget(P, Wc, P.wXr + k, rj) - wget(P, Wc, P.wXr + k, ri));
        S += BG[k];
      }
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        if (P.phase[k] != ph) continue;
        const double J = hrb * (Yp * BG[k] - Ys[k] * S);
        Fnu[k] = J;
        Jc = fma(J, P.cp[k], Jc);
        if (P.has_b) Jb = fma(J, P.b[k], Jb);
        if (P.has_q) Jq = fma(J, P.q[k], Jq);
      }
    }
    double Jh = Jc * (0.5 * (Ti + Tj));
    if (P.has_b) Jh = fma(Jb, 0.5 * (Pi + Pj), Jh);
    if (P.has_q) Jh += Jq;
    Fnu[NS + D] = Jh;
  }

  // viscous stress and heat conduction (Eq. DiffusionTerms), second-order
  // central: face averages of the two cells, normal derivative
  // (q_j - q_i)/dx, a tangential one the mean of the two cells' central
  // differences; the energy row carries -u.tau + q
  if (P.viscous) {
    double gu[3][3];  // gu[i][j] = d u_i / d x_j on the face
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) gu[i][j] = 0.0;
    double ui[3] = {0.0, 0.0, 0.0}, uj[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < D; ++i) {
      ui[i] = uget(P, Wc, i, ri);
      uj[i] = uget(P, Wc, i, rj);
      gu[i][d] = (uj[i] - ui[i]) * P.inv_dx;
    }
#pragma unroll
    for (int t = 0; t < D; ++t) {
      if (t == d) continue;
      int a0[3] = {ci[0], ci[1], ci[2]}, a1[3] = {ci[0], ci[1], ci[2]};
      a0[t] += 1;
      a1[t] -= 1;
      int b0[3] = {a0[0], a0[1], a0[2]}, b1[3] = {a1[0], a1[1], a1[2]};
      b0[d] += 1;
      b1[d] += 1;
      const CRef ip = map_cell_dt<d>(P, t, a0[0], a0[1], a0[2]), im = map_cell_dt<d>(P, t, a1[0], a1[1], a1[2]);
      const CRef jp = map_cell_dt<d>(P, t, b0[0], b0[1], b0[2]), jm = map_cell_dt<d>(P, t, b1[0], b1[1], b1[2]);
#pragma unroll
      for (int i = 0; i < D; ++i) {
        const double dip = uget(P, Wc, i, ip) -
                           uget(P, Wc, i, im);
        const double djp = uget(P, Wc, i, jp) -
                           uget(P, Wc, i, jm);
        gu[i][t] = 0.25 * P.inv_dx * (dip + djp);
      }
    }
    double div = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) div += gu[k][k];
    const double mub = 0.5 * (wget(P, Wc, P.wMu, ri) + wget(P, Wc, P.wMu, rj));
    const double lamb = 0.5 * (wget(P, Wc, P.wLam, ri) + wget(P, Wc, P.wLam, rj));
    double work = 0.0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const double tau = mub * (gu[i][d] + gu[d][i] - (i == d ? (2.0 / 3.0) * div : 0.0));
      Fnu[NS + i] = -tau;
      work += 0.5 * (ui[i] + uj[i]) * tau;
    }
    Fnu[NS + D] -= work + lamb * (Tj - Ti) * P.inv_dx;
  }
  if (P.diffusion || P.viscous) {
    double Ft[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Ft[v] = Fx[v] + Fnu[v];
    if (P.pos_limiter && !passes(Ft)) {
      fl |= F_DIFF_DROPPED;
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) Fx[v] = Ft[v];
    }
  }

#pragma unroll
  for (int v = 0; v < NV; ++v) F[(long long)v * nf + fid] = Fx[v];
  if (stats && fl) {
    if (fl & F_HLLC_FALLBACK) atomicAdd(stats + 1, 1ull);
    if (fl & F_CDI_DROPPED) atomicAdd(stats + 2, 1ull);
    if (fl & (F_THETA_P_L | F_THETA_P_R)) atomicAdd(stats + 3, 1ull);
    if (fl & (F_THETA_T_L | F_THETA_T_R)) atomicAdd(stats + 4, 1ull);
    if (fl & (F_YLIM_L | F_YLIM_R)) atomicAdd(stats + 5, 1ull);
    if (fl & F_DIFF_DROPPED) atomicAdd(stats + 6, 1ull);
  }
}

template <int NS, int D>
void prim(const KParams& P, cudaStream_t s, const double* U, const double* Uin, double* Wc, unsigned long long* red,
          int* status) {
  const int nt = block_threads(P.ncell + P.nextra, CELL_THREADS);
  fast::k_prim<NS, D><<<nblocks(P.ncell + P.nextra, nt), nt, 0, s>>>(P, U, Uin, Wc, red, status);
}

// the forward FP64 face pass of one direction with interpolation RC
template <int NS, int D, int RC>
struct FaceImpl {
  static void face(const KParams& P, cudaStream_t s, int d, const double* Wc, const double* Un, const double* Uk,
                   const double* Uin, const double* scal, double rk0, double rk1, double rk2, double* F,
                   uint32_t* /*flags: the recording kernels'*/, unsigned long long* stats) {
    long long nf = 1;
    for (int e = 0; e < 3; ++e) nf *= (long long)(P.n[e] + (e == d));
    if constexpr (D < 3) {
      // up to two split blocks per SM; with more the redundant X and c cost more
      // than the shorter chain gives (TENO6 faces of 322 x 51 cells: 130 us whole,
      // 274 us split; 5996 cells: 58 whole, 56 split).  3D grids in use have more
      // faces than that (24^3 cells: 14,400); the form is not built for them.
      if (nf <= 2 * 152 * 32) {
        constexpr int nt = 32 * SPLIT_WARPS<NS, D>;
        if (d == 0)
          fast::k_face<NS, D, 0, RC, true><<<nblocks(nf, 32), nt, 0, s>>>(P, Wc, Un, Uk, Uin, scal, rk0, rk1, rk2, F,
                 stats);
        else
          fast::k_face<NS, D, (D > 1 ? 1 : 0), RC, true><<<nblocks(nf, 32), nt, 0, s>>>(P, Wc, Un, Uk, Uin, scal,
                 rk0, rk1, rk2, F, stats);
        return;
      }
    }
    const int nt = block_threads(nf, FACE_THREADS);
    const unsigned nb = nblocks(nf, nt);
    if (d == 0)
      fast::k_face<NS, D, 0, RC><<<nb, nt, 0, s>>>(P, Wc, Un, Uk, Uin, scal, rk0, rk1, rk2, F, stats);
    else if (d == 1)
      fast::k_face<NS, D, (D > 1 ? 1 : 0), RC><<<nb, nt, 0, s>>>(P, Wc, Un, Uk, Uin, scal, rk0, rk1, rk2, F,
                                                                     stats);
    else
      fast::k_face<NS, D, (D > 2 ? 2 : 0), RC><<<nb, nt, 0, s>>>(P, Wc, Un, Uk, Uin, scal, rk0, rk1, rk2, F,
                                                                     stats);
  }
};

// the face pass of interpolation RC for (dimension, species count), or null
template <int RC>
FaceFn face(int dim, int ns) {
  switch (dim * 8 + ns) {
    case 9: return &FaceImpl<1, 1, RC>::face;
    case 10: return &FaceImpl<2, 1, RC>::face;
    case 11: return &FaceImpl<3, 1, RC>::face;
    case 12: return &FaceImpl<4, 1, RC>::face;
    case 17: return &FaceImpl<1, 2, RC>::face;
    case 18: return &FaceImpl<2, 2, RC>::face;
    case 19: return &FaceImpl<3, 2, RC>::face;
    case 20: return &FaceImpl<4, 2, RC>::face;
    case 25: return &FaceImpl<1, 3, RC>::face;
    case 26: return &FaceImpl<2, 3, RC>::face;
    case 27: return &FaceImpl<3, 3, RC>::face;
    case 28: return &FaceImpl<4, 3, RC>::face;
    default: return nullptr;
  }
}

}  // namespace fast
}  // namespace mpmc
