"""Host check of the face average's X and c and of the face sound speed
(csrc/mpmc_avg.h), compiled with the host compiler, against extended precision
(x87 or quad long double), with the FP64 form of the average beside them.

Reference of the average: p and T that hold the two cells' volume and energy
(with the kinetic energy that the average loses), by Newton steps on the energy
residual with T eliminated through the volume; then X and c by Eq. SpeedOfSound
and Appendix A.  FP64 form: the equilibrium of the averaged conserved vector in
double, as face_avg_fp64 takes it.  States: pure and mixed cells, traces down to
1e-14, jumps from rounding to a strong shock's, for gases with one liquid, two
liquids and a NASG liquid.

Bounds, relative, per class of states: a float-float operation is within 2^-46
of its result, the average and its sums chain at most thirty of them: 2^-41 of X
and c, or the FP64 form's own largest error where that is more (traces of gas in
a liquid: their share of the compressibility hangs on P, a small difference of
the liquid's energies).  Sound speed: twenty operations, 2^-41.  ff_sqrt: one
correction, 2^-44.  What leaves 2^-60 .. 2^60 is refused with nothing written."""
import os
import shutil
import subprocess

import pytest

HDR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_14063_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>
#include "mpmc_avg.h"
typedef long double R;
using mpmc::ff;
struct Sp { double cv, gam, q, b, pinf; };
static ff split(double x) { ff r; r.h = (float)x; r.l = (float)(x - (double)r.h); return r; }
template <class S> static S Rk(const Sp& s) { return (S)((s.gam - 1.0) * s.cv); }
// X and c at (p, T) for the partial densities M
template <class S, int NS>
static void xc(const Sp* sp, const S* M, S p, S T, S& X, S& c) {
  S cp = 0, s1 = 0, s2 = 0, m = 0;
  for (int k = 0; k < NS; ++k) {
    if (M[k] == 0) continue;
    const S r = 1 / (p + (S)sp[k].pinf);
    cp += (S)(sp[k].gam * sp[k].cv) * M[k];
    s1 += Rk<S>(sp[k]) * M[k] * r;
    s2 += Rk<S>(sp[k]) * M[k] * r * r;
    m += M[k];
  }
  X = T * s1 / cp;
  c = std::sqrt(cp * m / (T * (s2 * cp - s1 * s1)));
}
// p, T of total volume V and energy E (less reference) of the masses M
template <class S, int NS>
static void solve(const Sp* sp, const S* M, S V, S E, S p0, S& p, S& T) {
  S lo = -1e300, hi = std::numeric_limits<S>::infinity(), Cv = 0;
  for (int k = 0; k < NS; ++k)
    if (M[k] > 0) {
      Cv += (S)sp[k].cv * M[k];
      if (-(S)sp[k].pinf > lo) lo = -(S)sp[k].pinf;
    }
  S x = p0 > lo ? p0 : lo + 1;
  for (int it = 0; it < 400; ++it) {
    // V (Cv / s + g / s) - E, s = sum M R / (x + Pinf), g = sum M R Pinf / (x + Pinf)
    S s = 0, ds = 0, g = 0, dg = 0;
    for (int k = 0; k < NS; ++k) {
      if (!(M[k] > 0)) continue;
      const S r = 1 / (x + (S)sp[k].pinf), t = M[k] * Rk<S>(sp[k]) * r;
      s += t;
      ds -= t * r;
      g += t * (S)sp[k].pinf;
      dg -= t * r * (S)sp[k].pinf;
    }
    const S f = V * (Cv + g) / s - E, df = V * (dg * s - (Cv + g) * ds) / (s * s);
    (f > 0 ? hi : lo) = x;
    S xn = x - f / df;
    if (!(xn > lo && xn < hi)) xn = std::isinf((double)hi) ? 2 * x + 1 : (lo + hi) / 2;
    T = V / s;
    const bool done = xn == x || it == 399;
    x = xn;
    if (done) break;
  }
  S s = 0;
  for (int k = 0; k < NS; ++k)
    if (M[k] > 0) s += M[k] * Rk<S>(sp[k]) / (x + (S)sp[k].pinf);
  p = x;
  T = V / s;
}
template <int NS>
static void run(const char* name, const Sp* sp, long& bad) {
  mpmc::SpeciesFF sf[NS];
  for (int k = 0; k < NS; ++k)
    sf[k] = {split((sp[k].gam - 1.0) * sp[k].cv), split(sp[k].cv), split(sp[k].gam * sp[k].cv), split(sp[k].pinf),
             split(sp[k].q), split(sp[k].b)};
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> ud(0, 1);
  std::normal_distribution<double> nd(0, 1);
  for (int comp = 0; comp < 3; ++comp)      // pure, mixed, traces
    for (int jump = 0; jump < 4; ++jump) {  // rounding, weak, strong, shock
      double eX = 0, ec = 0, fX = 0, fc = 0, ea = 0;
      long refused = 0, n = 4000;
      for (int it = 0; it < n; ++it) {
        double m[2][NS], P[2], T[2], u[2][3];
        const double P0 = std::pow(10, 4 + 3 * ud(g)), T0 = 250 + 500 * ud(g);
        const double amp = jump == 0 ? 1e-15 : (jump == 1 ? 1e-4 : (jump == 2 ? 0.3 : 1.0));
        const int main = (int)(NS * ud(g)) % NS;
        for (int s = 0; s < 2; ++s) {
          P[s] = P0 * (1 + amp * (jump == 3 ? 8 * ud(g) : nd(g) * 0.5));
          if (!(P[s] > 100)) P[s] = 100;
          T[s] = T0 * (1 + 0.5 * amp * (jump == 3 ? 2 * ud(g) : nd(g)));
          if (!(T[s] > 50)) T[s] = 50;
          for (int d = 0; d < 3; ++d) u[s][d] = 300 * amp * nd(g);
          double al[NS], sum = 0;
          for (int k = 0; k < NS; ++k) {
            al[k] = comp == 0 ? (k == main ? 1.0 : 0.0)
                              : (comp == 1 ? 0.02 + ud(g) : (k == main ? 1.0 : std::pow(10, -14 * ud(g))));
            sum += al[k];
          }
          for (int k = 0; k < NS; ++k) m[s][k] = al[k] / sum / (Rk<double>(sp[k]) * T[s] / (P[s] + sp[k].pinf) + sp[k].b);
        }
        double X = 0, c = 0, ic = 0;
        if (!mpmc::face_avg_ff<NS, 3>(sf, m[0], m[1], P[0], P[1], T[0], T[1], u[0], u[1], X, c, ic)) { ++refused; continue; }
        // reference, and the FP64 form from stored (FP64) conserved vectors
        R M[NS], V = 0, E = 0, rho[2] = {0, 0}, du2 = 0, pr, Tr, Xr, cr;
        double U[NS], Ec[2], mom[3] = {0, 0, 0}, Ea, rh = 0, q = 0, b = 0;
        for (int k = 0; k < NS; ++k) M[k] = 0;
        for (int s = 0; s < 2; ++s) {
          double e = 0, rs = 0;
          for (int k = 0; k < NS; ++k) {
            const R r = (R)m[s][k] / ((R)P[s] + sp[k].pinf);
            M[k] += m[s][k];
            rho[s] += m[s][k];
            V += r * Rk<R>(sp[k]) * T[s];
            E += (R)sp[k].cv * m[s][k] * T[s] + r * Rk<R>(sp[k]) * T[s] * sp[k].pinf;
            rs += m[s][k];
            e += m[s][k] * (sp[k].cv * T[s] * (P[s] + sp[k].gam * sp[k].pinf) / (P[s] + sp[k].pinf) + sp[k].q);
          }
          double ke = 0;
          for (int d = 0; d < 3; ++d) { ke += u[s][d] * u[s][d]; mom[d] += 0.5 * (rs * u[s][d]); }
          Ec[s] = e + 0.5 * rs * ke;
        }
        for (int d = 0; d < 3; ++d) du2 += ((R)u[1][d] - u[0][d]) * ((R)u[1][d] - u[0][d]);
        E += du2 * rho[0] * rho[1] / (2 * (rho[0] + rho[1]));
        solve<R, NS>(sp, M, V, E, (R)(0.5 * (P[0] + P[1])), pr, Tr);
        xc<R, NS>(sp, M, pr, Tr, Xr, cr);
        for (int k = 0; k < NS; ++k) { U[k] = 0.5 * (m[0][k] + m[1][k]); rh += U[k]; q += U[k] * sp[k].q; b += U[k] * sp[k].b; }
        Ea = 0.5 * (Ec[0] + Ec[1]);
        for (int d = 0; d < 3; ++d) Ea -= 0.5 * mom[d] * mom[d] / rh;
        double pd, Td, Xd, cd;
        solve<double, NS>(sp, U, 1.0 - b, Ea - q, 0.5 * (P[0] + P[1]), pd, Td);
        xc<double, NS>(sp, U, pd, Td, Xd, cd);
        eX = std::fmax(eX, std::fabs((double)((X - Xr) / Xr)));
        ec = std::fmax(ec, std::fabs((double)((c - cr) / cr)));
        fX = std::fmax(fX, std::fabs((double)((Xd - Xr) / Xr)));
        fc = std::fmax(fc, std::fabs((double)((cd - cr) / cr)));
        if (std::fabs((double)((R)c * ic - 1)) > 3e-16) ++bad;
        // sound speed of the left cell
        double Y[NS], a = 0, v = 0;
        R cp = 0, s1 = 0, s2 = 0;
        for (int k = 0; k < NS; ++k) v += m[0][k];
        v = 1 / v;
        for (int k = 0; k < NS; ++k) {
          Y[k] = m[0][k] * v;
          const R r = 1 / ((R)P[0] + sp[k].pinf), z = Y[k] == 0 ? 0 : (R)Y[k] * Rk<R>(sp[k]) * r;
          cp += (R)Y[k] * (sp[k].gam * sp[k].cv);
          s1 += z;
          s2 += z * r;
        }
        if (!mpmc::sound_speed_ff<NS>(sf, Y, P[0], T[0], v, a)) { ++refused; continue; }
        const R ar = (R)v * std::sqrt(cp / (T[0] * (cp * s2 - s1 * s1)));
        ea = std::fmax(ea, std::fabs((double)((a - ar) / ar)));
      }
      const double lim = 0x1p-41;
      const bool ok = refused * 20 <= n && eX <= std::fmax(lim, fX) && ec <= std::fmax(lim, fc) && ea <= lim;
      std::printf("%-5s composition %d jump %d: X %.1e (FP64 form %.1e) c %.1e (%.1e) a %.1e, %ld refused%s\n", name,
                  comp, jump, eX, fX, ec, fc, ea, refused, ok ? "" : "  BAD");
      if (!ok) ++bad;
    }
}
int main() {
  long bad = 0;
  const Sp air{717.9, 1.4, 0, 0, 0}, he{3102.0, 1.67, 0, 0, 0}, sg{1.8e3, 4.4, 0, 0, 6e8}, lb{1.077e3, 2.35, 0, 0, 4e8},
      wat{4.185e3 / 1.0123, 1.0123, -1.143e6, 9.203e-4, 1.835e8};
  const Sp a[3] = {air, he, sg}, b[4] = {sg, lb, air, he}, c[2] = {wat, air};
  run<3>("one", a, bad);
  run<4>("two", b, bad);
  run<2>("nasg", c, bad);
  double es = 0;
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> ud(-80, 80);
  for (int i = 0; i < 200000; ++i) {
    const double x = std::exp2(ud(g));
    const ff s = mpmc::ff_sqrt(split(x));
    es = std::fmax(es, std::fabs((double)(((R)s.h + s.l) / std::sqrt((R)split(x).h + split(x).l) - 1)));
  }
  std::printf("ff_sqrt %.1e\n", es);
  if (es > 0x1p-44) ++bad;
  // refusals, nothing written
  mpmc::SpeciesFF sf[1] = {{split(287.0), split(717.5), split(1004.5), split(0.0), split(0.0), split(0.0)}};
  const double u0[3] = {0, 0, 0}, inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  for (double v : {1e30, 1e-30, inf, nan, -1e5, 0.0})
    for (int w = 0; w < 3; ++w) {
      double m[1] = {w == 0 ? v : 1.2}, P = w == 1 ? v : 1e5, T = w == 2 ? v : 300, X = 7, c = 7, ic = 7, a = 7, Y[1] = {1.0};
      if (mpmc::face_avg_ff<1, 3>(sf, m, m, P, P, T, T, u0, u0, X, c, ic) || X != 7 || c != 7 || ic != 7) {
        std::printf("average not refused: %g in place %d\n", v, w);
        ++bad;
      }
      if (w > 0 && !(v < 0) && (mpmc::sound_speed_ff<1>(sf, Y, P, T, 0.8, a) || a != 7)) {
        std::printf("sound speed not refused: %g in place %d\n", v, w);
        ++bad;
      }
    }
  return bad != 0;
}
"""


def test_face_average_and_sound_speed_against_extended_precision(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "a.cpp", tmp_path / "a"
    src.write_text(SRC)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I", HDR, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
