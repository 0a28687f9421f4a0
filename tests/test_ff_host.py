"""Host check of the float-float interpolations of the forward FP64 face pass
(csrc/mpmc_ff.h: WENO5-Z, WENO5-JS, TENO5, TENO6), compiled with the host
compiler and compared with the same interpolations in extended precision (x87
or quad long double) on both sides of a face.  Stencils whose TENO selection
is within 1e-9 of the cut are left out (either answer is right there).

Bound, per value: 4 ulp of FP64 of the stencil's largest value (three FP64
roundings of terms no larger than it, plus the differences') + 2^-40 of its
largest difference (the correction's chain of about ten float-float
operations, each within 2^-45, times weights that sum to one, times candidate
differences of at most 8/3 of it) + 1e-35 (the scaled underflow floor)."""
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
#include "mpmc_ff.h"
typedef long double R;
static R sq(R x) { return x * x; }
// v: six cells; tie: a TENO candidate is too close to the cut
template <int KIND>
static R side(const double* v, double eps, bool& tie) {
  const R d0 = (R)v[1] - v[0], d1 = (R)v[2] - v[1], d2 = (R)v[3] - v[2], d3 = (R)v[4] - v[3], d4 = (R)v[5] - v[4];
  R c[4] = {5 * d1 - 2 * d0, d1 + 2 * d2, 4 * d2 - d3, (9 * d2 - 4 * d3 + d4) / 2};
  const R t[3] = {d1 - d0, d2 - d1, d3 - d2}, s[3] = {3 * d1 - d0, d1 + d2, d3 - 3 * d2};
  R b[4] = {0, 0, 0, 0}, a[4] = {0, 0, 0, 0}, n = 0, w = 0;
  for (int k = 0; k < 3; ++k) b[k] = R(13) / 12 * t[k] * t[k] + s[k] * s[k] / 4;
  const R z = fabsl(b[0] - b[2]), g[4] = {1, 6, 3, 0};
  if (KIND == 0)
    for (int k = 0; k < 3; ++k) a[k] = g[k] * (1 + z / (b[k] + (R)eps));
  if (KIND == 1)
    for (int k = 0; k < 3; ++k) a[k] = g[k] / sq(1e-6L + b[k]);
  if (KIND >= 2) {
    const int K = KIND == 2 ? 3 : 4;
    R tau = z;
    if (KIND == 3) {
      const R e0 = -d0 - d1, e1 = -d1, e3 = d2, e4 = d2 + d3, e5 = d2 + d3 + d4;
      b[3] = sq(18 * e3 - 9 * e4 + 2 * e5) / 36 + R(13) / 12 * sq(-5 * e3 + 4 * e4 - e5) +
             R(781) / 720 * sq(3 * e3 - 3 * e4 + e5);
      const R b6 = sq(3 * e0 - 30 * e1 + 60 * e3 - 15 * e4 + 2 * e5) / 3600 +
                   sq(-11 * e0 + 174 * e1 + 174 * e3 - 11 * e4) / 15600 +
                   sq(-16315 * e0 - 16831 * e1 - 230474 * e3 + 115237 * e4 - 16487 * e5) / 3967729920.0L +
                   R(1421461) / 1310400 * sq(e0 - 4 * e1 - 4 * e3 + e4) +
                   R(21520059541.0L) / 19838649600.0L * sq(-e0 + 5 * e1 + 10 * e3 - 5 * e4 + e5);
      tau = fabsl(b6 - (b[0] + b[2] + 4 * b[1]) / 6);
    }
    R r[4], m = 0, gs = 0;
    for (int k = 0; k < K; ++k) m = fmaxl(m, r[k] = 1 + tau / (b[k] + 1e-40L));
    for (int k = 0; k < K; ++k) gs += (r[k] = sq(r[k] / m) * sq(r[k] / m) * sq(r[k] / m));
    const R ct = (KIND == 2 ? 1e-5L : 1e-7L) * gs, d5[4] = {1, 6, 3, 0}, d6[4] = {1, 9, 6, 4};
    for (int k = 0; k < K; ++k) {
      if (fabsl(r[k] / ct - 1) < 1e-9L) tie = true;
      if (!(r[k] < ct)) a[k] = KIND == 2 ? d5[k] : d6[k];
    }
  }
  for (int k = 0; k < 4; ++k) {
    n += a[k] * c[k];
    w += a[k];
  }
  return v[2] + n / (6 * w);
}
static mpmc::WenoEps split(double eps) {
  mpmc::WenoEps e;
  int k;
  const double f = 2.0 * std::frexp(4.0 * eps, &k);
  e.h = (float)f;
  e.l = (float)(f - (double)e.h);
  e.e = k - 1;
  return e;
}
template <int KIND>
static double run(long& bad, long& cases) {
  std::mt19937_64 g(7);
  std::normal_distribution<double> nd(0, 1);
  std::uniform_real_distribution<double> ud(0, 1);
  double worst = 0;
  const double epss[] = {1e-40, 1e-6, 1e-12, 1.0};
  for (int kind = 0; kind < 8; ++kind)
    for (int it = 0; it < 60000; ++it) {
      double v[6];
      const double a = nd(g), b = nd(g), ph = ud(g), sc = kind == 6 ? std::exp2(600 * (ud(g) - 0.5)) : 1e5;
      for (int j = 0; j < 6; ++j) {
        const double x = j - 2;
        if (kind == 0) v[j] = sc * (1 + 1e-3 * (a * std::sin(.3 * x + 6 * ph) + b * std::cos(.5 * x)));
        if (kind == 1) v[j] = sc * (1 + .3 * a * std::sin(.7 * x + 6 * ph));
        if (kind == 2) v[j] = 0.5 * (1 + std::tanh((x + 4 * (ph - .5)) * .5));
        if (kind == 3) v[j] = (x + 3 * (ph - .5) > 0 ? 1 : 2.4) * (1 + 1e-2 * nd(g));
        if (kind == 4) v[j] = 1e-8 + 0.5 * (1 + std::tanh((x + 30 * (ph - .5)) * .5));
        if (kind == 5) v[j] = sc * (1 + 1e-15 * nd(g));
        if (kind == 6) v[j] = sc * nd(g);
        if (kind == 7) v[j] = (it >> j) & 1 ? a : (it & 64 ? a : 0.0);   // steps and flats
      }
      const double eps = epss[it & 3];
      double L = 0, Rv = 0, m = 0, d = 0;
      const mpmc::WenoEps e4 = KIND == 0 ? split(eps) : (KIND == 1 ? mpmc::js_eps4(0) : mpmc::teno_eps4(0));
      if (!mpmc::eno_lr_ff<KIND>(v, e4, L, Rv)) { ++bad; continue; }
      const double w[6] = {v[5], v[4], v[3], v[2], v[1], v[0]};
      bool tie = false;
      const R rl = side<KIND>(v, eps, tie), rr = side<KIND>(w, eps, tie);
      if (tie) continue;
      for (int j = 0; j < 6; ++j) {
        m = std::fmax(m, std::fabs(v[j]));
        if (j) d = std::fmax(d, std::fabs(v[j] - v[j - 1]));
      }
      const double tol = std::ldexp(m, -51) + std::ldexp(d, -40) + 1e-35;
      const double e = std::fmax(std::fabs((double)(L - rl)), std::fabs((double)(Rv - rr)));
      worst = std::fmax(worst, e / tol);
      ++cases;
    }
  return worst;
}
int main() {
  long bad = 0, cases = 0;
  const double worst = std::fmax(std::fmax(run<0>(bad, cases), run<1>(bad, cases)),
                                 std::fmax(run<2>(bad, cases), run<3>(bad, cases)));
  // uniform stencils come back exactly, whatever their size
  for (double c : {0.0, 1.0, -3e300, 1e-310, 1e5}) {
    double v[6] = {c, c, c, c, c, c}, L = 9, Rv = 9;
    if (!mpmc::eno_lr_ff<0>(v, split(1e-40), L, Rv) || L != c || Rv != c) ++bad;
  }
  // stencils that the caller has to take in FP64
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  for (double c : {inf, -inf, nan, 1e300})
    for (int j = 0; j < 6; ++j) {
      double v[6] = {1, 2, 3, 4, 5, 6}, L = 9, Rv = 9;
      v[j] = c;
      if (mpmc::eno_lr_ff<0>(v, split(1e-40), L, Rv) || L != 9 || Rv != 9) ++bad;
    }
  std::printf("%ld cases, worst %.3g of the bound, %ld bad\n", cases, worst, bad);
  return worst <= 1.0 && bad == 0 ? 0 : 1;
}
"""


def test_float_float_interpolations_against_extended_precision(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(SRC)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", HDR, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
