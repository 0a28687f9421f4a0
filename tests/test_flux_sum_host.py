"""Host check of the mixed path's flux-difference sums (csrc/mpmc_ff.h,
ff_diff_sum), compiled with the host compiler and compared with the exact sums
(x87 or quad long double holds them but for a 2^-63 part, which the bound
allows for).

Bound, per sum: one FP64 rounding of it, 2^-53 |sum|, + 2^-61 of the sum of
the differences' magnitudes M.  (What the high parts' sum leaves is below
6 x 2^-24 x 3 M < 2^-19 M; the pair that holds it rounds its low part, at most
2^-24 of that, in up to four FP32 additions: 4 x 2^-24 x 2^-43 M = 2^-65 M;
its FP64 conversion rounds to 2^-72 M; long double's own sums to 2^-61 M.)
That is below the FP64 form's 2^-53 of every partial sum, which conservation
of the mixed path to FP64 rounding rests on."""
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
template <int D>
static double run(long& bad) {
  std::mt19937_64 g(11);
  std::normal_distribution<double> nd(0, 1);
  std::uniform_real_distribution<double> ud(0, 1);
  double worst = 0;
  for (int it = 0; it < 400000; ++it) {
    float a[D], b[D];
    const double s = std::exp(40 * (ud(g) - 0.5));   // fluxes of 2e-9 .. 5e8
    for (int d = 0; d < D; ++d) {
      const double m = s * nd(g) * (it & 1 ? 1.0 : std::exp(20 * (ud(g) - 0.5)));
      a[d] = (float)m;
      b[d] = (float)(it & 2 ? s * nd(g) : m * (1 + std::exp(-16 * ud(g)) * nd(g)));
      if (it % 7 == 0 && d) { a[d] = b[0]; b[d] = a[0]; }   // cancelling directions
    }
    bool ok = true;
    const double f = mpmc::ff_diff_sum<D>(a, b, ok);
    if (!ok) { ++bad; continue; }
    R x = 0, M = 0;
    for (int d = 0; d < D; ++d) {
      x += (R)a[d] - (R)b[d];
      M += std::fabs((double)a[d] - (double)b[d]);
    }
    const double e = (double)fabsl((R)f - x), tol = std::ldexp((double)fabsl(x), -53) + (double)(M * 0x1p-61L);
    if (tol == 0 ? e != 0 : e > tol) ++bad;
    if (tol > 0) worst = std::fmax(worst, e / tol);
  }
  // what the caller has to take in FP64
  const float big = std::numeric_limits<float>::max(), inf = std::numeric_limits<float>::infinity();
  for (float c : {inf, -inf, std::numeric_limits<float>::quiet_NaN(), big, 1e-40f}) {
    float a[D], b[D];
    for (int d = 0; d < D; ++d) a[d] = b[d] = 1.f;
    a[D - 1] = c;
    b[D - 1] = c == big ? -big : (c == 1e-40f ? 0.f : 1.f);
    bool ok = true;
    mpmc::ff_diff_sum<D>(a, b, ok);
    if (ok) ++bad;
  }
  return worst;
}
int main() {
  long bad = 0;
  const double w1 = run<1>(bad), w2 = run<2>(bad), w3 = run<3>(bad);
  std::printf("worst %.3g %.3g %.3g of the bound, %ld bad\n", w1, w2, w3, bad);
  return bad != 0;
}
"""


def test_flux_difference_sums_round_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "s.cpp", tmp_path / "s"
    src.write_text(SRC)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", HDR, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
