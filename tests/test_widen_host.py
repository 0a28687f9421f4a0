"""Host check of the FP32 -> FP64 widening of the mixed path's flux sums
(csrc/mpmc_narrow.h): bit for bit the C conversion for normal numbers and
zeros, and `widens` true for exactly those."""
import os
import shutil
import subprocess

import pytest

HDR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_14063_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include "mpmc_narrow.h"
int main() {
  unsigned long long bad = 0, n = 0;
  for (uint64_t i = 0; i < (1ull << 32); i += (i & 0x7fffffu) < 8 || (i & 0x7fffffu) > 0x7ffff0u ? 1 : 7919) {
    const uint32_t b = (uint32_t)i;
    float f;
    std::memcpy(&f, &b, 4);
    const bool ok = std::isnormal(f) || f == 0.f;
    ++n;
    if (mpmc::widens(f) != ok) ++bad;
    if (!ok) continue;
    const double a = mpmc::widen(f), c = (double)f;
    if (std::memcmp(&a, &c, 8)) ++bad;
  }
  std::printf("%llu of %llu differ\n", bad, n);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_widen_is_the_conversion(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", HDR, str(tmp_path / "t.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
