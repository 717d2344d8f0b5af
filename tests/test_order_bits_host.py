"""The ratio test's minima by integer keys (csrc/order_bits.h, compiled for the host) against fmin."""
import os
import shutil
import subprocess

import pytest

from paper_2405_03584_gb300 import build

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include "order_bits.h"
static long long bits(double v) { long long b; std::memcpy(&b, &v, 8); return b; }
static double number(long long b) { double v; std::memcpy(&v, &b, 8); return v; }
int main() {
  const double v[] = {0.0, -0.0, 1e-320, -1e-320, 1e-300, -1e-300, 0.5, -0.5, 1.0, 1.0 + 2.3e-16, -1.0, -2.0, 7e5, 1e308, -1e308,
                      INFINITY, -INFINITY, number(0x7ff8000000000000ll), number((long long)0xfff8000000000000ull),
                      number(0x7fffffffffffffffll), number((long long)0xffffffffffffffffull)};
  const int n = sizeof(v) / sizeof(v[0]);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) {
      long long m = ipmk::kInfBits;
      for (double q : {v[i], v[j]}) {
        const long long k = ipmk::min_key(bits(q));
        if (k < m) m = k;
      }
      const double got = number(ipmk::min_key_bits(m)), want = std::fmin(std::fmin(INFINITY, v[i]), v[j]);
      if (!(got == want)) {
        std::printf("%g (%llx), %g (%llx): %g, not %g\n", v[i], (unsigned long long)bits(v[i]), v[j], (unsigned long long)bits(v[j]), got, want);
        return 1;
      }
    }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_minima_are_fmins(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    r = subprocess.run([shutil.which("g++"), "-std=c++17", "-O2", "-I" + build.CSRC, str(tmp_path / "t.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
