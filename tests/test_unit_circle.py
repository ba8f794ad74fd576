"""The constants of the transforms in registers (csrc/unit_circle.cuh) against long
double: every cosine and sine is the nearest double (0.5 units of the last place and
what long double itself may be off)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_04989_gb300", "csrc")

CODE = r"""
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include "unit_circle.cuh"
int main() {
  const long double tau = 2 * 3.14159265358979323846264338327950288L;
  double worst = 0;
  int axes = 0;
  for (long n : {2, 4, 8, 16, 32, 64, 128, 256})
    for (long p = 0; p < n; ++p)
      for (int q = 0; q < 2; ++q) {
        const long double want = q ? sinl(tau * p / n) : cosl(tau * p / n);
        const double got = q ? tsvd::ct::sin2pi(p, n) : tsvd::ct::cos2pi(p, n);
        if (fabsl(want) < 1e-17L) { axes += got != 0.0; continue; }
        worst = fmax(worst, (double)fabsl(got - want) / ldexp(1.0, std::ilogb((double)want) - 52));
      }
  printf("%d %.6f", axes, worst);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_nearest_doubles(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(CODE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    axes, worst = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert int(axes) == 0
    assert float(worst) <= 0.5 + 2.0 ** -8, worst
