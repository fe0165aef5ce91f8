"""Pivots of the FP64 panels (csrc/pivot.h), compiled for the host: the root and the
quotients are no further off than a square root (2^-53) and a division by it (2^-52),
the reciprocal square root being off by up to an ulp."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_10944_gb300", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include "pivot.h"
using std::fma;
int main() {
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(0, 1);
  double worst_d = 0, worst_q = 0;
  for (int i = 0; i < 1000000; ++i) {
    const double p = 1 + 3 * U(g), a = 1 + U(g);
    double r = 1.0 / std::sqrt(p);
    if (i % 3 == 0) r = std::nextafter(r, 2.0);
    if (i % 3 == 1) r = std::nextafter(r, 0.0);
    const double d = geneo::pivot_root(p, r), q = geneo::pivot_quotient(a, d, r);
    // relative error of d: (d^2 - p) / (2 p); of q: q s - a over a with s = sqrt(p) = d - ed d
    const double ed = fma(d, d, -p) / (2 * p);
    const double eq = fma(q, d, -a) / a - ed;
    worst_d = std::max(worst_d, std::fabs(ed));
    worst_q = std::max(worst_q, std::fabs(eq));
  }
  std::printf("%.17g %.17g\n", worst_d * 0x1p53, worst_q * 0x1p53);
}
"""


def test_root_and_quotient_round_as_square_root_and_division(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs a host C++ compiler")
    src = tmp_path / "pivot.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "pivot")
    subprocess.run([gxx, "-O1", "-std=c++17", "-ffp-contract=off", "-I" + CSRC, str(src), "-o", exe], check=True)
    d, q = map(float, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert d <= 1.0 and q <= 2.0, (d, q)
