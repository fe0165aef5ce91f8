"""The FP64 Jacobi rotation (csrc/jacobi_rotation.h), compiled for the host and
compared with about 100 bits over pivots of every size, its FP32 starting values off
by up to 1e-6 more.  The plain formula's roundings, each at most 2^-53, bound the tangent
by 2^-50; the refined one, whose last step leaves the rounding of its residual and of
its result, is held to half of that, and so is the cosine."""
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
#include "jacobi_rotation.h"

// double-double, enough for a reference of 1e-30
struct DD { double h, l; };
static DD two_sum(double a, double b) { double s = a + b, v = s - a; return {s, (a - (s - v)) + (b - v)}; }
static DD add(DD a, DD b) { DD s = two_sum(a.h, b.h); s.l += a.l + b.l; return two_sum(s.h, s.l); }
static DD mul(DD a, DD b) { double p = a.h * b.h, e = std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h); return two_sum(p, e); }
static DD neg(DD a) { return {-a.h, -a.l}; }
static DD dvd(DD a, DD b) {
  double q = a.h / b.h;
  DD r = add(a, neg(mul({q, 0}, b)));
  double q2 = r.h / b.h;
  r = add(r, neg(mul({q2, 0}, b)));
  return add(two_sum(q, q2), {r.h / b.h, 0});
}
static DD root(DD a) {
  double s = std::sqrt(a.h);
  DD r = add(a, neg(mul({s, 0}, {s, 0})));
  DD t = two_sum(s, r.h / (2 * s));
  r = add(a, neg(mul(t, t)));
  return add(t, {r.h / (2 * s), 0});
}
int main() {
  std::mt19937_64 g(1);
  std::normal_distribution<double> N(0, 1);
  std::uniform_real_distribution<double> U(-1, 1);
  double et = 0, ec = 0, ft = 0, fc = 0;
  // conversions: exact to FP32 where it is normal, out of range beyond
  for (int i = 0; i < 200000; ++i) {
    const double x = N(g) * std::pow(10.0, 36 * U(g));
    const float f = geneo::jacobi_f32(x);
    if (std::fabs(x) >= 0x1p-126 && !(std::fabs((double)f - x) <= 0x1p-23 * std::fabs(x))) et = 1;
    if (geneo::jacobi_f64(f) != (double)f) et = 1;
  }
  for (double x : {1e39, -1e300, HUGE_VAL, std::nan("")})
    if (geneo::jacobi_in_range(0.f, geneo::jacobi_f32_inf(x))) et = 1;
  for (double x : {0.0, -0.0, 1e-39, 5e-324})
    if (geneo::jacobi_f32(x) != 0.f) et = 1;
  for (int i = 0; i < 1000000; ++i) {
    const double apq = N(g) * std::pow(10.0, -4 + 19 * U(g));
    double dd = N(g) * std::pow(10.0, 20 * U(g));
    if (i % 5 == 0) dd = apq * N(g);
    if (i % 97 == 0) dd = 0.0;
    const float af = geneo::jacobi_f32_inf(apq), df = geneo::jacobi_f32_inf(dd), theta = df / (2.f * af);
    if (!geneo::jacobi_in_range(theta, af)) continue;
    const DD th = dvd({dd, 0}, {2 * apq, 0});
    const DD ab = th.h < 0 ? neg(th) : th;
    DD t = dvd({th.h >= 0 ? 1.0 : -1.0, 0}, add(ab, root(add(mul(ab, ab), {1, 0}))));
    DD c = dvd({1, 0}, root(add(mul(t, t), {1, 0})));
    auto err = [](double x, DD v) { return std::fabs(((x - v.h) - v.l) / v.h); };
    // starting values as the device's approximate operations may leave them
    auto off = [&]() { return (float)(1.0 + 1e-6 * U(g)); };
    const float ta = std::fabs(theta);
    const float t0 = (theta >= 0.f ? 1.f : -1.f) / (ta < 1e9f ? ta + std::sqrt(ta * ta + 1.f) : 2.f * ta) * off();
    double tt, cc;
    geneo::jacobi_refine(dd, apq, t0, 1.f / std::sqrt(1.f + t0 * t0) * off(), 1.f / (2.f * af * t0 + df) * off(), tt, cc);
    et = std::max(et, err(tt, t));
    ec = std::max(ec, err(cc, c));
    const double p = geneo::jacobi_tangent_formula(dd, apq);
    ft = std::max(ft, err(p, t));
    fc = std::max(fc, err(1.0 / std::sqrt(p * p + 1.0), c));
  }
  std::printf("%.17g %.17g %.17g %.17g\n", et, ec, ft, fc);
}
"""


def test_rotation_to_fp64_rounding(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs a host C++ compiler")
    src = tmp_path / "rotation.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "rotation")
    subprocess.run([gxx, "-O1", "-std=c++17", "-ffp-contract=off", "-I" + CSRC, str(src), "-o", exe], check=True)
    et, ec, ft, fc = map(float, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert max(ft, fc) <= 2.0 ** -50
    assert max(et, ec) <= 2.0 ** -51, (et, ec, ft, fc)
