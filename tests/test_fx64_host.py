"""The fixed-point 2^x / log2 functions of csrc/fx64.cuh, compiled for the host (their arithmetic is the device's, bit
for bit): accuracy against extended precision over the potential's ranges and far beyond, and what they refuse."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1909_11474_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __host__
#define __device__
#define __forceinline__ inline
#include "fx64.cuh"
using namespace tsf;
#include "fx64_tables.inc"
typedef long double Q;
int main() {
  const FxTables &t = kFxTables;
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(0, 1);
  double worst[2][3] = {{0, 0, 0}, {0, 0, 0}};
  int refused[2] = {0, 0};
  for (int i = 0; i < 400000; ++i) {
    const int wide = i & 1;
    double D0 = 3.2 * (0.7 + 0.6 * U(g)), al = 1.43 * (0.7 + 0.6 * U(g)), r0 = 2.238 * (0.7 + 0.6 * U(g));
    double be = 0.28 * (0.7 + 0.6 * U(g)), n = 0.6 * (0.7 + 0.6 * U(g)), r = 1.9 + 1.3 * U(g), S = 0.001 + 2 * U(g);
    if (wide) {
      D0 = std::exp((U(g) - 0.5) * 60); al = 4 * U(g); be = std::exp((U(g) - 0.5) * 40); n = 0.02 + 3.9 * U(g);
      r = 0.2 + 6 * U(g); S = std::exp((U(g) - 0.7) * 60);
    }
    if (i % 17 == 0) S = 0;
    if (i % 19 == 0) S = std::ldexp(1.0 + (i % 5 - 2) * 0x1p-52, i % 7 - 3);   // beside powers of two
    if (i % 23 == 0) r = r0;
    const double k = -al * 1.4426950408889634, in = -0.5 / n;
    double fR, bh, cc;
    if (!fx_bond(r, S, fx_lane(r0, k, 2 * k, D0, D0, be, n, in, t), t, fR, bh, cc)) { ++refused[wide]; continue; }
    const Q x = std::exp2((Q)k * ((Q)r - (Q)r0)), hA = D0 * x;
    Q z = (Q)be * (Q)S;
    if (z < (Q)1e-30) z = 1e-30;
    const Q zn = std::pow(z, (Q)n), b = std::pow(1 + zn, (Q)in);
    const Q ref[3] = {hA * x, b * hA, (Q)be * b * hA * zn / (2 * z * (1 + zn))};
    const double got[3] = {fR, bh, cc};
    for (int q = 0; q < 3; ++q) {
      const double e = (double)std::fabs((got[q] - ref[q]) / ref[q]);
      if (!(e <= worst[wide][q])) worst[wide][q] = e;
    }
  }
  const double inf = INFINITY, nan = NAN;
  double a, b, c;
  const FxLane ok = fx_lane(2.2, -2.0, -4.0, 3.2, 3.2, 0.28, 0.6, -0.5 / 0.6, t);
  int bad = !ok.ok;
  for (double r : {16.0, 1e300, inf, nan, -inf}) bad += fx_bond(r, 1.0, ok, t, a, b, c);
  for (double S : {inf, nan, 1e80}) bad += fx_bond(2.3, S, ok, t, a, b, c);
  for (double v : {0.0, -1.0, inf, nan, 1e-70, 1e70, 5e-324}) bad += fx_lane(2.2, -2, -4, v, 3.2, 0.28, 0.6, -0.5 / 0.6, t).ok;
  for (double v : {0.0, -1.0, inf, nan}) bad += fx_lane(2.2, -2, -4, 3.2, 3.2, v, 0.6, -0.5 / 0.6, t).ok;
  for (double v : {0.0, -0.6, 4.0, 0.015, inf, nan}) bad += fx_lane(2.2, -2, -4, 3.2, 3.2, 0.28, v, -0.5 / v, t).ok;
  for (double v : {16.0, inf, nan}) bad += fx_lane(v, -2, -4, 3.2, 3.2, 0.28, 0.6, -0.5 / 0.6, t).ok + fx_lane(2.2, v, -4, 3.2, 3.2, 0.28, 0.6, -0.5 / 0.6, t).ok;
  std::printf("%.17g %.17g %.17g %.17g %.17g %.17g %d %d %d\n", worst[0][0], worst[0][1], worst[0][2], worst[1][0],
              worst[1][1], worst[1][2], refused[0], refused[1], bad);
}
"""


def test_fixed_point_bond_functions(tmp_path):
    """Within the potential's ranges every value is within 1.5 x 2^-52 relative (2^-53 of rounding, the rest
    the fixed-point errors stated in fx64.cuh) plus, far beyond them, the 2^-54 absolute error of an exponent times the
    largest factor it meets (1/(2n) <= 25: 2^-54 ln2 25 < 1e-15). Nothing in range is refused; every argument outside
    the ranges is."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "fx.cpp"
    src.write_text(SRC)
    exe = tmp_path / "fx"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    v = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    worst, (refused, refused_wide, bad) = [float(x) for x in v[:6]], [int(x) for x in v[6:]]
    assert max(worst[:3]) <= 1.5 * 2.0 ** -52, worst
    assert max(worst[3:]) <= 1.5e-15, worst
    assert refused == 0 and bad == 0
    assert refused_wide < 0.05 * 200000


RANGE_SRC = SRC[:SRC.index("int main()")] + r"""
int main() {
  const FxTables &t = kFxTables;
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1, 1);
  auto pow2 = [&](double top) { return std::exp2(top * U(g)); };
  long taken = 0, wrong = 0;
  for (int i = 0; i < 2000000; ++i) {
    const double D0 = pow2(i & 1 ? 201 : 20), be = pow2(i & 2 ? 201 : 20), n = i & 4 ? 2 + 2 * U(g) : 0.3 + 0.29 * U(g);
    const double r0 = 16 * U(g), r = 8 + 8 * U(g), k = i & 8 ? 16 * U(g) : 2 * U(g), in = -0.5 / n;
    double S = i & 16 ? pow2(201) : pow2(20);
    if (i % 31 == 0) S = std::ldexp(1 + 0.5 * U(g), -150 - i % 925);         // down to subnormals
    if (i % 37 == 0) S = 0;
    double fR, bh, cc;
    if (!fx_bond(r, S, fx_lane(r0, k, 2 * k, D0, D0, be, n, in, t), t, fR, bh, cc)) continue;
    ++taken;
    const Q x = std::exp2((Q)k * ((Q)r - (Q)r0)), hA = D0 * x;
    Q z = (Q)be * (Q)S;
    if (z < (Q)1e-30) z = 1e-30;
    const Q zn = std::exp2((Q)n * std::log2(z)), b = std::exp2((Q)in * std::log2(1 + zn));
    const Q ref[3] = {hA * x, b * hA, (Q)be * b * hA * (zn / (1 + zn)) / (2 * z)};
    const double got[3] = {fR, bh, cc};
    for (int q = 0; q < 3; ++q) wrong += !(std::fabs((got[q] - ref[q]) / ref[q]) <= (Q)1e-14);
  }
  double a, b, c;   // zeta = 2^262, n = 3.9: zeta^n is far outside, b f_A / 2 is 1.0e-39
  wrong += fx_bond(2.35, std::ldexp(1, 63), fx_lane(2.35, -2, -4, 3.2, 3.2, std::ldexp(1, 199), 3.9, -0.5 / 3.9, t), t, a, b, c);
  std::printf("%ld %ld\n", taken, wrong);
}
"""


def test_fixed_point_bond_functions_at_the_ends_of_their_ranges(tmp_path):
    """Whatever is not refused is right, at the ends of every range that fx_lane and fx_bond accept. The exponents err by at
    most 2^-46.6 (1/(2n) <= 32 times the errors of n L and of log2(1 + zeta^n), and log2(1 + zeta^n) <= 250 times the
    2^-56 to which 1/(2n) is held), the values by ln2 times that, 6.5e-15, and cc by another 2^-49."""
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "fxr.cpp"
    src.write_text(RANGE_SRC)
    exe = tmp_path / "fxr"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    taken, wrong = (int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert taken > 200000 and wrong == 0, (taken, wrong)


def test_fixed_point_tables_recomputed():
    """Every entry of fx64_tables.inc from its definition, in 60-digit decimal arithmetic, and the bound that the
    logarithm's polynomial rests on: |m c_j - 1| < 2^-8.6 over the interval of j."""
    import re
    from decimal import ROUND_HALF_EVEN, Decimal, getcontext
    getcontext().prec = 60
    body = open(os.path.join(CSRC, "fx64_tables.inc")).read().split("= {", 1)[1]
    exp2, log_inv, inv = ([int(x, 0) for x in re.findall(r"0x[0-9a-f]+|\d+", part.replace("ull", ""))]
                          for part in re.findall(r"\{([^{}]*)\}", body))
    assert len(exp2) == len(log_inv) == len(inv) == 256
    ln2 = Decimal(2).ln()
    nearest = lambda x: int(x.to_integral_value(rounding=ROUND_HALF_EVEN))   # noqa: E731
    for j in range(256):
        assert exp2[j] == nearest((ln2 * j / 256).exp() * 2 ** 63)
        assert inv[j] == nearest(Decimal(2 ** 11) / (1 + (Decimal(j) + Decimal("0.5")) / 256))
        c = Decimal(inv[j]) / 2 ** 11
        assert log_inv[j] == nearest(-c.ln() / ln2 * 2 ** 62)
        for m in (1 + Decimal(j) / 256, 1 + Decimal(j + 1) / 256):
            assert abs(m * c - 1) < Decimal(2) ** Decimal("-8.6")
