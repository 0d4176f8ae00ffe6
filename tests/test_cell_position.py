"""csrc/cell.h, which places a direction in a pattern's grid by a known reciprocal and integer range tests,
against the plain FP64 formulas (a division, a second one for the remainder modulo the azimuth
count, floating-point clamps): the same bits, over steps from tiny to huge, directions in and out of the
table, on nodes and one ulp beside them, at the wrap, zeros of both signs, subnormals, infinities, NaN."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <limits>
#include <random>
#include "cell.h"
using namespace aerafold;
static long cases = 0, bad = 0;
static bool same(double a, double b) { return fp64_bits(a) == fp64_bits(b) || (std::isnan(a) && std::isnan(b)); }
static void quotient(double a, double b) {
  ++cases;
  if (!same(divide_by(a, b, reciprocal_of(b)), a / b)) { if (bad++ < 20) std::printf("%a / %a\n", a, b); }
}
static void place(double x, double x0, double dx, int n) {
  const double steps = divide_by(x - x0, dx, reciprocal_of(dx));
  double ua = 0.0, u;
  bool ok = std::isfinite(x);
  if (ok) { ua = (x - x0) / dx; ok = std::fabs(ua) < 0x1p52; }
  if (ok) { ua = ua - double(n) * std::floor(ua / double(n)); ok = ua >= 0.0 && ua <= double(n); }
  ++cases;
  if (azimuth_place(steps, x, n, &u) != ok || (ok && !same(u, ua))) { if (bad++ < 20) std::printf("azimuth %a %a %a %d\n", x, x0, dx, n); }
  double uz = (x - x0) / dx;
  bool clamp = false, c;
  if (uz < 0.0) { uz = 0.0; clamp = true; }
  if (uz > double(n - 1)) { uz = double(n - 1); clamp = true; }
  const bool zok = zenith_place(steps, x, n, &u, &c);
  if (zok != std::isfinite(x) || (zok && (c != clamp || !same(u, uz)))) { if (bad++ < 20) std::printf("zenith %a %a %a %d\n", x, x0, dx, n); }
}
int main() {
  std::mt19937_64 r(7);
  const double inf = std::numeric_limits<double>::infinity(), pi = 3.14159265358979323846;
  const double special[] = {0.0, -0.0, 5e-324, -5e-324, 1e-310, 0x1p-1000, -0x1p-1001, -0x1p-999, 1e-300, 1e300, -1e300, 1.7e308,
                            inf, -inf, std::nan(""), 1.0, -1.0, 0x1p52, 0x1p53, -0x1p52};
  auto mantissa = [&](int k) {   // random, few bits, nearly all ones, nearly a power of two
    const uint64_t m = r() >> 12;
    const uint64_t f = k == 0 ? m : k == 1 ? m & ~((uint64_t{1} << 40) - 1) : k == 2 ? (uint64_t{1} << 52) - 1 - (m >> 48) : m >> 48;
    uint64_t b = (uint64_t{1023} << 52) | f;
    double x;
    memcpy(&x, &b, 8);
    return x;
  };
  for (long i = 0; i < 3000000; ++i) {
    const double a = mantissa(i % 4), b = mantissa((i / 4) % 4);
    quotient(a, b);
    quotient(i & 1 ? -a : a, std::ldexp(b, int(r() % 1400) - 700));
    quotient(std::ldexp(a, int(r() % 2000) - 1000), std::ldexp(b, int(r() % 1200) - 600));
    quotient(std::nextafter(a * b, i & 1 ? 0.0 : 9.0), b);   // beside an exact quotient
  }
  for (double a : special) for (double b : {5e-324, 1e-310, 1e-200, 0x1p-400, 0.3, 1.0, 0x1p400, 1e200, 1.7e308}) quotient(a, b);
  const int counts[] = {2, 3, 7, 24, 72, 120, 360, 1000, 65536, 2147483647};
  for (int n : counts)
    for (double x0 : {0.0, -pi, 0.1, 1e-9, 1e6})
      for (double dx : {2 * pi / n, std::nextafter(2 * pi / n, 0.0), 2 * pi / n * (1 + 1e-9), 1.0, 1e-250, 1e250}) {
        for (double x : special) place(x, x0, dx, n), place(x0 + x, x0, dx, n);
        for (int i = -2 * 24; i <= 3 * 24; ++i) {   // nodes near both ends and throughout
          const double k = i < 24 ? i : i < 48 ? n - 36 + i : std::floor(double(n) * (i - 48) / 12);
          const double x = x0 + k * dx;
          place(x, x0, dx, n), place(std::nextafter(x, -inf), x0, dx, n), place(std::nextafter(x, inf), x0, dx, n);
        }
        for (int i = 0; i < 3000; ++i) place((double(r() >> 11) * 0x1p-53 * 6 - 3) * 2 * pi, x0, dx, n);
      }
  std::printf("%ld cases, %ld bad\n", cases, bad);
  return bad != 0;
}
"""


def test_positions_equal_the_plain_formulas(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "cell.cpp", tmp_path / "cell"
    src.write_text(SOURCE)
    subprocess.check_call([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I",
                           os.path.join(ROOT, "paper_1507_07733_gb300", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
