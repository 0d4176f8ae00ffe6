"""band_window (csrc/band.h), which finds the band's bins by bisection, against the definition: every
bin k of [0, n) with 30 MHz <= k fs / n <= 80 MHz. Compiled for the host; exact equality over the three
trace lengths and others, rates from far below the band to far above it, and rates that put a bin
on a band edge to the last bit or one ulp beside it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include "band.h"
int main() {
  int bad = 0, cases = 0;
  auto check = [&](int n, double fs) {
    int lo = -1, cnt = 0, hi = -1, a, c, b;
    for (int k = 0; k < n; ++k) {
      const double f = static_cast<double>(k) * fs / static_cast<double>(n);
      if (f >= 30e6 && f <= 80e6) {
        if (lo < 0) lo = k;
        hi = k;
        ++cnt;
      }
    }
    aerafold::band_window(n, fs, &a, &c, &b);
    ++cases;
    if (a != lo || b != hi || c != cnt) { std::printf("n=%d fs=%.17g: %d %d %d, not %d %d %d\n", n, fs, a, c, b, lo, cnt, hi); ++bad; }
  };
  for (int n : {1, 2, 7, 1024, 2048, 4096}) {
    for (double fs : {1e-300, 1.0, 29e6, 30e6, 80e6, 160e6, 200e6, 204.8e6, 220e6, 240e6, 1e9, 1e12, 1e300}) check(n, fs);
    for (int k = 1; k < n; k += n / 64 + 1)
      for (double edge : {30e6, 80e6}) {
        const double fs = edge * n / k;
        check(n, fs);
        check(n, std::nextafter(fs, 0.0));
        check(n, std::nextafter(fs, 1e300));
      }
    std::srand(n);
    for (int i = 0; i < 300; ++i) check(n, 1e6 * std::pow(10.0, 4.0 * std::rand() / RAND_MAX));
  }
  std::printf("%d cases, %d bad\n", cases, bad);
  return bad != 0;
}
"""


def test_band_window_equals_the_walk_over_the_bins(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "band.cpp", tmp_path / "band"
    src.write_text(SOURCE)
    subprocess.check_call([gxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I",
                           os.path.join(ROOT, "paper_1507_07733_gb300", "csrc"), str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
