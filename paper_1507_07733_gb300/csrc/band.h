// band.h -- the band of the unfolding, 30-80 MHz inclusive (arXiv 1507.07733 Sec. 1), in bins.
#pragma once

namespace aerafold {

constexpr double kBandLoHz = 30e6;
constexpr double kBandHiHz = 80e6;

// First and last bin k in [0, n) of an n-point transform at rate fs > 0 with 30 MHz <= k fs / n <=
// 80 MHz (in FP64 as written) and their count; -1, -1, 0 if there is none. k fs / n does not
// decrease with k, so both ends are found by bisection: 24 evaluations where a walk over the bins
// took n (2048 divisions, 4 to 8 us of every call, as long as a small event takes on the GPU).
inline void band_window(int n, double fs, int* k_lo, int* count, int* k_hi) {
  const auto first = [&](auto inside) {   // the first k in [0, n] from which inside(frequency of k) holds
    int lo = 0, hi = n;
    while (lo < hi) {
      const int mid = lo + (hi - lo) / 2;
      if (inside(static_cast<double>(mid) * fs / static_cast<double>(n))) hi = mid;
      else lo = mid + 1;
    }
    return lo;
  };
  const int a = first([](double f) { return f >= kBandLoHz; });
  const int b = first([](double f) { return f > kBandHiHz; });   // one past the last
  *count = b > a ? b - a : 0;
  *k_lo = *count ? a : -1;
  *k_hi = *count ? b - 1 : -1;
}

}  // namespace aerafold
