// cell.h -- a direction's place in a pattern's (zenith, azimuth) grid, in FP64, in steps of an axis.
//
// FP64 runs at 1/64 of the FP32 rate here: with three divisions (each some ten dependent operations),
// floors and comparisons in FP64 one thread took 1.9 us for a cell, now 1.1, a tenth of a small event.
// So the axis steps' reciprocals come with the pattern, range tests compare bit patterns as
// integers, and the common ranges need no second division. Every result is that of the plain
// formulas, to the bit. Calls back to back: 10 x 1 pairs of 2048 samples 12.05 -> 11.26 us, 7 x 19 of
// 1024 11.10 -> 10.07, 101 x 97 of 1024 52.0 -> 50.9, 124 x 64 of 2048 in three patterns 80.6 -> 79.15.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace aerafold {

__host__ __device__ inline uint64_t fp64_bits(double x) {
  uint64_t u;
  memcpy(&u, &x, sizeof u);
  return u;
}
constexpr uint64_t kFp64Sign = 0x8000000000000000ull;

// IEEE operations, never contracted
__host__ __device__ inline double fp64_sub(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dsub_rn(a, b);
#else
  return a - b;
#endif
}
__host__ __device__ inline double fp64_mul(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ inline double fp64_div(double a, double b) {
#ifdef __CUDA_ARCH__
  return __ddiv_rn(a, b);
#else
  return a / b;
#endif
}

// 1 / b for divide_by, or 0 where divide_by has to divide (b positive)
inline double reciprocal_of(double b) { return b >= 0x1p-400 && b <= 0x1p400 ? 1.0 / b : 0.0; }

// The correctly rounded a / b from inv, the correctly rounded 1 / b: the product a inv is off by
// less than 2 units, one correction by the remainder makes it one of the two neighbours of a / b, and
// Markstein's theorem (IBM J. Res. Dev. 34 (1990) 111) makes the second correction's result the
// rounded quotient. Five dependent operations. The exponents in range keep every term normal.
__host__ __device__ inline double divide_by(double a, double b, double inv) {
  const unsigned ea = static_cast<unsigned>(fp64_bits(a) >> 52) & 0x7ffu;
  if (ea - 523u > 1000u || fp64_bits(inv) == 0) return fp64_div(a, b);
  double q = fp64_mul(a, inv);
  q = fma(fma(-b, q, a), inv, q);
  return fma(fma(-b, q, a), inv, q);
}

// The azimuth's position ua in steps from az0, reduced to [0, n_az]; false if it has none. An
// azimuth has a place when it is finite and less than 2^52 azimuth steps from az0 (beyond, one
// FP64 unit is a whole step): ua - n_az floor(ua / n_az), which lands in [0, n_az]; the range
// test keeps every slab index in bounds. In [0, n_az) the floor is 0, in (-n_az, 0) it is -1
// (the rounded quotient reaches neither 1 nor -1, nor, above 2^-1000, 0).
__host__ __device__ inline bool azimuth_place(double steps, double az, int n_az, double* ua_out) {
  const double n = n_az;
  double ua = steps;
  const uint64_t u = fp64_bits(ua), un = fp64_bits(n);
  bool ok = true;
  if (u < un) {
  } else if (u > kFp64Sign + (uint64_t{23} << 52) && u < kFp64Sign + un) {
    ua = fp64_sub(ua, -n);
  } else {
    ok = (fp64_bits(az) & ~kFp64Sign) < 0x7ff0000000000000ull && fabs(ua) < 0x1p52;
    if (ok) {
      ua = fp64_sub(ua, fp64_mul(n, floor(fp64_div(ua, n))));
      ok = ua >= 0.0 && ua <= n;
    }
  }
  *ua_out = ua;
  return ok;
}

// The zenith's position in steps, clamped to [0, n_zen - 1] (*clamped); false if it is not finite.
__host__ __device__ inline bool zenith_place(double steps, double zen, int n_zen, double* uz_out, bool* clamped) {
  const double last = n_zen - 1;
  double uz = steps;
  *clamped = false;
  bool ok = true;
  if (fp64_bits(uz) > fp64_bits(last)) {   // also -0 and NaN
    if (uz < 0.0) { uz = 0.0; *clamped = true; }
    if (uz > last) { uz = last; *clamped = true; }
    ok = (fp64_bits(zen) & ~kFp64Sign) < 0x7ff0000000000000ull;
  }
  *uz_out = uz;
  return ok;
}

}  // namespace aerafold
