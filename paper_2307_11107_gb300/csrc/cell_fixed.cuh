// FP64 positions' cells and cloud-in-cell weights in integer arithmetic.  The
// GPU's FP64 pipe takes two lanes per cycle and SM (64 times fewer than the
// integer pipes): a coordinate costs it one fused product and one conversion
// here, against some forty instructions for divisions, floors, comparisons
// and four rounded products.  Included inside namespace apic::{anonymous}.
#pragma once

struct W4 {
  unsigned long long w00, w10, w01, w11;
};

// Cell of a logical coordinate u = (x + 1) s 2^-b (in cells; s holds the factor
// 2^b, which the caller multiplies in once) and the fraction in it in units of
// 2^-b: index and fraction fit a signed 64-bit word (u < 2^(62 - b) cells; with
// b = kCellBits up to 4096 of them), and the fraction's rounding is below the
// resolution of an FP64 coordinate in cells from u = 2^(53 - b) on and below
// the deposit's own rounding before.  A coordinate outside [0, n] takes the edge cell
// and its edge.
constexpr int kCellBits = 50;
constexpr double kCellOne = (double)(1ll << kCellBits);
__device__ __forceinline__ int cell_fixed(double x, double s, int n, int b, unsigned long long& f) {
  const long long t = __double2ll_rn(fma(x, s, s));
  const int i = (int)(t >> b);
  f = i < 0 ? 0ull : (i > n - 1 ? 1ull << b : (unsigned long long)t & ((1ull << b) - 1ull));
  return min(max(i, 0), n - 1);
}

// Corner weights of the fractions f1, f2 (units of 2^-b), each the exact
// product rounded to F < 2 b bits.
__device__ __forceinline__ W4 weights_fixed(unsigned long long f1, unsigned long long f2, int b, int F) {
  const unsigned long long one = 1ull << b, g1 = one - f1, g2 = one - f2;
  const int sh = 2 * b - F;
  const unsigned __int128 half = (unsigned __int128)1 << (sh - 1);
  W4 w;
  w.w00 = (unsigned long long)(((unsigned __int128)g1 * g2 + half) >> sh);
  w.w10 = (unsigned long long)(((unsigned __int128)f1 * g2 + half) >> sh);
  w.w01 = (unsigned long long)(((unsigned __int128)g1 * f2 + half) >> sh);
  w.w11 = (unsigned long long)(((unsigned __int128)f1 * f2 + half) >> sh);
  return w;
}
