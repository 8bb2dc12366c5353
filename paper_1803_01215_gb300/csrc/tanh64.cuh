// tanh of an FP64 argument in 14 FP64 instructions, without a branch: Taylor's
// expansion about the nearest multiple of 1/16 from a table of its coefficients.
//
// tanh' = 1 - tanh^2 gives every coefficient from the first: with t = sum c_n b^n,
// c_1 = 1 - c_0^2 and (n + 1) c_{n+1} = - sum_i c_i c_{n-i}.  |b| <= 1/32 and degree 10
// leave a remainder below 2^-63 (|c_11| <= 0.004), so the error is that of the last
// fused multiply-add and of c_0, under 1 ulp in all but the smallest arguments' row,
// where c_0 = 0 and the sum is b (1 + ...).  From 19.0625 on tanh rounds to 1.
#pragma once
#include <cuda_runtime.h>

namespace hj {

constexpr int kTanhRows = 306;    // |x| up to 19.0625
constexpr int kTanhRow = 12;      // 11 coefficients, rows of a whole number of 16-byte vectors

// the table, by a CTA's threads (the caller synchronises before it is read)
__device__ inline void tanh_taylor_table(double* tab, int tid, int nthr) {
  for (int k = tid; k < kTanhRows; k += nthr) {
    double c[kTanhRow];
    c[0] = tanh(0.0625 * k);
    // 1 - tanh^2 without cancellation: 1 / cosh^2
    const double ch = cosh(0.0625 * k);
    c[1] = 1.0 / (ch * ch);
    for (int n = 1; n < 10; ++n) {
      double s = 0.0;
      for (int i = 0; i <= n; ++i) s += c[i] * c[n - i];
      c[n + 1] = -s / (n + 1);
    }
    c[11] = 0.0;
    for (int n = 0; n < kTanhRow; ++n) tab[k * kTanhRow + n] = c[n];
  }
}

__device__ __forceinline__ double tanh_taylor(double x, const double* tab) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int ahi = hi & 0x7fffffff;
  // |x| capped at 19.0625 by its bits; NaN is returned as it came (below)
  const bool big = ahi >= 0x40331000;
  const double ax = __hiloint2double(big ? 0x40331000 : ahi, big ? 0 : lo);
  const double t = fma(ax, 16.0, 0x1.8p52);          // nearest multiple of 1/16 in the low word
  const double b = fma(t - 0x1.8p52, -0.0625, ax);   // exact
  const double2* c = reinterpret_cast<const double2*>(tab + __double2loint(t) * kTanhRow);
  const double2 c0 = c[0], c2 = c[1], c4 = c[2], c6 = c[3], c8 = c[4];
  double r = fma(c[5].x, b, c8.y);
  r = fma(r, b, c8.x);
  r = fma(r, b, c6.y);
  r = fma(r, b, c6.x);
  r = fma(r, b, c4.y);
  r = fma(r, b, c4.x);
  r = fma(r, b, c2.y);
  r = fma(r, b, c2.x);
  r = fma(r, b, c0.y);
  r = fma(r, b, c0.x);
  const bool nan = ahi > 0x7ff00000 || (ahi == 0x7ff00000 && lo != 0);
  return nan ? x : __hiloint2double(__double2hiint(r) | (hi & 0x80000000), __double2loint(r));
}

}  // namespace hj
