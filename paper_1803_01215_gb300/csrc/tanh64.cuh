// tanh of an FP64 argument in 13 FP64 instructions, without a branch: Taylor's
// expansion about the nearest multiple of 1/16 from a table of its coefficients.
//
// tanh' = 1 - tanh^2 gives every coefficient from the first: with t = sum c_n b^n,
// c_1 = 1 - c_0^2 and (n + 1) c_{n+1} = - sum_i c_i c_{n-i}.  |b| <= 1/32 and degree 10
// leave a remainder below 2^-61 (|c_11| <= 0.0089, its largest in the first row, where
// it is 2^-56 of the result).  c_0 is a pair of doubles, good to 2^-100, so what is left
// is the rounding of the last addition, of c_1 b and of c_1: 0.87 ulp at most (at
// 0.0313, where c_1 b and the result are of one size) and 0.64 from 0.1 on, by the same
// arithmetic on the host against 113-bit values at 6e6 arguments.  CUDA's tanh, measured
// the same way, is off by 1.40 ulp at most (at 0.549).  With c_0 one double from a
// tanh call, and the sum folded into it by one multiply-add, the table's largest error
// was 1.3 to 1.9 ulp, in 13 instructions too: the two more for the sum are won back by
// finding the row in FP32 and integer instructions, which do not wait for the FP64 pipe
// (d = 8, N = 10, 400 points: 6.11 ms with the one-double table, 6.36 with the row found
// in FP64, 5.93 so; d = N = 40, 160 points 71.0, 72.2 and 69.9).  From 19.0625 on tanh
// rounds to 1.
#pragma once
#include <cuda_runtime.h>

namespace hj {

constexpr int kTanhRows = 306;    // |x| up to 19.0625
constexpr int kTanhRow = 12;      // c_0's high part, c_1 .. c_10, c_0's low part: whole 16-byte vectors

// the product of two unevaluated sums (h, l), to about 2^-103 of it
__device__ inline double2 pair_mul(double2 a, double2 b) {
  const double p = __dmul_rn(a.x, b.x);
  const double e = __fma_rn(a.x, b.y, __fma_rn(a.y, b.x, __fma_rn(a.x, b.x, -p)));
  const double h = __dadd_rn(p, e);
  return make_double2(h, __dsub_rn(e, __dsub_rn(h, p)));
}

// the table, by a CTA's threads (the caller synchronises before it is read)
__device__ inline void tanh_taylor_table(double* tab, int tid, int nthr) {
  for (int k = tid; k < kTanhRows; k += nthr) {
    // u = e^{-2 k / 16} by binary powers of e^{-1/8}; tanh(k / 16) = (1 - u) / (1 + u)
    double2 u = make_double2(1.0, 0.0), s = make_double2(0x1.c3d6a24ed8222p-1, -0x1.e1e0a76cb0685p-55);
    for (int n = k; n > 0; n >>= 1) {
      if (n & 1) u = pair_mul(u, s);
      s = pair_mul(s, s);
    }
    const double nh = __dsub_rn(1.0, u.x);
    const double nl = __dsub_rn(__dsub_rn(__dsub_rn(1.0, nh), u.x), u.y);
    const double dh = __dadd_rn(1.0, u.x);
    const double dl = __dadd_rn(__dsub_rn(u.x, __dsub_rn(dh, 1.0)), u.y);
    const double q = __ddiv_rn(nh, dh);
    const double rem = __fma_rn(-q, dl, __dadd_rn(__fma_rn(-q, dh, nh), nl));
    const double q2 = __ddiv_rn(rem, dh);
    double c[kTanhRow];
    c[0] = __dadd_rn(q, q2);
    const double lo = __dsub_rn(q2, __dsub_rn(c[0], q));
    c[1] = __fma_rn(-2.0 * c[0], lo, __fma_rn(-c[0], c[0], 1.0));
    for (int n = 1; n < 10; ++n) {
      double sum = 0.0;
      for (int i = 0; i <= n; ++i) sum += c[i] * c[n - i];
      c[n + 1] = -sum / (n + 1);
    }
    c[11] = lo;
    for (int n = 0; n < kTanhRow; ++n) tab[k * kTanhRow + n] = c[n];
  }
}

__device__ __forceinline__ double tanh_taylor(double x, const double* tab) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int ahi = hi & 0x7fffffff;
  // |x| capped at 19.0625 by its bits; NaN is returned as it came (below)
  const bool big = ahi >= 0x40331000;
  const double ax = __hiloint2double(big ? 0x40331000 : ahi, big ? 0 : lo);
  // k / 16, the nearest multiple (to |x|'s upper 20 bits), in FP32 and integer
  // instructions: |x| as a float, 0 below 2^-127; k in the low bits of 1.5 2^23 + 16 |x|;
  // k as a float, and its bits as those of the double k / 16
  const int fi = max((big ? 0x40331000 : ahi) - (896 << 20), 0) << 3;
  const float m = fmaf(__int_as_float(fi), 16.0f, 12582912.0f);
  const int k = __float_as_int(m) - 0x4b400000;
  const int ci = (__float_as_int(m - 12582912.0f) >> 3) + (892 << 20);
  const double b = ax - __hiloint2double(k == 0 ? 0 : ci, 0);   // exact
  const double2* c = reinterpret_cast<const double2*>(tab + k * kTanhRow);
  const double2 c0 = c[0], c2 = c[1], c4 = c[2], c6 = c[3], c8 = c[4], c10 = c[5];
  double r = fma(c10.x, b, c8.y);
  r = fma(r, b, c8.x);
  r = fma(r, b, c6.y);
  r = fma(r, b, c6.x);
  r = fma(r, b, c4.y);
  r = fma(r, b, c4.x);
  r = fma(r, b, c2.y);
  r = fma(r, b, c2.x);                               // (tanh - c_0 - c_1 b) / b^2
  r = fma(c0.y, b, fma(r, __dmul_rn(b, b), c10.y));  // c_1 b and all that is smaller, rounded once
  r = __dadd_rn(c0.x, r);
  const bool nan = ahi > 0x7ff00000 || (ahi == 0x7ff00000 && lo != 0);
  return nan ? x : __hiloint2double(__double2hiint(r) | (hi & 0x80000000), __double2loint(r));
}

}  // namespace hj
