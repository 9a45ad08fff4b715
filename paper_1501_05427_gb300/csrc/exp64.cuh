// exp(-dist / 2) in double precision for the kernel values of the FP64 path.
//
// Table-driven exponential (P. T. P. Tang, "Table-driven implementation of the exponential
// function in IEEE floating-point arithmetic", ACM TOMS 15, 1989): with N = 2048,
//     -dist / 2 = k ln2 / N + r,  |r| <= h = ln2 / (2N),   exp = 2^(k >> 11) T[k mod N] e^r,
// e^r by its Taylor polynomial of degree 3 whose r^2 coefficient takes up the r^4 term
// (r^4 / 24 ~ c r^2 / 24 with c = (2 sqrt 2 - 2) h^2, the minimax choice on |r| <= h): the
// polynomial's error is 0.172 h^4 / 24 = 6e-18 relative, below the rounding of the last
// operation.  The reduction is done on s = -2 r = dist + k 2 ln2 / N with one rounded constant:
// its error, dist 2^-55 in the exponent, is below the rounding of dist itself.
//
// Why: GB300's FP64 pipe issues about 1.7 lanes per clock per SM (measured, DFMA and DADD
// alike), so the kernel values' cost is their count of FP64 operations.  This form takes 7
// (the library call and its argument scaling about 16); everything else is integer work and
// one table load from the L1.
#pragma once

#include <cuda_runtime.h>

namespace ulisse {

constexpr int kExpTabBits = 11;
constexpr int kExpTabN = 1 << kExpTabBits;
constexpr double kExpLn2 = 0.693147180559945309417232121458;

// T[j] = 2^(j / N), kExpTabN doubles, filled once per context.
cudaError_t launch_fill_exp_tab(double* tab, cudaStream_t s);

__device__ __forceinline__ double exp_neg_half(double dist, const double* __restrict__ tab) {
  constexpr double kMagic = 6755399441055744.0;   // 1.5 * 2^52: the sum's low word is k
  constexpr double kInv = -(double)kExpTabN / (2.0 * kExpLn2);
  constexpr double kStep = 2.0 * kExpLn2 / (double)kExpTabN;
  constexpr double kH = kExpLn2 / (2.0 * kExpTabN);
  constexpr double kC2 = 0.125 + 0.82842712474619009760 * kH * kH / 96.0;
  // beyond 1400 the result leaves the normal range (and k its exact one); a NaN comes here or, with
  // its sign set, stays one below
  if (__double2hiint(dist) >= 0x4095E000) return exp(-0.5 * dist);
  const double z = fma(dist, kInv, kMagic);
  const int k = __double2loint(z);
  const double s = fma(z - kMagic, kStep, dist);
  const double t = __ldg(tab + (k & (kExpTabN - 1)));
  const double q = fma(s, fma(s, -1.0 / 48.0, kC2), -0.5);
  const double p = fma(t * s, q, t);
  return __hiloint2double(__double2hiint(p) + ((k >> kExpTabBits) << 20), __double2loint(p));
}

}  // namespace ulisse
