// FP64 reciprocal, reciprocal square root and logarithm of a ratio for the
// step kernels.  GB300's FP64 pipe takes 64 cycles per warp instruction and
// sub-partition, so the FP64 kernels cost what their FP64 instructions count;
// these take 3, 5 and 17 of them in place of a division (about 9), a division
// by a square root (about 17) and a division and a logarithm (about 36).
// With the short collision of lbm_node.cuh: 64 uneven FP64 cases 3.39 -> 2.21
// ms per step.  The reverse mode and the steps of handles that have it attached
// take the division, root and logarithm (lbm_handle::plain): d psi/d phi reaches 1e10,
// and the derivatives of a run move by up to 1e-8 with its states' last bits.
//   rcp, rsq: the hardware's approximation (PTX rcp/rsqrt.approx.ftz.f64, 20
//   bits) and one third-order Newton step: with e = 1 - x y, 1/x = y (1 + e +
//   e^2 + ...); with e = 1 - x y^2, 1/sqrt(x) = y (1 + e/2 + 3 e^2/8 + ...).
//   The remainder is below 2^-58; the results are within 2 ulp.  For normal
//   arguments (densities, relaxation times, |12 grad psi|^2 above its cut).
//   ln(a/b) = ln a - ln b, each by table and Taylor polynomial (P. T. P. Tang,
//   "Table-driven implementation of the logarithm function in IEEE
//   floating-point arithmetic", ACM TOMS 16, 1990): x = 2^e y, r = c y - 1
//   with c of the table, |r| < 2^-8.9, ln x = e ln 2 - ln c + ln(1 + r), five
//   terms (remainder r^6/6 < 2^-55).  Absolute error below 1e-15 (2e-16 for
//   |ln(a/b)| < 1).  Zero, subnormal, infinite or NaN arguments take log.
#pragma once
#include <cuda_runtime.h>

#include "lbm_logtab.h"

namespace lbmk {

__device__ __forceinline__ double rcp64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

__device__ __forceinline__ double rsq64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

// ln(1 + r) of x = 2^e y, e and -ln c (see above)
__device__ __forceinline__ double log64_part(double x, int& e, double& lc) {
  const int hi = __double2hiint(x);
  e = hi >> 20;
  const double2 t = __ldg(&kLogTab[(hi >> 12) & 0xFF]);
  const double y = __hiloint2double((hi & 0xFFFFF) | 0x3FF00000, __double2loint(x));
  lc = t.y;
  const double r = fma(y, t.x, -1.0);
  const double q = fma(r, fma(r, fma(r, 0.2, -0.25), 1.0 / 3.0), -0.5);
  return fma(r * r, q, r);
}

__device__ __forceinline__ double lratio64(double a, double b) {
  const unsigned ua = (unsigned)__double2hiint(a) - 0x00100000u;
  const unsigned ub = (unsigned)__double2hiint(b) - 0x00100000u;
  if (ua >= 0x7FE00000u || ub >= 0x7FE00000u) return log(a / b);
  int ea, eb;
  double la, lb;
  const double pa = log64_part(a, ea, la), pb = log64_part(b, eb, lb);
  // (double)(ea - eb) by one subtraction: 2^52 + 2^31 + n minus 2^52 + 2^31
  const double n = __hiloint2double(0x43300000, (ea - eb) ^ (int)0x80000000) - 4503601774854144.0;
  return fma(n, 0.69314718055994530942, (la - lb) + (pa - pb));
}

}  // namespace lbmk
