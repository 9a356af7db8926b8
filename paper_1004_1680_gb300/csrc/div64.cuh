// FP64 quotients for the FP64 sweeps (sweep_f64.cu): IEEE division's results with
// fewer FP64 operations.
//
// A division is about 14 FP64 operations here, and a fluid cell has 18 of them;
// written out for operands of ordinary size they are 7, and 3 more for each
// further quotient by the same divisor:
//   y0, the hardware's approximate reciprocal: |1 - r y0| <= 2^-19.93, and y0
//       depends on r's high word alone (measured over every high word),
//   y1 = y0 + y0 (1 - r y0), y = y1 + y1 (1 - r y1): two Newton steps, which
//       leave 2^-79 before y's own rounding: |y - 1/r| <= (1/2 + 2^-26) ulp(y),
//   q  = a y, then q + (a - q r) y (Markstein, "Computation of elementary
//       functions on the IBM RISC System/6000 processor", 1990).
// The result is a / r rounded to nearest.  Scale a and r so that r = B 2^-52 is
// in [1, 2) and Q = a / r in [1, 2), spacing u = 2^-52.  The last operation
// rounds s = q + (a - q r) y, and s - Q = r (q - Q) (1/r - y), below 1.5 r u 2^-53.9
// in any case.  Q is never a midpoint m of two neighbours, and not nearer to one
// than 1 / (2^53 B) = 2^-105 / r, since Q - m is an integer over 2^53 B.  Only
// where Q is about that near can s lie on the other side of m; q is then one of m's two
// neighbours (a y is within (1 - 2^-22) u of Q), the remainder exact in its FMA, |q - Q|
// at most u/2 and what lies beyond it, and |s - Q| <= r 2^-107 (1 + 2^-25), which is less than
// 2^-105 / r as long as r^2 (1 + 2^-25) < 4: for r < 2 (1 - 2^-21).
// So divisors whose mantissa begins with 20 ones take the division, and so do
// operands whose exponents could spoil the remainder (zeros, infinities and
// NaNs among them).
#pragma once
#include <cuda_runtime.h>

namespace mhd {

__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double ddiv(double a, double b) { return __ddiv_rn(a, b); }

__device__ __forceinline__ double approx_rcp(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ double reciprocal(double r) {
  const double y0 = approx_rcp(r);
  const double y1 = __fma_rn(__fma_rn(-r, y0, 1.0), y0, y0);
  return __fma_rn(__fma_rn(-r, y1, 1.0), y1, y1);
}
// a / r by y = reciprocal(r), for a plain_exponent(a) and a plain_divisor(r)
__device__ __forceinline__ double ddiv_by(double a, double r, double y) {
  const double q = dmul(a, y);
  return __fma_rn(__fma_rn(-q, r, a), y, q);
}
// 2^-500 <= |x| < 2^500 (from the exponent: no FP64 comparison)
__device__ __forceinline__ bool plain_exponent(double x) {
  return ((unsigned)__double2hiint(x) >> 20 & 0x7ffu) - 523u < 1000u;
}
__device__ __forceinline__ bool plain_divisor(double x) {
  return plain_exponent(x) && (~__double2hiint(x) & 0xfffff) != 0;
}

// half the van Leer limiter, phi(a, b) / 2 = ab / (a + b) for ab > 0, else 0
__device__ __forceinline__ double vl_half(double a, double b) {
  const double ab = dmul(a, b), s = dadd(a, b);
  const int hi = __double2hiint(ab);
  double q = 0.0;
  // (2^-500 <= ab < 2^500 leaves |s| between 2^-250 and 2^1023, its remainder normal)
  if ((unsigned)hi - (523u << 20) < (1000u << 20) && plain_divisor(s)) q = ddiv_by(ab, s, reciprocal(s));
  else if (hi >= 0 && (hi | __double2loint(ab)) != 0) q = ab > 0.0 ? ddiv(ab, s) : 0.0;
  return q;
}

}  // namespace mhd
