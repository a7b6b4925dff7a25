// One divisor, many dividends: quotients rounded as a division rounds them (to within 2^-52 of a last place
// beside a tie).
#pragma once

namespace gdsw {

// Whether quotient_by may be used: d and 1 / d far from the ends of the range, so that neither the quotient
// nor its remainder is cut off for dividends of up to |d|.
__device__ __forceinline__ bool quotient_ok(double d) { return d >= 0x1p-900 && d <= 0x1p900; }

// v / d from r = 1 / d: v r is up to two roundings off; its remainder v - q d is exact in one fused step and
// corrects it (P. Markstein, Computation of elementary functions on the IBM RISC System/6000 processor,
// 1990).  Three FP64 instructions, where a division is a dozen: FP64 is what bounds a pass like this here.
// Dividends below 2^-900 in magnitude may be one rounding more off.
__device__ __forceinline__ double quotient_by(double v, double d, double r) {
  const double q = v * r;
  return fma(fma(-q, d, v), r, q);
}

}  // namespace gdsw
