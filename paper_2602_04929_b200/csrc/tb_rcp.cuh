// Reciprocal of a pivot.
#pragma once

namespace tb {

// 1 / p for 2^-1000 <= p <= 2^1000: one step of the hyperpower iteration of order three (M. Altman, "An optimum cubically
// convergent iterative method of inverting a linear bounded operator in Hilbert space", Pacific J. Math. 10, 1960), here for
// a number: r' = r (1 + e + e^2), e = 1 - p r, whose error is e^3.  The first r is the hardware's approximation, good to
// 2^-20 (rcp.approx.ftz.f64 in the PTX document), so e^3 is below 2^-60; the multiply-adds before the last one are rounded
// at 2^-73, the last one to half a unit of the last place.  So the error is below 0.51 units, and the result is the
// correctly rounded one or its neighbour.
__device__ __forceinline__ double panel_rcp(double p) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(p));
  const double e = fma(-p, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace tb
