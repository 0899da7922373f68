// Float64 quotients from a shared reciprocal (keyframe alignment).
#pragma once

// The reciprocal of a normal x > 0 to about one unit in the last place: the
// hardware's float64 seed (some 20 bits) and two Newton steps, each squaring
// the relative error.
__device__ __forceinline__ double ka_rcp(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// a / b from r = ka_rcp(b), correctly rounded: the quotient a r corrected by
// its exact remainder (P. Markstein, IBM J. Res. Dev. 34(1), 1990).  What is
// rounded last lies within 2^-51 units in the last place of a / b, so that
// the result is that of the division unless a / b is that close to a
// midpoint.  Divisions by one value share its reciprocal: three operations
// each instead of a division sequence.  b is normal and below 2^1022: depths and
// their products are, and the callers see to the Cauchy scale's.
__device__ __forceinline__ double ka_div(double a, double b, double r) {
  const double q = a * r;
  return fma(fma(-b, q, a), r, q);
}
