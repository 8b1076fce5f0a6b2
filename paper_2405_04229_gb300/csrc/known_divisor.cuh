// Division by a number whose reciprocal is known.
#pragma once

#include <math.h>

namespace cs {

// x / c for rc = 1 / c correctly rounded (Markstein, "Computation of elementary functions on the IBM
// RISC System/6000", 1990): the remainder of the first quotient, exact through FMA, corrects it.  The
// rounding is the division's while the remainder does not underflow (|x| from about 2^-960 on); c, rc
// and the quotient must be normal numbers.
__host__ __device__ inline double div_known(double x, double c, double rc) {
    const double q = x * rc;
    return fma(fma(-q, c, x), rc, q);
}

}  // namespace cs
