// Division by a number whose reciprocal is at hand.  (Also read by a host compiler: nothing but C++ here.)
#pragma once

#include <math.h>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

// a / b with y = 1 / b rounded: two of Markstein's corrections, each with an exact remainder, give the
// rounded quotient ("Computation of elementary functions on the IBM RISC System/6000 processor", 1990).
// The remainder is exact, and the quotient that of a division bit for bit, where nothing leaves the range of
// normal numbers: a = 0 or |a| >= 2^-968, 2^-1021 <= |b| <= 2^1020 and 2^-1020 <= |a / b| <= 2^1020.  Below that
// the last bit may differ; infinite a or b give NaN.
__host__ __device__ __forceinline__ double divide_by(double a, double b, double y) {
  double q = a * y;
  q = fma(fma(-b, q, a), y, q);
  return fma(fma(-b, q, a), y, q);
}
