// w / b where r = 1 / b rounded to nearest is at hand: one correction of the product
// w r (Markstein's division step, 1990), three operations instead of the some twenty
// of an FP64 division.  The remainder w - q b of the second line is exact or rounded
// in its last bit, so the result is within 1/2 ulp and 2^-50 of one of the quotient:
// the rounded quotient except beside a midpoint of two numbers, then its neighbour.  For
// finite b whose reciprocal is a normal number, and quotients whose remainder (2^-53
// of w) does not underflow; a zero w gives a zero.
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define FTSP2_HD __host__ __device__ __forceinline__
#else
#define FTSP2_HD inline
#endif

namespace ftsp2 {

FTSP2_HD double div_by(double w, double b, double r) {
    const double q = w * r;
    return fma(fma(-q, b, w), r, q);
}

}  // namespace ftsp2
