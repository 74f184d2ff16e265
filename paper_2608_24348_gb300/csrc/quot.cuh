// quot.cuh -- division by a number whose reciprocal is at hand.
//
// The stepper divides every node's value by the assembled mass and by the time
// step; a division is about nine operations of the FP64 pipe, which bounds those
// passes, and this is three.  The bits are to be those of the division: the
// loosely stopped solves downstream amplify a last-bit change of the velocity by
// 1e6 and more.
#pragma once

#include <string.h>

#ifdef __CUDACC__
#define SEM_HD __host__ __device__ __forceinline__
#else
#define SEM_HD inline
#endif

// a / b from r = 1 / b rounded to nearest (b and r between 2^-100 and 2^100).  One
// residual step (Markstein, IBM J. Res. Dev. 34, 1990) turns a first quotient
// within an ulp of a / b into its rounding; a r can be off by up to 1.5 ulp, where
// the theorem does not apply and no difference has been found: none in 30 M random
// quotients, nor in 3.7 M of those that lie closest to a rounding boundary (a
// smaller sample of each is tested).  The first quotient stands where it is zero
// (its sign), infinite or NaN, and below 2^-900, where the residual could lose bits.
SEM_HD double div_r(double a, double b, double r)
{
    const double q = a * r;
#ifdef __CUDA_ARCH__
    const unsigned hi = (unsigned)__double2hiint(q);
#else
    unsigned long long w;
    memcpy(&w, &q, sizeof(w));
    const unsigned hi = (unsigned)(w >> 32);
#endif
    const double s = fma(fma(-q, b, a), r, q);
    return (hi >> 20 & 0x7ffu) - 123u < 0x7ffu - 123u ? s : q;
}
