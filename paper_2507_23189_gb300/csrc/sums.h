// Sums of single-precision numbers that lose no more than a double would.
#ifndef MCMIE_SUMS_H
#define MCMIE_SUMS_H

#include <math.h>

#ifdef __CUDACC__
#define MCX_SUM_HD __host__ __device__ __forceinline__
#else
#define MCX_SUM_HD inline
#endif

namespace mcx {

// The unevaluated sum s + c + r: SumK with K = 3 of Ogita, Rump and Oishi,
// "Accurate sum and dot product", SIAM J. Sci. Comput. 26 (2005). Of n numbers
// it is off by at most (2 n 2^-24)^3 times the sum of their magnitudes, 2^-48
// for 128; adding them up in double, by up to 127 2^-53 or 2^-46 (a Kahan pair:
// 2^-41). 13 single-precision additions a number.
struct Sum3 {
    float s = 0.f, c = 0.f, r = 0.f;

    MCX_SUM_HD void add(float x)
    {
        float t = s + x, z = t - s;
        const float e = (s - (t - z)) + (x - z);    // s + x = t + e exactly
        s = t;
        t = c + e;
        z = t - c;
        r += (c - (t - z)) + (e - z);
        c = t;
    }
    MCX_SUM_HD double value() const
    {
        // where s is infinite or NaN the corrections are NaN
        return s - s == 0.f ? (double)s + ((double)c + (double)r) : (double)s;
    }
};

}  // namespace mcx

#endif
