// slice_math.h -- two exact rewritings in the Gibbs/measure kernel (slice.cu) that keep its per-site
// loops off the FP64 pipe (two operations per cycle and SM).  For host and device alike.
//
// With these and the unrolled transforms the kernel takes 161 instead of 177 us for 64 chains of
// L = 32 (M = 80), the grouped form 37.5 instead of 43.5 us for 32 of L = 12 (M = 120).
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define HQMC_HD __host__ __device__ __forceinline__
#else
#define HQMC_HD inline
#endif

namespace hqmc {

// Integer threshold of a Gibbs draw: with u = k 2^-53 (k the word's leading 53 bits),
// u < p if and only if k < ceil(p 2^53); p 2^53 is exact.
HQMC_HD unsigned long long gibbs_threshold(double p) { return (unsigned long long)ceil(p * 0x1.0p53); }

// x / N for an integer N < 2^15 with inv = 1 / N correctly rounded: the correctly rounded quotient by
// one residual (Markstein, IBM J. Res. Dev. 34, 1990), exact in one product when N is a power of two.
HQMC_HD double div_n(double x, double n, double inv, bool pow2) {
    const double q = x * inv;
    return pow2 ? q : fma(fma(-q, n, x), inv, q);
}

}  // namespace hqmc
