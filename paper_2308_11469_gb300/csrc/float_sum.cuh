// Sums of a few floats to FP64's accuracy without the FP64 pipe.
#pragma once
#include <cuda_runtime.h>
#ifdef __CUDACC__
#include "fp_bits.cuh"
#endif

namespace helm {

// float -> double, exact for every value, without the FP64 pipe unless it is subnormal
__host__ __device__ __forceinline__ double widen_any(float f)
{
#ifdef __CUDA_ARCH__
    const unsigned mag = __float_as_uint(f) & 0x7fffffffu;
    return mag - 1u < 0x007fffffu ? (double)f : f2d_bits(f);
#else
    return (double)f;
#endif
}

// a + b as the rounded sum (returned) and its error (err), which is a float (Knuth's two-sum)
__host__ __device__ __forceinline__ float two_sum(float a, float b, float& err)
{
    const float t = a + b, bb = t - a;
    err = (a - (t - bb)) + (b - bb);
    return t;
}

// Sum of n non-negative floats, rounded once (to 2^-53 of it; in FP64 one by one, once for each):
// kept as three floats, the errors of the first sum being summed in the second and the second's
// in the third, so that only the last two additions are FP64: a warp's FP64 instruction holds
// its pipe for 64 clocks, and a thread adding eight warps' values in FP64 kept the whole CTA
// waiting.  Sums beyond the floats' range (and infinities and NaN) are added in FP64.
__host__ __device__ __forceinline__ double sum_floats(const float* p, int n)
{
    float s = 0.f, c = 0.f, d = 0.f;
    for (int i = 0; i < n; ++i) {
        float e, f;
        s = two_sum(s, p[i], e);
        c = two_sum(c, e, f);
        d += f;
    }
    if (s <= 3.402823466e38f) return widen_any(s) + (widen_any(c) + widen_any(d));
    double t = 0.0;
    for (int i = 0; i < n; ++i) t += (double)p[i];
    return t;
}

}  // namespace helm
