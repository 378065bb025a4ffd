// FP64 multigrid sweeps and transfers on shared-memory windows in 64-bit fixed point.
//
// GB300's FP64 pipe serves about 2 lanes of an SM a clock, its integer pipes 64 and more: a
// Gauss-Seidel update (10 FP64 operations for a complex node) takes 5.9 clocks of an SM, its
// integer form (30 integer operations) half a clock.  A window's FP64 values are put on one
// fixed-point scale, as in fixed_lap.cuh but rounded to nearest: v becomes v 2^(1080 - emax),
// emax at least the largest biased exponent of the window's iterate and of h^2 rhs.  Sums of
// neighbours are then exact; the divisions by 4 and 16 of the local solve and of the transfers
// are shifts, rounded to nearest, ties to even (rounding ties up adds an eighth of a unit on
// average to every node: a constant that the coarse levels amplify by N^2 / 14, 1.4e-14 of a
// 1023^2 cycle's result for a rough right-hand side).  One unit is 2^-58 (2^-56 in the descent, whose residuals need headroom)
// of the window's largest value, where FP64 rounds every partial sum at 2^-53 of its own size:
// the cycle's error is no larger, as a part of the window's largest value (measured against
// 64-bit cycles in tests/test_gpu_fixed_win.py; values below 2^-5 of it, 2^-3 in the descent, keep
// fewer than FP64's 53 bits).  Values return to FP64 rounded to nearest, ties to even.
//
// 1023^2 FP64 solve, V(0,1), 17 steps: 3.77 -> 2.78 ms; 63^2, V(2,2): 1294 -> 1137 us.
//
// The FP64 code remains for what has no such form: a shift sigma > 0 (the local solve's factor
// is then no power of two) and windows whose largest value is zero, below 2^-951 or above
// 2^1003, an infinity or a NaN.
#pragma once
#include "fixed_lap.cuh"
#include "launch.h"

namespace helm {
namespace {

// v 2^(1080 - emax) rounded to nearest, |result| <= 2^58 (a PTX right shift by 64 or more
// gives 0: no test for far smaller values)
__device__ __forceinline__ long long fx_q(double v, int emax)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned mh = (hi & 0x000fffffu) | 0x00100000u;
    unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, 10) << 32) | (lo << 10);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(emax - e + 4));
    m = (m + 1) >> 1;
    const long long sg = (long long)((int)hi >> 31);
    return ((long long)m ^ sg) - sg;
}
__device__ __forceinline__ longlong2 fx_q2(double2 v, int emax)
{
    return make_longlong2(fx_q(v.x, emax), fx_q(v.y, emax));
}
__device__ __forceinline__ double2 fx_d2(longlong2 v, int emax)
{
    return make_double2(fx_to_double(v.x, emax), fx_to_double(v.y, emax));
}

__device__ __forceinline__ int fx_exp2(double2 v) { return max(fx_exp(v.x), fx_exp(v.y)); }

// largest of the threads' exponents (one shared word per warp; the caller's barrier
// follows before any thread reads the result)
template <int NT>
__device__ __forceinline__ int block_max_exp(int ex, int* sx)
{
    ex = __reduce_max_sync(0xffffffffu, ex);
    if ((threadIdx.x & 31) == 0) sx[threadIdx.x >> 5] = ex;
    __syncthreads();
    int m = sx[0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) m = max(m, sx[w]);
    return m;
}

// may a window with largest biased exponent emax use fixed point (with room for the scales
// derived from it)?
__device__ __forceinline__ bool fx_usable(int emax) { return emax >= FX_EMIN + 8 && emax <= FX_EMAX - 8; }

// v 2^(1080 - emax) truncated (fx_fix without its range test)
__device__ __forceinline__ long long fx_qt(double v, int emax)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned mh = (hi & 0x000fffffu) | 0x00100000u;
    unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, 10) << 32) | (lo << 10);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(emax + 5 - (int)((hi >> 20) & 0x7ffu)));
    const long long sg = (long long)((int)hi >> 31);
    return ((long long)m ^ sg) - sg;
}

// v 2^(emax - 1080) rounded to nearest, ties to even, in the inner precision; binary32 results
// below the normal range become zero (as d2f_bits does)
__device__ __forceinline__ double fx_inner(long long v, int emax, double) { return fx_to_double(v, emax); }
__device__ __forceinline__ float fx_inner(long long v, int emax, float)
{
    const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
    const int lz = __clzll((long long)a);
    const unsigned long long m = a << (lz & 63);          // leading 1 at bit 63
    // 32 bits with the rest folded into the last one: the rounding to 24 sees the same
    const unsigned b = __float_as_uint(__uint2float_rn((unsigned)(m >> 32) | ((unsigned)m != 0u)));
    // b = top * 2^0 with top in [2^31, 2^32]; the value is top * 2^(32 - lz + emax - 1080)
    const int E = (int)(b >> 23) + 32 - lz + emax - 1080;
    const unsigned f = (unsigned)E - 1u < 254u ? ((unsigned)E << 23) | (b & 0x007fffffu) : (E >= 255 ? 0x7f800000u : 0u);
    return __uint_as_float(a == 0ull ? 0u : f | ((unsigned)(v >> 32) & 0x80000000u));
}

// h^2 as a scale: the exponents h^2 adds to a value's (exactly for a power of two, else at most)
struct FxH2 {
    double h2;
    int add;
    bool pow2;
    __device__ explicit FxH2(double h2_) : h2(h2_)
    {
        const unsigned long long b = fx_bits(h2);
        pow2 = (b & 0x000fffffffffffffull) == 0ull;
        add = (int)(b >> 52) - 1023 + (pow2 ? 0 : 1);
    }
    // is the scale emax in range, also less these exponents?
    __device__ bool usable(int emax) const { return fx_usable(emax) && fx_usable(emax - add); }
    __device__ longlong2 q2(double2 r, int emax) const
    {
        if (pow2) return fx_q2(r, emax - add);
        return fx_q2(make_double2(r.x * h2, r.y * h2), emax);
    }
    // v 2^(emax - 1080) / h^2
    __device__ double2 over(longlong2 v, int emax) const
    {
        if (pow2) return fx_d2(v, emax - add);
        const double2 w = fx_d2(v, emax);
        return make_double2(w.x / h2, w.y / h2);
    }
};

// s / 2^k rounded to nearest, ties to even
template <int K> __device__ __forceinline__ long long fx_shr(long long s)
{
    return (s + ((1 << (K - 1)) - 1) + ((unsigned)(s >> K) & 1u)) >> K;
}

__device__ __forceinline__ longlong2 fx_gs(longlong2 a, longlong2 b, longlong2 c, longlong2 d, longlong2 r)
{
    return make_longlong2(fx_shr<2>(((a.x + b.x) + (c.x + d.x)) - r.x), fx_shr<2>(((a.y + b.y) + (c.y + d.y)) - r.y));
}

}  // namespace
}  // namespace helm
