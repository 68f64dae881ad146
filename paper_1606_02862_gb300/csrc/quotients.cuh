// quotients.cuh -- the reciprocals and quotients of the Boris push, cheaper than
// the compiler's for the range they meet: divisors of 1 and more.
#pragma once

#include <cmath>

namespace pic {

// 1 / sqrt(x) for x >= 1: rsqrtf without its care for denormals, the same bits.
__device__ __forceinline__ float rsqrt_ge1(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 2 / x for x >= 1: the approximate reciprocal and one step of Newton's
// iteration for it, of x / 4, whose reciprocal is in FP32's normal range for
// every finite x: within 0.501 ulp of 2 / x (the step leaves the square of the
// approximation's 2^-23 and one rounding; x above 2^127 one rounding more).  An
// x that overflowed gives 0, as the division does (Newton's step alone would
// give 0 * infinity).
__device__ __forceinline__ float two_over_ge1(float x)
{
    const float h = 0.25f * x;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(h));
    r = fmaf(r, fmaf(-h, r, 1.0f), r);
    return x == INFINITY ? 0.0f : 0.5f * r;
}

// Quotients n / g of one divisor, each rounded once: a step of Newton's on
// n rg with the rounded reciprocal rg (Markstein 1990; n and n / g normal).  n
// rg alone moved the stored positions of a few particles by a last bit, which
// shows in the displacements of slow ones (1e-11 of the largest).  g beyond the
// largest double: 0, as n / g is.
struct Over64 {
    double g, rg;
    __device__ __forceinline__ explicit Over64(double v) : g(v), rg(1.0 / v) {}
    __device__ __forceinline__ double operator()(double n) const
    {
        const double q = n * rg;
        return rg != 0.0 ? fma(fma(-q, g, n), rg, q) : q;
    }
};

}  // namespace pic
