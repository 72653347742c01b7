// mm_fp64.cuh -- FP64 reciprocal, quotient, square root and its reciprocal by
// one step of Chebyshev's third-order iteration.
//
// GB300 issues an FP64 instruction in 16 cycles of the SM's pipe, so their
// number is what the kernels with FP64 arithmetic cost.  The hardware's seed
// (rcp/rsqrt.approx.ftz.f64, upper words only: a relative error of 2^-19 at
// most) with residual e = 1 - x y gives 1/x = y / (1 - e) = y (1 + e + e^2) +
// O(e^3): 2^-57 relative, then one rounding, in three instructions.  Outside
// 2^+-1000 the seed would flush and the library operation is taken.  The
// bounds, the ends of the range and zeros, infinities and NaN are checked
// against CUDA's operations by tests/test_gpu_fp64.py.
#pragma once

namespace mm {

__device__ __forceinline__ bool seed_range(double x)
{
    return (((unsigned)__double2hiint(x) >> 20) & 0x7ffu) - 23u < 2000u;
}

// The library's operations, out of line: they are for the ends of the range only
static __device__ __noinline__ double rcp_any(double x) { return 1.0 / x; }
static __device__ __noinline__ double quot_any(double a, double b) { return a / b; }
static __device__ __noinline__ double rsqrt_any(double x) { return rsqrt(x); }
static __device__ __noinline__ double sqrt_any(double x) { return sqrt(x); }

__device__ __forceinline__ double rcp64(double x)
{
    if (!seed_range(x)) return rcp_any(x);
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = __fma_rn(-x, y, 1.0);
    return __fma_rn(y, __fma_rn(e, e, e), y);
}

// |x| in [2^-500, 2^500): a quotient of two such, and its residual, are far
// from the ends of the range
__device__ __forceinline__ bool mid_range(double x)
{
    return (((unsigned)__double2hiint(x) >> 20) & 0x7ffu) - 523u < 1000u;
}

// a / b with the quotient's own residual folded back in.  Anything else than
// two numbers of the middle range is the library's quotient (infinities, NaN,
// a residual that would underflow), but for the frequent zero dividend.
__device__ __forceinline__ double div64(double a, double b)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = __fma_rn(-b, y, 1.0);
    y = __fma_rn(y, __fma_rn(e, e, e), y);
    const double q = __dmul_rn(a, y);
    if (mid_range(b)) {
        if (mid_range(a)) return __fma_rn(__fma_rn(-b, q, a), y, q);
        if ((__double_as_longlong(a) << 1) == 0) return q;
    }
    return quot_any(a, b);
}

// 1 / sqrt(x), x > 0: with e = 1 - x y^2, y (1 + e/2 + 3 e^2 / 8)
__device__ __forceinline__ double rsqrt64(double x)
{
    if (!seed_range(x)) return rsqrt_any(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double t = __dmul_rn(x, y);  // and its rounding, or e would carry it
    const double e = __fma_rn(-__fma_rn(x, y, -t), y, __fma_rn(-t, y, 1.0));
    return __fma_rn(__dmul_rn(y, e), __fma_rn(e, 0.375, 0.5), y);
}

// sqrt(x): the same iteration on t = x y, then one residual step,
// s + (x - s^2) y / 2 (y / 2 by its exponent: y is a normal number)
__device__ __forceinline__ double sqrt64(double x)
{
    if (!seed_range(x) || __double_as_longlong(x) < 0) return sqrt_any(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double t = __dmul_rn(x, y), e = __fma_rn(-t, y, 1.0);
    const double s = __fma_rn(__dmul_rn(t, e), __fma_rn(e, 0.375, 0.5), t);
    return __fma_rn(__fma_rn(-s, s, x), __longlong_as_double(__double_as_longlong(y) - (1LL << 52)), s);
}

}  // namespace mm
