// FP64 helpers shared by the pointwise physics and the WENO5-Z kernels.
#pragma once

namespace ffe {

// Sign and magnitude of a double as integers: a comparison of two doubles takes a
// slot of the FP64 pipe (2 lanes a clock and SM), one of integers a slot of a pipe
// that is 32 times wider.
__device__ __forceinline__ unsigned long long fbits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ unsigned long long fmag(double x) { return fbits(x) & 0x7fffffffffffffffULL; }
__device__ __forceinline__ bool fneg(double x) { return __double_as_longlong(x) < 0; }
__device__ __forceinline__ unsigned long long umax(unsigned long long a, unsigned long long b) { return a > b ? a : b; }
__device__ __forceinline__ unsigned long long umin(unsigned long long a, unsigned long long b) { return a < b ? a : b; }
__device__ __forceinline__ double flip(double x, unsigned long long sign) {
    return __longlong_as_double((long long)(fbits(x) ^ sign));
}
__device__ __forceinline__ bool is_finite(double x) { return fmag(x) < 0x7ff0000000000000ULL; }
// x > y for x >= 0 and y >= 0 (false where one is NaN, as the FP64 comparison)
__device__ __forceinline__ bool above(double x, double y) { return fbits(x) > fbits(y) && fbits(x) <= 0x7ff0000000000000ULL; }
__device__ __forceinline__ bool is_zero(double x) { return fmag(x) == 0; }

// 1/d for a normal d whose reciprocal is normal: the hardware
// approximation rcp.approx.ftz.f64 refined by two Newton-Raphson steps for
// f(y) = 1/y - d, y <- y + y (1 - d y) (each squares the relative error; the
// residual 1 - d y is exact in one FMA when y is close to 1/d).  Within about
// one ulp of the rounded quotient (ffe_eval_recip exposes it for tests); used
// for the adjoint's WENO5-Z weight denominators (positive sums bounded away from
// zero; for sums above 2^1022 the flushed reciprocal is 0) and, through recip_any,
// for the pointwise physics.
__device__ __forceinline__ double recip_nr(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    double r = fma(-d, y, 1.0);
    y = fma(y, r, y);
    r = fma(-d, y, 1.0);
    return fma(y, r, y);
}

// The same in one step of third order, y + y (e + e^2) with e = 1 - d y, in one FP64
// operation less (the adjoint's recomputation keeps recip_nr and its last bits).  The
// approximation's e is at most 2^-19.9 and the result within one ulp of the rounded
// quotient over 1.6e8 random arguments on a GB300; e^3 is what the step leaves.
__device__ __forceinline__ double recip_nr3(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// 2^-floor(log2 x) for a positive normal x below 2^1022: x times it lies in
// [1, 2) and the product is exact (integer operations on the exponent field).
__device__ __forceinline__ double pow2_inv_scale(double x) {
    const long long e = __double_as_longlong(x) >> 52;
    return __longlong_as_double((2046LL - e) << 52);
}

// 1/x for any finite nonzero x: recip_nr inside the range where it is
// defined (2^-1000 <= |x| < 2^1000), the IEEE quotient outside it.
__device__ __forceinline__ double recip_any(double x) {
    const unsigned e = (unsigned)(fmag(x) >> 52) - (1023u - 1000u);
    return e < 2000u ? recip_nr(x) : 1.0 / x;
}

}  // namespace ffe
