// Line contractions of the DG kernels in block fixed point, on the integer pipes.
//
// A contraction sum_m D_m u_m along a line of an element is FP64 work of 6 slots a
// value on a pipe with 2 lanes a clock and SM; the integer multiply-adds run 32
// lanes or more.  The values of a block (a variable, or variables that meet in one
// sum) are therefore scaled by one power of two per element and held as integers
// of up to 58 bits in two limbs, z = hi 2^28 + lo with |lo| <= 2^27; the operator's
// rows likewise.  A product is three 32 x 32 -> 64 bit multiply-adds into two
// 64-bit sums (hi hi into a, hi lo + lo hi into b; lo lo stays below the quantum),
// exact until the one rounding of the result to double.
//
// Error: the operands are cut at 2^-58 of the block's largest value and 2^-56 of
// the operator's largest entry, where the FP64 sum rounds each product and partial
// sum at 2^-53 of their size, so the sum's error is smaller by 2^3 or more wherever
// the line holds values of the size of the block's largest.  Blocks with values of
// 2^900 or more, infinities or NaN take the FP64 form (FX_EMAX); values below
// 2^-958 count as zero.
#pragma once
#include "ffe_internal.h"
#include "fp64util.cuh"

namespace ffe {

constexpr int FX_BITS = 58;              // |z| < 2^FX_BITS
constexpr int FX_EMIN = 1023 - 900;      // biased exponents of a block's largest value
constexpr int FX_EMAX = 1023 + 900;

// the biased exponent's word of a value (its maximum over a block is the block's)
__device__ __forceinline__ unsigned fx_word(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
// exponent of a block from the largest word
__device__ __forceinline__ int fx_exp(unsigned word) {
    const int e = (int)(word >> 20);
    return e < FX_EMIN ? FX_EMIN : e;
}

// x of a block with exponent e, in units of 2^(e - 1022 - bits): |z| < 2^bits, cut towards zero
__device__ __forceinline__ long long fx_from(double x, int e, int bits) {
    const unsigned long long b = fbits(x);
    const unsigned long long m = (b & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
    const int s = e - (int)((b >> 52) & 0x7ff);
    const long long z = (long long)((m << (bits - 53)) >> (s < 63 ? s : 63));
    return (long long)b < 0 ? -z : z;
}
__device__ __forceinline__ Fx fx_limbs(long long z) {
    Fx r;
    r.lo = ((int)(unsigned)z << 4) >> 4;
    r.hi = (int)((z - r.lo) >> 28);
    return r;
}
__device__ __forceinline__ Fx fx_neg(Fx a) { return {-a.hi, -a.lo}; }

// sum of products, in units of 2^28: a 2^28 + b
struct FxSum {
    long long a = 0, b = 0;
    __device__ __forceinline__ void add(Fx x, Fx y) {
        a += (long long)x.hi * y.hi;
        b += (long long)x.hi * y.lo;
        b += (long long)x.lo * y.hi;
    }
    // in units of 2^56, rounded
    __device__ __forceinline__ long long top() const { return a + ((b + (1LL << 27)) >> 28); }
};

// h 2^e, rounded to nearest: integer operations only (the conversion instruction is
// FP64 work).  The result's exponent must be normal.
__device__ __forceinline__ double fx_double(long long h, int e) {
    const unsigned long long a = h < 0 ? (unsigned long long)-h : (unsigned long long)h;
    if (a == 0) return 0.0;
    const int lz = __clzll((long long)a);
    const unsigned long long m = a << lz;
    const unsigned long long mant = (m >> 11) + ((m >> 10) & 1ULL);   // [2^52, 2^53]
    const unsigned long long bits = mant + ((unsigned long long)(63 - lz + e + 1022) << 52);
    return __longlong_as_double((long long)(bits | ((unsigned long long)h & 0x8000000000000000ULL)));
}

}  // namespace ffe
