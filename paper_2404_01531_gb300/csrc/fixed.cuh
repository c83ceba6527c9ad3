// Line contractions of the DG kernels in block fixed point, on the integer pipes.
//
// A contraction sum_m D_m u_m along a line of an element is FP64 work of 6 slots a
// value on a pipe with 2 lanes a clock and SM; the integer multiply-adds run 32
// lanes or more.  The values of a variable are therefore scaled by one power of two
// per element and held as integers of up to 60 bits in two limbs, z = hi 2^30 + lo
// with |lo| <= 2^29; the operator's rows likewise.  A product is three
// 32 x 32 -> 64 bit multiply-adds into two 64-bit sums (hi hi into a, hi lo + lo hi
// into b; lo lo stays below the quantum), exact until the one rounding of the result.
// Sums of several variables or axes are formed at the scale of the largest of them.
//
// Error: the operands are cut at 2^-59 of the variable's largest value in the element
// and 2^-60 of the operator's largest row sum, where the FP64 sum rounds each product
// and partial sum at 2^-53 of their size.  So the sum is the more accurate one on a
// line that holds values of 2^-6 of the variable's largest in the element or more, and
// the less accurate one on lines far below that (absolute error 2^-58 of the largest).
// The sizes of other variables and, on boxes, the widths along other axes do not
// enter.  Elements with a variable whose largest value is 2^900 or more, not finite,
// or below 2^-800 but not zero take the FP64 form (fx_inside).
#pragma once
#include "ffe_internal.h"
#include "fp64util.cuh"

namespace ffe {

constexpr int FX_BITS = 60;              // |z| < 2^FX_BITS
constexpr int FX_EMIN = 1023 - 800;      // biased exponents of a variable's largest value
constexpr int FX_EMAX = 1023 + 900;

// the biased exponent's word of a value (its maximum over an element is the largest
// value's); not zero where the value is not
__device__ __forceinline__ unsigned fx_word(double x) {
    const unsigned long long m = fbits(x);
    return ((unsigned)(m >> 32) & 0x7fffffffu) | ((unsigned)m != 0u);
}
// exponent of a variable from its largest word, and whether fixed point holds it
__device__ __forceinline__ int fx_exp(unsigned word) {
    const int e = (int)(word >> 20);
    return e < FX_EMIN ? FX_EMIN : e;
}
__device__ __forceinline__ bool fx_inside(unsigned word) {
    return word == 0u || word - ((unsigned)FX_EMIN << 20) < (unsigned)(FX_EMAX - FX_EMIN) << 20;
}
// Largest words of N variables over a warp, added to top[N] (shared); every lane calls it
template <int N>
__device__ __forceinline__ void fx_largest(const unsigned* word, unsigned* top) {
    static_assert(N <= 32, "a lane per variable");
    unsigned mine = 0;
#pragma unroll
    for (int v = 0; v < N; ++v) {
        const unsigned w = __reduce_max_sync(0xffffffffu, word[v]);
        if ((int)(threadIdx.x & 31) == v) mine = w;
    }
    if ((threadIdx.x & 31) < N && mine) atomicMax(top + (threadIdx.x & 31), mine);
}

// x of a variable with exponent e, in units of 2^(e - 1022 - bits): |z| < 2^bits, cut towards zero
__device__ __forceinline__ long long fx_from(double x, int e, int bits) {
    const unsigned long long b = fbits(x);
    const unsigned long long m = (b & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
    const int s = e - (int)((b >> 52) & 0x7ff);
    const long long z = (long long)((m << (bits - 53)) >> (s < 63 ? s : 63));
    return (long long)b < 0 ? -z : z;
}
__device__ __forceinline__ Fx fx_limbs(long long z) {
    Fx r;
    r.lo = ((int)((unsigned)z << 2)) >> 2;
    r.hi = (int)((z - r.lo) >> 30);
    return r;
}

// sum of products, in units of 2^30: a 2^30 + b
struct FxSum {
    long long a = 0, b = 0;
    __device__ __forceinline__ void add(Fx x, Fx y) {
        a += (long long)x.hi * y.hi;
        b += (long long)x.hi * y.lo;
        b += (long long)x.lo * y.hi;
    }
    // in units of 2^60, rounded
    __device__ __forceinline__ long long top() const { return a + ((b + (1LL << 29)) >> 30); }
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
