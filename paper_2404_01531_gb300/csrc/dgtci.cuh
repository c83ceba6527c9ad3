// Troubled-cell indicator (Sec. III.C.3) of one DG element in shared memory:
// ratio = sqrt(sum u^^2 / sum u^2) with u = |B~| and u^ = u - (Pi x Pi x Pi) u.
#pragma once
#include "ffe_internal.h"
#include "fixed.cuh"

namespace ffe {

// mag: u at the thread's node (act: it has one); the result is thread 0's.  Every
// thread of the CTA calls it (it holds barriers).  z [3][nn] is scratch, *word is zero
// on entry, red holds two doubles.  The low-pass lines run in fixed point (fixed.cuh),
// and two warps add the squares, in a fixed order: 5 FP64 operations a node instead
// of 32.  Fields beyond 2^+-511, whose squares leave FP64's range, count as smooth.
template <int P, int NT>
__device__ __forceinline__ double indicator_ratio(const Tables& T, bool act, double mag, long long* z, unsigned* word, double* red) {
    constexpr int np1 = P + 1, nl = np1 * np1, nn = nl * np1, NW = NT / 32;
    const int tid = threadIdx.x;
    const unsigned w = __reduce_max_sync(0xffffffffu, act ? fx_word(mag) : 0u);
    if ((tid & 31) == 0) atomicMax(word, w);
    __syncthreads();
    const unsigned top = *word;
    const bool inside = top >= (1023u - 511u) << 20 && top < (1023u + 511u) << 20;
    const int e = fx_exp(top), bits = T.fx_pi;
    const int c[3] = {tid % np1, (tid / np1) % np1, tid / nl};
    const long long z0 = act && inside ? fx_from(mag, e, bits) : 0;
    if (act) z[tid] = z0;
    __syncthreads();
    long long low = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int stride = k == 0 ? 1 : (k == 1 ? np1 : nl);
        if (act) {
            const long long* line = z + k * nn + tid - c[k] * stride;
            FxSum s;
#pragma unroll
            for (int m = 0; m < np1; ++m) s.add(T.FxPi[c[k]][m], fx_limbs(line[m * stride]));
            low = s.top();
            if (k < 2) z[(k + 1) * nn + tid] = low;
        }
        if (k < 2) __syncthreads();
    }
    // the squares, in place of the fields that nobody reads any more (z[2] is being read)
    double* num = (double*)z;
    double* den = (double*)(z + nn);
    if (act) {
        const double uh = inside ? fx_double(z0 - low, e - 1022 - bits) : 0.0;
        num[tid] = uh * uh;
        den[tid] = inside ? mag * mag : 0.0;
    }
    __syncthreads();
    for (int q = tid >> 5; q < 2; q += NW) {
        const double* x = q ? den : num;
        double s = 0.0;
        for (int t = tid & 31; t < nn; t += 32) s += x[t];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if ((tid & 31) == 0) red[q] = s;
    }
    __syncthreads();
    return tid == 0 && red[1] > 0.0 ? sqrt(red[0] / red[1]) : 0.0;
}

}  // namespace ffe
