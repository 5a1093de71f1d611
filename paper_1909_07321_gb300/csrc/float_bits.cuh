// Sums and conversions of floats on their bits, where the FP64 unit (2
// operations per clock and SM) is what holds a kernel: the same results to
// the bit as the plain FP64 operations.
#pragma once

#include <stdint.h>

namespace rmgb {

// s = v[0] + v[1] + ... (FP64, in this order) of n <= 8 floats. The FP64 unit
// does 2 additions or conversions per clock and SM, and the 17 of an entry of 8
// segments held the reduction at 5.3 ms for 256 energies of 1000 channels
// (2.05 with this; the partials' traffic is 1.0). While the exponents of the
// nonzero values lie within 26 of one another, every partial sum is a multiple
// of the smallest unit below 2^53 of it, so the FP64 sum is exact: the
// mantissas are then summed as integers and converted once. Otherwise (and for
// subnormal or non-finite values) the plain sum is taken.
__device__ __forceinline__ double pe_sum(const float (&v)[8], int n)
{
    int lo = 255, hi = 0;
    bool odd = false;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (q >= n) continue;
        const uint32_t u = __float_as_uint(v[q]) & 0x7fffffffu;
        const int e = (int)(u >> 23);
        odd = odd || e == 255 || (e == 0 && u != 0u);
        if (u != 0u) {
            lo = min(lo, e);
            hi = max(hi, e);
        }
    }
    if (odd || hi - lo > 26) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < n) s += (double)v[q];
        return s;
    }
    long long sum = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (q >= n) continue;
        const uint32_t u = __float_as_uint(v[q]);
        const int e = (int)((u >> 23) & 255u);
        const int m = e ? (int)((u & 0x7fffffu) | 0x800000u) : 0;
        sum += (long long)((u >> 31) ? -m : m) * (long long)(1 << (e ? e - lo : 0));
    }
    if (sum == 0) return 0.0;
    const double d = (double)sum;   // exact
    return __hiloint2double(__double2hiint(d) + ((lo - 150) << 20), __double2loint(d));
}

// (float)v without the FP64 unit: round to nearest even on the bits where the
// result is a normal float, the conversion instruction elsewhere.
__device__ __forceinline__ float to_float(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned mh = hi & 0x7fffffffu;
    // 2^-126 <= |v| < 2^127
    if (mh - 0x38100000u >= 0x47e00000u - 0x38100000u) return (float)v;
    const unsigned t = ((mh - 0x38000000u) << 3) | (lo >> 29);   // exponent and 23 bits
    const unsigned rest = lo << 3;                                // the bits below
    const unsigned up = (rest > 0x80000000u || (rest == 0x80000000u && (t & 1u))) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (t + up));
}

}  // namespace rmgb
