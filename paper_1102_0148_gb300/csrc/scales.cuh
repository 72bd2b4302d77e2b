// Pre-cast scale of one antenna and channel from its mean power, and the
// pair order of the outputs (device functions).
#pragma once

#include <cstdint>

namespace gbcorr {

// Upper triangle of n antennas, row-major with autos: first pair of row i, and
// the row of pair pl.
__device__ __forceinline__ int triangle_start(int i, int n) { return i * n - i * (i - 1) / 2; }
__device__ __forceinline__ int triangle_row(int pl, int n) {
    const float b = 2.0f * n + 1.0f;
    int i = (int)(0.5f * (b - sqrtf(b * b - 8.0f * pl)));
    i = min(max(i, 0), n - 1);
    while (pl < triangle_start(i, n)) --i;             // the root is rounded: a step or two off
    while (i + 1 < n && pl >= triangle_start(i + 1, n)) ++i;
    return i;
}

// 2^rint(log2(target / sqrt(power / 2))), power = mean |Y|^2 and target a power
// of two; a silent channel keeps scale 1.  With power = m 2^x, 1 <= m < 2, the
// exponent is log2(target) - floor(x / 2), rounded to nearest, unless m is 1 or
// next to 2, where the rounding is a tie or the logarithm's own rounding
// decides: those (and targets, subnormals, infinities and NaN outside the
// shortcut's range) take the FP64 functions, which run at a few per clock and
// SM here.
__device__ __forceinline__ float scale_for(double power, float target) {
    if (!(power > 0.0)) return 1.0f;
    const long long b = __double_as_longlong(power);
    const int x = (int)(b >> 52) - 1023;
    const long long m = b & 0xfffffffffffffll;
    const int t = __float_as_int(target);
    if ((t & 0x7fffff) == 0 && t > 0x00800000 && t < 0x7f800000 && x > -1000 && x < 1024 && m > 64 &&
        m < 0xfffffffffffffll - 64) {
        const int e = ((t >> 23) - 127) - (x >> 1);
        return __int_as_float((min(max(e, -60), 60) + 127) << 23);
    }
    const double e = rint(log2((double)target / sqrt(power * 0.5)));
    return (float)exp2(fmin(fmax(e, -60.0), 60.0));
}

}  // namespace gbcorr
