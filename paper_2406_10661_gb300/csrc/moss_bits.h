// Comparisons of doubles on their bit patterns, as plain integer functions
// that a host compiler takes too.  Doubles >= 0 are ordered like their bits;
// the differences are formed without sign, where they wrap (with sign they
// would leave the range for x < 0).
#pragma once

#ifdef __CUDACC__
#define MOSS_BITS_FN __host__ __device__ __forceinline__
#else
#define MOSS_BITS_FN inline
#endif

namespace moss {

// x > t for t >= +0, false for NaN; xb, tb: the bits of x and t
MOSS_BITS_FN bool bits_gt(unsigned long long xb, unsigned long long tb) {
    return xb - tb - 1ull < 0x7ff0000000000000ull - tb;
}

// |x| < band * scale is false whatever their fractions are; from the upper
// halves: |x| >= 2^ex, band * scale <= 2^(eb + es + 2), exponents biased by 1023
MOSS_BITS_FN bool bits_not_within(int x_hi, int band_hi, int scale_hi) {
    const int ex = (x_hi >> 20) & 0x7ff, eb = (band_hi >> 20) & 0x7ff, es = (scale_hi >> 20) & 0x7ff;
    return ex + 1023 >= eb + es + 2;
}

}  // namespace moss
