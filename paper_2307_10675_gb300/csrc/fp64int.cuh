// Exact integer forms of FP64 conversions, comparisons and sign changes.
//
// An SM sub-partition of this part takes 64 clocks for any FP64 warp
// instruction, whatever the number of active lanes (measured: 64.6 clocks for a
// dependent FMA at 1 to 32 lanes), and conversions, comparisons and |x| run on
// the same pipe (92 to 104 clocks in a chain).  The integer pipe does them in a
// few instructions with the same result.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ifci {

__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ long long dmag(double x) { return dbits(x) & 0x7FFFFFFFFFFFFFFFll; }   // |x| orders like its bits
__device__ __forceinline__ int dexp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
// x with the sign bit flipped where neg = 0x80000000
__device__ __forceinline__ double dflip(double x, uint32_t neg) {
    return __hiloint2double(__double2hiint(x) ^ (int)neg, __double2loint(x));
}
// x < y as signed integer keys (-0 orders below +0)
__device__ __forceinline__ long long dkey(double x) {
    const long long b = dbits(x);
    return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll);
}

// (double)f: a normal number is re-biased, anything else takes the conversion
__device__ __forceinline__ double f2d(float f) {
    const uint32_t b = __float_as_uint(f), e = b >> 23 & 0xFFu;
    if (e == 0u || e == 255u) return b << 1 ? (double)f : __hiloint2double((int)b, 0);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// (float)x, round to nearest even: where the result is a normal number the
// mantissa is rounded by an integer addition, anything else takes the conversion
__device__ __forceinline__ float d2f(double x) {
    const long long m = dmag(x);
    const int e = dexp_field(x);
    if (e < 1023 - 126 || e > 1023 + 126) return (float)x;
    const unsigned long long r = (unsigned long long)m + 0x0FFFFFFFull + ((unsigned long long)m >> 29 & 1ull);
    const uint32_t b = (uint32_t)(r >> 29) - (uint32_t)((1023 - 127) << 23);
    return __uint_as_float(b | ((uint32_t)__double2hiint(x) & 0x80000000u));
}

}  // namespace ifci
