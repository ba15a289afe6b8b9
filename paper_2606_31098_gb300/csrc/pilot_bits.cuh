// FP64 values handled by their words.  A sub-partition of an SM takes one FP64 warp instruction
// per 64 cycles -- comparisons and conversions included, however few lanes are active (measured
// on GB300: a chain of dependent FMAs and four independent ones per step both run at 64 cycles
// each, with 32 lanes or with one) -- and an integer one per cycle or two, so conversions,
// comparisons and truncations that are exact on the words are done there.
#pragma once

#include <cuda_runtime.h>

namespace pilot {

__device__ __forceinline__ unsigned long long bits(double v) { return (unsigned long long)__double_as_longlong(v); }

constexpr unsigned long long kInfBits = 0x7ff0000000000000ull, kOneBits = 0x3ff0000000000000ull;

// a / b with inv close to 1 / b: the product and one correction by its remainder, which FMA
// gives exactly (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", IBM J. Res. Dev. 34(1), 1990).
__device__ __forceinline__ double quotient(double a, double b, double inv) {
    const double q = a * inv;
    return fma(fma(-q, b, a), inv, q);
}

// FP32 to FP64 by moving bits (exact); subnormal and non-finite values by the conversion.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), e = u & 0x7f800000u;
    if (e == 0u || e == 0x7f800000u) return u == 0u ? 0.0 : (double)f;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen(unsigned char v) { return widen((float)v); }

// FP64 to FP32, to nearest even, on the bits; outside the normal FP32 range by the conversion.
__device__ __forceinline__ float narrow(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e < 897u || e > 1150u) return (bits(v) << 1) == 0ull ? __uint_as_float(hi) : (float)v;
    const unsigned m = ((hi & 0x7fffffffu) - 0x38000000u) << 3 | lo >> 29;   // exponent and the upper 23 bits
    const unsigned rest = lo & 0x1fffffffu;                                   // the 29 dropped ones
    const unsigned up = rest > 0x10000000u || (rest == 0x10000000u && (m & 1u));
    return __uint_as_float((hi & 0x80000000u) | (m + up));
}

// 0 <= v <= top (top >= 0, no NaN): the unsigned order of the words
__device__ __forceinline__ bool within(double v, double top) { return bits(v) <= bits(top); }

// Non-negative v < 2^31: its integer part, and the same as FP64.
__device__ __forceinline__ int whole_part(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e = (int)(hi >> 20) - 1023;
    return e < 0 ? 0 : (int)((((hi & 0xfffffu) | 0x100000u) << 11 | lo >> 21) >> (31 - e));
}
__device__ __forceinline__ double as_double(int i) {     // 0 <= i
    return i < (1 << 24) ? widen((float)i) : (double)i;
}

// 2^k v for a normal v whose scaled value is normal too
__device__ __forceinline__ double scale2(double v, int k) {
    return __hiloint2double(__double2hiint(v) + (k << 20), __double2loint(v));
}

}  // namespace pilot
