// Conversions, reciprocals and tests of FP64 numbers in integer and FP32 arithmetic (device code;
// no other header, so that tests/test_bits.py can compile it for the host).
#pragma once

namespace wf {

// FP64 runs at 1/64 of the FP32 rate, and conversions to and from it as slowly as arithmetic: a
// pass over pixels or a_lm with a handful of FP64 operations per element is bound by them before
// it is bound by memory (one operation per element of 12 nside^2 pixels: 85 us at nside 2048).

// (double)f in integer arithmetic
__device__ __forceinline__ double widen(float f)
{
    const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
    if (a - 0x00800000u >= 0x7f000000u && a != 0u) return (double)f;  // denormal, infinity, NaN
    return a == 0u ? __hiloint2double((int)u, 0) : __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(a << 29));
}

// (float)v, rounded to nearest even, in integer arithmetic
__device__ __forceinline__ float narrow(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e - 897u >= 253u) return (float)v;  // zero, not a normal FP32 number, or next to the largest
    const unsigned f = ((hi & 0x7fffffffu) - 0x38000000u) << 3 | lo >> 29, rest = lo & 0x1fffffffu;
    const unsigned up = rest > 0x10000000u || (rest == 0x10000000u && (f & 1u)) ? 1u : 0u;  // (a carry raises the exponent)
    return __uint_as_float((hi & 0x80000000u) | (f + up));
}

// 1 / v to within 0.51 units in the last place by three FP64 operations: with y the FP32
// reciprocal of the leading 24 bits of v, r = 1 - v y is below 2^-21, and
// 1 / v = y (1 + r + r^2 + ...), the first term left out below 2^-63
__device__ __forceinline__ double inverse(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e - 23u > 2000u) return 1.0 / v;  // zero, infinity, NaN, or 1 / v next to the ends of the range
    const float f = __frcp_rn(__uint_as_float(0x3f800000u | (hi & 0xfffffu) << 3 | lo >> 29));  // (0.5, 1]
    const unsigned u = __float_as_uint(f);
    const double y = __hiloint2double((int)((hi & 0x80000000u) | ((u >> 3) + 0x38000000u + ((1023u - e) << 20))), (int)(u << 29));
    const double r = fma(-v, y, 1.0);
    return fma(y, fma(r, r, r), y);
}

__device__ __forceinline__ unsigned long long bits64(double v) { return (unsigned long long)__double_as_longlong(v); }

// 0 < v < infinity, by its bits (unsigned: -0.0 is the least signed number)
__device__ __forceinline__ bool positive_finite(double v)
{
    return bits64(v) - 1ULL < 0x7fefffffffffffffULL;
}
__device__ __forceinline__ bool finite_bits(double v)
{
    return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

// v > 0 (infinity included), and v != 0 (NaN included)
__device__ __forceinline__ bool positive(double v) { return bits64(v) - 1ULL < 0x7ff0000000000000ULL; }
__device__ __forceinline__ bool nonzero(double v) { return bits64(v) << 1 != 0; }

}  // namespace wf
