// FP64 values as scaled 64-bit integers, one scale per complex number, for the
// vector kernels that the FP64 pipe would bound (device code):
//  - a component with largest biased exponent e is an integer in units of
//    2^(e-1081), below 2^59 (fix_conv: kFixFrac = 58); a coefficient one in
//    units of 2^(e-1084), below 2^62;
//  - their product, hi*hi and the two cross terms of balanced 32-bit limbs,
//    has scale S = e + e', units of 2^(S-2101), and is below 2^57 (a complex
//    one below 2^58).  A component with exponent e is the same integer at
//    scale e + 1020.
// The error of a sum is relative to the modulus of its largest complex term,
// as in complex arithmetic with complex coefficients; the smaller of re and im
// does not keep 53 bits of its own.
// Values outside the ranges below (zeros are inside) take FP64 arithmetic:
// components 2^(-423..478), coefficients 2^(-200..201).
#pragma once

#include "hop_fix.cuh"

namespace wl {

constexpr int kShiftMinExp = 600, kShiftMaxExp = 1500;
constexpr int kShiftCoefMin = 823, kShiftCoefMax = 1223;
constexpr int kShiftUnit = 1020;   // scale of a component: exponent + this

// Largest biased exponent of v, zero as the smallest one; special: outside the range.
__device__ __forceinline__ int shift_exp(cx<double> v, int lo, int hi, bool &special)
{
    const int A = fix_absmax(0, make_double2(v.re, v.im)), e = A >> 20;
    special = special || e > hi || (e < lo && (A | fix_lobits(make_double2(v.re, v.im))) != 0);
    return max(e, lo);
}
__device__ __forceinline__ i64 shift_conv(double x, int e)
{
    int neg = 0;
    const i64 q = fix_conv(x, e, 0, neg);
    return q - neg;
}

// v 2^(S-2101), rounded to FP64 (|v| < 2^62; never subnormal within the ranges).
__device__ __forceinline__ double shift_out(i64 v, int S)
{
    const i64 m = v >> 63;
    const u64 a = (u64)((v ^ m) - m);
    const int n = __clzll((i64)a) - 1;
    const u64 mant = ((a << n) + (1ull << 9)) >> 10;
    const u64 bits = mant + ((u64)(unsigned)(S - kShiftUnit + 3 - n) << 52);
    return a ? __longlong_as_double((i64)(bits | ((u64)m & (1ull << 63)))) : 0.0;
}

}  // namespace wl
