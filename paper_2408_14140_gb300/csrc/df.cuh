// Double-float arithmetic for the FP64-field pass sums.
//
// GB300 issues two FP64 operations per clock per SM against 128 FP32 (or
// INT32) operations, so the FP64 forms of the interpolation and gather sums
// were bound by the FP64 pipe.  Here a double value is carried as an
// unevaluated pair of floats hi + lo (Dekker 1971, "A floating-point
// technique for extending the available precision"), with
//   * products from the FMA remainder: fma(a, b, -a*b) is the exact error of
//     the float product a*b (the cross terms a.hi*b.lo + a.lo*b.hi are
//     added, a.lo*b.lo is dropped);
//   * sums from Knuth's TwoSum (the exact rounding error of a float sum from
//     six additions), followed by a renormalisation of (hi, lo);
//   * conversions between double and float pairs by bit manipulation on the
//     integer pipe: a double's top 24 significant bits (truncated) form hi and
//     its next 29 bits, rounded to 24, form lo, so a split is within 2^-47 of
//     the double (|x| >= 2^-74; smaller magnitudes keep only hi, and values
//     below 2^-126 become 0).
// Every float operation is an explicit _rn intrinsic, so the compiler cannot
// contract a product into a following sum (which would break TwoSum).
// The pair carries about 48 significant bits; sums of a few dozen terms stay
// within ~1e-13 of the exact result, inside the library's 1e-12 gate for
// FP64 fields.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gbib {

// double -> (hi, lo), integer pipe only.  Outside [2^-74, 2^128): below 2^-126
// a zero, below 2^-74 no low part, above (and Inf, NaN) the class is kept.
__device__ __forceinline__ float2 df_split(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned h32 = (unsigned)(b >> 32), l32 = (unsigned)b;
    const unsigned mag = h32 & 0x7fffffffu, sgn = h32 & 0x80000000u;
    // the exponent rebiased from 1023 to 127 and the top 23 stored bits
    const unsigned hi = __funnelshift_l(l32, mag - (896u << 20), 3) | sgn;
    if (mag - (949u << 20) < (202u << 20)) {
        // the remaining 29 bits r, worth r * 2^(e - 1075), e the double's exponent
        const float scale = __uint_as_float((hi & 0xff800000u) - (52u << 23));
        return make_float2(__uint_as_float(hi), __fmul_rn(__uint2float_rn(l32 & 0x1fffffffu), scale));
    }
    const unsigned e = mag >> 20;
    if (e <= 896) return make_float2(__uint_as_float(sgn), __uint_as_float(sgn));
    if (e >= 1151) {
        const unsigned nan = (e == 2047 && ((h32 & 0xfffffu) | l32)) ? 0x400000u : 0u;
        return make_float2(__uint_as_float(sgn | 0x7f800000u | nan), 0.0f);
    }
    return make_float2(__uint_as_float(hi), 0.0f);
}

// (float)x, and that with the rest (float)(x - (float)x): round to nearest, the
// bits the conversions give, on the integer pipe (a double's conversions run at
// the FP64 rate; the conversions serve what is outside FP32's normal range,
// out of line, where the compiler cannot run them for every value).
static __device__ __noinline__ float df_round_rare(double x) { return (float)x; }
static __device__ __noinline__ float2 df_round_pair_rare(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}
// the magnitude's top 24 bits rounded to nearest (even), exponent rebiased to
// FP32's; mag and l32 the double's words, its sign cleared
__device__ __forceinline__ unsigned df_round_bits(unsigned mag, unsigned l32, unsigned &up) {
    const unsigned t = __funnelshift_l(l32, mag - (896u << 20), 3);
    up = (l32 & 0x1fffffffu) + (t & 1u) > 0x10000000u ? 1u : 0u;
    return t + up;
}
__device__ __forceinline__ float df_round(double x) {
    const unsigned h32 = (unsigned)__double2hiint(x), l32 = (unsigned)__double2loint(x);
    const unsigned mag = h32 & 0x7fffffffu, sgn = h32 & 0x80000000u;
    if ((mag | l32) == 0) return __uint_as_float(sgn);
    if (mag - (897u << 20) >= (253u << 20)) return df_round_rare(x);
    unsigned up;
    return __uint_as_float(df_round_bits(mag, l32, up) | sgn);
}
__device__ __forceinline__ float2 df_round_pair(double x) {
    const unsigned h32 = (unsigned)__double2hiint(x), l32 = (unsigned)__double2loint(x);
    const unsigned mag = h32 & 0x7fffffffu, sgn = h32 & 0x80000000u;
    if ((mag | l32) == 0) return make_float2(__uint_as_float(sgn), 0.0f);
    if (mag - (949u << 20) >= (201u << 20)) return df_round_pair_rare(x);
    unsigned up;
    const unsigned r = df_round_bits(mag, l32, up);
    // what rounding left, in units of 2^(e - 1075), e the double's exponent
    int rest = (int)(l32 & 0x1fffffffu) - (int)(up << 29);
    rest = sgn ? -rest : rest;
    const float scale = __uint_as_float(((mag >> 20) - 948u) << 23);
    return make_float2(__uint_as_float(r | sgn), __fmul_rn(__int2float_rn(rest), scale));
}

// float -> double, exact, integer pipe only (float subnormals become 0).
__device__ __forceinline__ double df_widen(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned sgn = b & 0x80000000u;
    const unsigned e = (b >> 23) & 0xffu;
    const unsigned m = b & 0x7fffffu;
    unsigned h32, l32;
    if (e == 0) {
        h32 = sgn;
        l32 = 0;
    } else if (e == 255) {
        h32 = sgn | 0x7ff00000u | (m >> 3) | (m ? 0x80000u : 0u);
        l32 = 0;
    } else {
        h32 = sgn | ((e + 896u) << 20) | (m >> 3);
        l32 = m << 29;
    }
    return __hiloint2double((int)h32, (int)l32);
}

// (hi, lo) -> double: one FP64 addition.
__device__ __forceinline__ double df_to_double(float2 v) { return __dadd_rn(df_widen(v.x), df_widen(v.y)); }

// Renormalise s + e (|e| small against s) into a pair.
__device__ __forceinline__ float2 df_fast_two_sum(float s, float e) {
    const float h = __fadd_rn(s, e);
    return make_float2(h, __fsub_rn(e, __fsub_rn(h, s)));
}

// a * b of two pairs.
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, e);
    e = __fmaf_rn(a.y, b.x, e);
    return df_fast_two_sum(p, e);
}

// a + b of two pairs: TwoSum of the high parts, the low parts added to its
// error, renormalised.
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
    const float s = __fadd_rn(a.x, b.x);
    const float bb = __fsub_rn(s, a.x);
    const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bb)), __fsub_rn(b.x, bb));
    return df_fast_two_sum(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}

__device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }

// a * k for a power of two k: exact.
__device__ __forceinline__ float2 df_scale(float2 a, float k) { return make_float2(__fmul_rn(a.x, k), __fmul_rn(a.y, k)); }

// Square root of a pair a > 0 (a.x a normal float): one Newton (Heron) step
// q = q0 + (a - q0^2) / (2 q0) from the FP32 root q0, the residual from the
// exact FMA square (a.x - q0^2 is exact: q0^2 is within a factor 2 of a.x).
// The start's relative error below 2^-24 leaves about 2^-47.
__device__ __forceinline__ float2 df_sqrt(float2 a) {
    const float q0 = __fsqrt_rn(a.x);
    const float p = __fmul_rn(q0, q0);
    const float pe = __fmaf_rn(q0, q0, -p);
    const float res = __fadd_rn(__fsub_rn(__fsub_rn(a.x, p), pe), a.y);
    return df_fast_two_sum(q0, __fmul_rn(res, __fdiv_rn(0.5f, q0)));
}

// Running sum of pair products, renormalised after every term.
struct DFAcc {
    float hi, lo;
    __device__ __forceinline__ DFAcc() : hi(0.0f), lo(0.0f) {}
    __device__ __forceinline__ void add_prod(float2 a, float2 b) {
        const float p = __fmul_rn(a.x, b.x);
        float pe = __fmaf_rn(a.x, b.x, -p);
        pe = __fmaf_rn(a.x, b.y, pe);
        pe = __fmaf_rn(a.y, b.x, pe);
        // TwoSum(hi, p)
        const float s = __fadd_rn(hi, p);
        const float bb = __fsub_rn(s, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
        const float2 r = df_fast_two_sum(s, __fadd_rn(lo, __fadd_rn(err, pe)));
        hi = r.x;
        lo = r.y;
    }
    __device__ __forceinline__ float2 get() const { return make_float2(hi, lo); }
    __device__ __forceinline__ double value() const { return df_to_double(get()); }
};

}  // namespace gbib
