// Line FFTs of the fluid step in registers, for FP32 and for FP64 fields.
//
// Form: Stockham passes of radix up to E with E complex points per thread
// (Govindaraju et al. 2008, "High performance discrete Fourier transforms on
// graphics processors"): the thread t of a line holds the points t + TPL m
// (TPL = N / E threads per line) before and after the transform, and the
// passes exchange through shared memory.  Two arithmetics:
//
//  * Fp32: float pairs.
//  * Fx64: 64-bit block fixed point, the transform of FP64 fields.  GB300
//    issues 2 FP64 operations per clock and SM (a warp instruction holds the
//    pipe for 16 clocks) but 64 or more integer ones.  A line's components
//    are scaled by one power of two, so that the sum of their magnitudes stays
//    below 2^61 and no sum of the transform can overflow, and rounded to
//    integers; butterflies are then exact 64-bit additions, and only the
//    products with twiddle factors (Q62) round, where an FP64 transform rounds
//    every addition to 2^-53 of its result.  A product leaves out those of the
//    low halves, up to one unit each: with the rounding half, a component of a
//    complex product is off by at most 2.5 units (0.6 in the mean square), a
//    product with a real constant by 1.5.  (A scale by the
//    largest component and N, one reduction less, wastes log2 N bits on a line
//    of a few large points, as smooth fields' spectra are: 5.5e-16 against
//    3.0e-16 in the predictor's u* at 16x16x256.)  The result goes back to FP64
//    with one rounding.  A line with a NaN or an infinity gives NaN.
#pragma once

#include "gbib_internal.cuh"

namespace gbib {

constexpr int kRoots = 2048;              // (cos, sin)(2 pi k / kRoots), for the symbols

// ---------------------------------------------------------------------------
// arithmetic
// ---------------------------------------------------------------------------
struct Fx64On32;
struct Fp32 {
    using Pressure = Fx64On32;           // the pressure solve's x passes
    using Real = float;                  // the field's element
    using C = float2;                    // a point in registers
    using Mem = float2;                  // a point in memory
    using W = float2;                    // a twiddle factor
    static constexpr bool kFixed = false;
    static __host__ __device__ constexpr int points(int logN) {
        return logN == 7 || logN == 8 || logN == 10 ? 16 : 8;
    }
    // adjacent lines of one CTA in the strided passes: 128-byte rows (64 for
    // long lines, which fill the CTA's threads and shared memory)
    static __host__ __device__ constexpr int lanes(int logN) { return logN >= 9 ? 8 : 16; }
};
struct Fx64 {
    using Pressure = Fx64;
    using Real = double;
    using C = longlong2;
    using Mem = double2;
    using W = int4;                      // (re hi, re lo, im hi, im lo) in Q62, signed halves
    static constexpr bool kFixed = true;
    static __host__ __device__ constexpr int points(int) { return 8; }
    static __host__ __device__ constexpr int lanes(int logN) { return logN >= 10 ? 4 : 8; }
};

// Fx64's arithmetic on FP32 values: the x passes of the FP32 pressure solve.
// They bring the error of the pressure's nearly checkerboard modes down to
// what the right-hand side's own rounding leaves (the first pass spreads its
// rounding over all modes, and these are amplified most), and the last pass
// adds none to the gradient.
struct Fx64On32 : Fx64 {
    using Real = float;
    using Mem = float2;
};

__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ longlong2 operator+(longlong2 a, longlong2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ longlong2 operator-(longlong2 a, longlong2 b) { return {a.x - b.x, a.y - b.y}; }

// a times -i (forward) or +i (inverse)
template <bool INV, typename C> __device__ __forceinline__ C rot90(C a) {
    return INV ? C{-a.y, a.x} : C{a.y, -a.x};
}

// Balanced halves: a = hi 2^32 + lo with lo signed.
struct Halves {
    int hi, lo;
};
__device__ __forceinline__ Halves halves(long long a) {
    const int lo = (int)(unsigned)a;
    return {(int)(a >> 32) + (int)((unsigned)lo >> 31), lo};
}
// S 2^64 + T 2^32 (T with its rounding half) as a Q62 product's integer
__device__ __forceinline__ long long q62(long long S, long long T) { return (S << 2) + (T >> 30); }
constexpr long long kQ62Half = 1LL << 29;

__device__ __forceinline__ long long fx_mul(long long a, int bh, int bl) {
    const Halves h = halves(a);
    return q62((long long)h.hi * bh, (long long)h.hi * bl + ((long long)h.lo * bh + kQ62Half));
}

template <bool INV> __device__ __forceinline__ float2 cmulw(float2 a, float2 w) {
    const float s = INV ? -w.y : w.y;
    return {fmaf(a.x, w.x, -(a.y * s)), fmaf(a.x, s, a.y * w.x)};
}
template <bool INV> __device__ __forceinline__ longlong2 cmulw(longlong2 a, int4 w) {
    const Halves x = halves(a.x), y = halves(a.y);
    const int ih = INV ? -w.z : w.z, il = INV ? -w.w : w.w, nh = -ih, nl = -il;
    const long long sr = (long long)x.hi * w.x + (long long)y.hi * nh;
    const long long si = (long long)x.hi * ih + (long long)y.hi * w.x;
    const long long tr = (long long)x.hi * w.y + ((long long)x.lo * w.x + ((long long)y.hi * nl +
                         ((long long)y.lo * nh + kQ62Half)));
    const long long ti = (long long)x.hi * il + ((long long)x.lo * ih + ((long long)y.hi * w.y +
                         ((long long)y.lo * w.x + kQ62Half)));
    return {q62(sr, tr), q62(si, ti)};
}

// a times the real constants cos(pi/4), cos(pi/8), sin(pi/8) in Q62 halves
struct Q62Const {
    int hi, lo;
};
constexpr Q62Const q62_const(long long v) {
    return {(int)((v + 0x80000000LL) >> 32), (int)(v - (((v + 0x80000000LL) >> 32) << 32))};
}
constexpr long long kHalfRoot = 3260954456333195553LL;  // round(2^62 / sqrt 2)
__device__ __forceinline__ float mul_half_root(float a) { return a * 0.70710678118654752f; }
__device__ __forceinline__ long long mul_half_root(long long a) {
    constexpr Q62Const c = q62_const(kHalfRoot);
    return fx_mul(a, c.hi, c.lo);
}

// ---------------------------------------------------------------------------
// butterflies, natural order in and out
// ---------------------------------------------------------------------------
template <bool INV, typename C> __device__ __forceinline__ void radix2(C &a, C &b) {
    const C t = a - b;
    a = a + b;
    b = t;
}
template <bool INV, typename C> __device__ __forceinline__ void radix4(C &x0, C &x1, C &x2, C &x3) {
    const C a = x0 + x2, b = x0 - x2, c = x1 + x3, d = rot90<INV>(x1 - x3);
    x0 = a + c;
    x1 = b + d;
    x2 = a - c;
    x3 = b - d;
}
// times exp(-+ i pi / 4) and exp(-+ 3 i pi / 4)
template <bool INV, typename C> __device__ __forceinline__ C rot45(C a) {
    return INV ? C{mul_half_root(a.x - a.y), mul_half_root(a.x + a.y)}
               : C{mul_half_root(a.x + a.y), mul_half_root(a.y - a.x)};
}
template <bool INV, typename C> __device__ __forceinline__ C rot135(C a) { return rot90<INV>(rot45<INV>(a)); }

template <bool INV, typename C> __device__ __forceinline__ void radix8(C *x) {
    radix4<INV>(x[0], x[2], x[4], x[6]);
    radix4<INV>(x[1], x[3], x[5], x[7]);
    const C o1 = rot45<INV>(x[3]), o2 = rot90<INV>(x[5]), o3 = rot135<INV>(x[7]);
    const C e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1];
    x[0] = e0 + o0, x[4] = e0 - o0;
    x[1] = e1 + o1, x[5] = e1 - o1;
    x[2] = e2 + o2, x[6] = e2 - o2;
    x[3] = e3 + o3, x[7] = e3 - o3;
}
// FP32 only: two radix-4 stages with the 16th roots between them
template <bool INV> __device__ __forceinline__ void radix16(float2 *x) {
    constexpr float c = 0.92387953251128674f, s = 0.38268343236508977f;
    const float2 w1 = {c, -s}, w3 = {s, -c}, w9 = {-c, s};
#pragma unroll
    for (int k = 0; k < 4; ++k) radix4<INV>(x[k], x[k + 4], x[k + 8], x[k + 12]);
    // point n2 + 4 k1 holds the sub-transform k1 of the residue n2: times w16^(n2 k1)
    x[5] = cmulw<INV>(x[5], w1);
    x[6] = rot45<INV>(x[6]);
    x[7] = cmulw<INV>(x[7], w3);
    x[9] = rot45<INV>(x[9]);
    x[10] = rot90<INV>(x[10]);
    x[11] = rot135<INV>(x[11]);
    x[13] = cmulw<INV>(x[13], w3);
    x[14] = rot135<INV>(x[14]);
    x[15] = cmulw<INV>(x[15], w9);
    float2 y[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        radix4<INV>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) y[k1 + 4 * k2] = x[4 * k1 + k2];
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = y[k];
}
template <int R, bool INV, typename C> __device__ __forceinline__ void radix(C *x) {
    if constexpr (R == 2) radix2<INV>(x[0], x[1]);
    else if constexpr (R == 4) radix4<INV>(x[0], x[1], x[2], x[3]);
    else if constexpr (R == 8) radix8<INV>(x);
    else radix16<INV>(x);
}

// ---------------------------------------------------------------------------
// a line's scale
// ---------------------------------------------------------------------------
// A line's fixed-point units before its first pass and after its last one.  With
// S the sum of its points' magnitudes and X their largest, no value after passes
// of radices R1 ... Rk exceeds min(S, R1 ... Rk X); `sum` and a pass's growth
// are these two as bits above the largest component's exponent, and the unit
// keeps the smaller one below 2^61.  Lines of 256 points and more start in the
// unit of their first pass and are shifted, rounded, to the next pass's: S alone
// left a flat line's points 51 bits of 256 points and 49 of 1024, and the
// rounding of the input was then 0.9 and 2.6 times an FP64 transform's whole
// error (now 0.4 and 0.6).  A line of a few large points has S near X, and its
// shifts are zero.  Shorter lines keep one unit (at most 0.6 times).
struct LineScale {
    int first, last, sum;
};
template <class A, int LOGN> constexpr bool scaled_passes() { return A::kFixed && LOGN >= 8; }
// bits of the bound after passes over sub-transforms of length NS; PAIR: the line
// is the sum of two
template <bool PAIR> constexpr int growth_bits(int ns) {
    int l = 0;
    while ((1 << l) < ns) ++l;
    return l + (PAIR ? 3 : 2);  // |z| <= sqrt 2 of the larger component, that below 2 of its exponent
}
__device__ __forceinline__ longlong2 shift_rounded(longlong2 a, int s) {
    const long long half = (1LL << s) >> 1;
    return {(a.x + half) >> s, (a.y + half) >> s};
}

// ---------------------------------------------------------------------------
// a line's transform: v[m] is the point t + TPL m on entry and on exit
// ---------------------------------------------------------------------------
// `at(p)`: index of the line's point p in the CTA's shared buffer (every
// thread of the CTA calls this together).
template <class A, int LOGN, bool INV, bool PAIR, int NS, typename At>
__device__ __forceinline__ void fft_passes(typename A::C *v, int t, typename A::C *sm, At at,
                                           const typename A::W *__restrict__ tw, int sum) {
    using C = typename A::C;
    constexpr int N = 1 << LOGN, E = A::points(LOGN), TPL = N / E, R = N / NS < E ? N / NS : E, B = E / R;
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int j = t + b * TPL, k = j & (NS - 1);
        C x[R];
#pragma unroll
        for (int i = 0; i < R; ++i) x[i] = v[b + i * B];
        if constexpr (NS > 1) {
#pragma unroll
            for (int i = 1; i < R; ++i) x[i] = cmulw<INV>(x[i], __ldg(tw + (twiddle_offset(NS, R) + i * NS) + k));
        }
        radix<R, INV>(x);
#pragma unroll
        for (int i = 0; i < R; ++i) v[b + i * B] = x[i];
    }
    static_assert(NS == 1 || twiddle_offset(NS, R) >= 0, "a pass without twiddle factors");
    if constexpr (NS * R < N) {
        if constexpr (scaled_passes<A, LOGN>()) {
            constexpr int NEXT = N / (NS * R) < E ? N : NS * R * E;  // the next pass's sub-transforms
            const int shift = min(sum, growth_bits<PAIR>(NEXT)) - min(sum, growth_bits<PAIR>(NS * R));
#pragma unroll
            for (int m = 0; m < E; ++m) v[m] = shift_rounded(v[m], shift);
        }
        __syncthreads();
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int j = t + b * TPL, k = j & (NS - 1), p = (j - k) * R + k;
#pragma unroll
            for (int i = 0; i < R; ++i) sm[at(p + i * NS)] = v[b + i * B];
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = sm[at(t + TPL * m)];
        fft_passes<A, LOGN, INV, PAIR, NS * R>(v, t, sm, at, tw, sum);
    }
}
// `sum`: the line's LineScale::sum; PAIR as in its line_scale
template <class A, int LOGN, bool INV, bool PAIR = false, typename At>
__device__ __forceinline__ void fft_line(typename A::C *v, int t, typename A::C *sm, At at,
                                         const typename A::W *__restrict__ tw, int sum) {
    fft_passes<A, LOGN, INV, PAIR, 1>(v, t, sm, at, tw, sum);
}

// ---------------------------------------------------------------------------
// floating point <-> block fixed point
// ---------------------------------------------------------------------------
// A value's magnitude as an ordered integer (for FP64 its high word), and the
// exponent field of the largest (at least 1).
__device__ __forceinline__ int magnitude(double x) { return (int)((unsigned)__double2hiint(x) & 0x7fffffffu); }
__device__ __forceinline__ int magnitude(float x) { return (int)((unsigned)__float_as_int(x) & 0x7fffffffu); }
template <typename R> __device__ __forceinline__ int exponent_of(int mag) {
    const int e = mag >> (sizeof(R) == 8 ? 20 : 23);
    return e ? e : 1;
}

// Fixed-point values count units of 2^(unit - bias + 1), bias 1023 or 127.
constexpr int kUnitNan = 1 << 14;

// x in units (kUnitMin at least), rounded; |x| below 2^62 units.
__device__ __forceinline__ long long fixed_of(unsigned long long m63, int e, int unit, bool neg) {
    // the mantissa in 63 bits, then right
    int s = unit - (e ? e : 1) + 63;
    s = s > 64 ? 64 : s;
    const unsigned long long r = ((m63 >> (s - 1)) + 1) >> 1;
    return neg ? -(long long)r : (long long)r;
}
__device__ __forceinline__ long long to_fixed(double x, int unit) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    return fixed_of(((b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull)) << 10, e, unit, (long long)b < 0);
}
__device__ __forceinline__ long long to_fixed(float x, int unit) {
    const unsigned b = (unsigned)__float_as_int(x);
    const int e = (int)(b >> 23) & 0xff;
    return fixed_of((unsigned long long)((b & 0x7fffffu) | (e ? 1u << 23 : 0u)) << 39, e, unit, (int)b < 0);
}

// u units at or beyond the ends of the normal range, by two scalings; calls,
// so that the transforms' code stays small.
static __device__ __noinline__ unsigned long long scaled_bits64(unsigned long long u, int unit) {
    const int k = unit - 1022;
    return (unsigned long long)__double_as_longlong(ldexp(ldexp((double)(long long)u, k / 2), k - k / 2));
}
static __device__ __noinline__ unsigned scaled_bits32(unsigned long long u, int unit) {
    const int k = unit - 126;
    return (unsigned)__float_as_int(ldexpf(ldexpf((float)(long long)u, k / 2), k - k / 2));
}

// F units, rounded; NaN for kUnitNan.
__device__ __forceinline__ void from_fixed(long long F, int unit, double &out) {
    const unsigned long long u = F < 0 ? 0ull - (unsigned long long)F : (unsigned long long)F;
    const int lz = __clzll((long long)u);
    const unsigned long long n = u << (lz & 63);
    const unsigned long long m = (n >> 11) + ((n >> 10) & 1ull);  // 53 bits, rounded
    const int e = 64 - lz + unit;                                 // biased exponent of the leading bit
    unsigned long long r = ((unsigned long long)(unsigned)(e - 1) << 52) + m;
    if (unit == kUnitNan) r = 0x7ff8000000000000ull;
    else if (u == 0) r = 0;
    else if (e < 1 || e > 2045) r = scaled_bits64(u, unit);
    out = __longlong_as_double((long long)(r | ((unsigned long long)F & 0x8000000000000000ull)));
}
__device__ __forceinline__ void from_fixed(long long F, int unit, float &out) {
    const unsigned long long u = F < 0 ? 0ull - (unsigned long long)F : (unsigned long long)F;
    const int lz = __clzll((long long)u);
    const unsigned long long n = u << (lz & 63);
    const unsigned m = (unsigned)(n >> 40) + ((unsigned)(n >> 39) & 1u);  // 24 bits, rounded
    const int e = 64 - lz + unit;
    unsigned r = ((unsigned)(e - 1) << 23) + m;
    if (unit == kUnitNan) r = 0x7fc00000u;
    else if (u == 0) r = 0;
    else if (e < 1 || e > 253) r = scaled_bits32(u, unit);
    out = __int_as_float((int)(r | (F < 0 ? 0x80000000u : 0u)));
}

// An upper bound of a value's magnitude relative to the exponent emax, in units
// of 2^-19 of that exponent's power of two.
template <typename R> __device__ __forceinline__ unsigned bound_of(int mag, int emax) {
    const int e = mag >> (sizeof(R) == 8 ? 20 : 23);
    const unsigned m = (((unsigned)mag >> (sizeof(R) == 8 ? 1 : 4)) & 0x7ffffu) + (e ? 0x80001u : 1u);
    const int d = emax - (e ? e : 1);
    return (m >> (d < 31 ? d : 31)) + 1u;
}
// The units of a line of points whose summed bound is s (each point's larger
// component; |re| + |im| add up to twice that at most).  The first is at least
// kUnitMin, the finest that fixed_of shifts to from the smallest exponent: a line
// of zeros or subnormals needs none below a subnormal's last bit.
constexpr int kUnitMin = -61;
template <class A, int LOGN, bool PAIR> __device__ __forceinline__ LineScale line_scale(int emax, unsigned s) {
    const int sum = (32 - __clz((int)s)) + 1 - 19;
    const int b0 = scaled_passes<A, LOGN>() ? min(sum, growth_bits<PAIR>(A::points(LOGN))) : sum;
    const int b1 = scaled_passes<A, LOGN>() ? min(sum, growth_bits<PAIR>(1 << LOGN)) : sum;
    if (emax == (sizeof(typename A::Real) == 8 ? 0x7ff : 0xff)) return {kUnitNan, kUnitNan, sum};
    const int first = max(emax + b0 - 62, kUnitMin);
    return {first, first + b1 - b0, sum};
}

}  // namespace gbib
