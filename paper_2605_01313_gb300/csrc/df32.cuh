// Double-single arithmetic for the FP64 plans: a value carried as an unevaluated
// sum hi + lo of two FP32 numbers (|lo| <= ulp(hi) / 2, 48 significant bits),
// so that FP64-accurate work runs on the FP32 units, which GB300 has at 64 times
// its FP64 rate.  Built on error-free transformations (Knuth's TwoSum, the
// FMA-based TwoProduct); the operations use the _rn intrinsics so that no product
// is contracted into a neighbouring addition, which would break them.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

// (global namespace: the complex overloads must join the generic cmake / cmul
// of common.cuh in the same overload set)

struct df32 {
    float hi, lo;
    __host__ __device__ constexpr df32() : hi(0.f), lo(0.f) {}
    __host__ __device__ constexpr df32(float h, float l) : hi(h), lo(l) {}
    // constants (folded at compile time); not for values computed at run time
    __host__ __device__ constexpr df32(double d)
        : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ constexpr df32(int i) : df32((double)i) {}
};

// s + e = a + b exactly.
__device__ __forceinline__ df32 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

// s + e = a + b exactly, for |a| >= |b| (or a = 0).
__device__ __forceinline__ df32 quick_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// Arithmetic on double-single values ("sloppy" addition: the low parts are
// added without their own error term, which keeps normwise accuracy of about
// u^2 for the FFT's butterflies), complex numbers of two of them, and the
// helpers the FFT engine uses (cmake, cmul, twiddle loads).
__device__ __forceinline__ df32 operator+(df32 a, df32 b) {
    df32 s = two_sum(a.hi, b.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return quick_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ df32 operator-(df32 a) { return df32(-a.hi, -a.lo); }
__device__ __forceinline__ df32 operator-(df32 a, df32 b) { return a + (-b); }
__device__ __forceinline__ df32 operator*(df32 a, df32 b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return quick_two_sum(p, e);
}

struct dfc {
    df32 x, y;
};
__device__ __forceinline__ dfc cmake(df32 a, df32 b) { return dfc{a, b}; }
__device__ __forceinline__ dfc operator+(dfc a, dfc b) { return dfc{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ dfc operator-(dfc a, dfc b) { return dfc{a.x - b.x, a.y - b.y}; }
// a b + sgn c d (sgn = 1 or -1): both leading products with their errors, one
// TwoSum of them, every error and cross term in one FP32 sum (19 operations; two
// products and a sum one by one, each normalised, take 25).
template <int SGN>
__device__ __forceinline__ df32 df_mul_pair(df32 a, df32 b, df32 c, df32 d) {
    const float ch = SGN < 0 ? -c.hi : c.hi, cl = SGN < 0 ? -c.lo : c.lo;
    const float p = __fmul_rn(a.hi, b.hi), q = __fmul_rn(ch, d.hi);
    float e = __fadd_rn(fmaf(a.hi, b.hi, -p), fmaf(ch, d.hi, -q));
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    e = fmaf(ch, d.lo, e);
    e = fmaf(cl, d.hi, e);
    const df32 s = two_sum(p, q);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, e));
}
__device__ __forceinline__ dfc cmul(dfc a, dfc b) {
    return dfc{df_mul_pair<-1>(a.x, b.x, a.y, b.y), df_mul_pair<1>(a.x, b.y, a.y, b.x)};
}

// The butterflies' sums, inside a radix-8 step: as operator+ without the final
// normalisation, so that the low part may grow to a few units in the last place
// of the high one (8 operations against 11).  The step's last sums and the
// multiplications normalise.  With df_mul_pair and the diagonal rotations as sums
// first, the 2048 x 1024 FP64 step went from 1396 to 1334 us, its error against 64
// bits from 3.9e-14 to 3.8e-14.
__device__ __forceinline__ df32 add_lazy(df32 a, df32 b) {
    df32 s = two_sum(a.hi, b.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return s;
}
__device__ __forceinline__ dfc add_lazy(dfc a, dfc b) {
    return dfc{add_lazy(a.x, b.x), add_lazy(a.y, b.y)};
}
__device__ __forceinline__ dfc sub_lazy(dfc a, dfc b) {
    return dfc{add_lazy(a.x, -b.x), add_lazy(a.y, -b.y)};
}
// A complex FP64 value (user data) as double-single.
__device__ __forceinline__ dfc to_dfc(double2 v);
// Read-only loads of table entries.
__device__ __forceinline__ dfc ldt(const dfc *p) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return dfc{df32(v.x, v.y), df32(v.z, v.w)};
}
__device__ __forceinline__ float2 ldt(const float2 *p) { return __ldg(p); }
__device__ __forceinline__ double2 ldt(const double2 *p) { return __ldg(p); }

// A double as hi + lo: hi holds the top 24 bits of the significand (truncated),
// lo the remaining 29 rounded to 24, by integer operations on the bit pattern
// (no FP64 arithmetic).  Magnitudes outside [2^-100, 2^100) take the plain
// conversion.
__device__ __forceinline__ df32 split_double(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e < 1023 - 100 || e >= 1023 + 100) return {__double2float_rn(v), 0.f};
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const unsigned long long m = b & 0xfffffffffffffULL;
    const float hi = __uint_as_float(sign | ((unsigned)(e - 1023 + 127) << 23) |
                                     (unsigned)(m >> 29));
    // lo = (m mod 2^29) 2^(e - 1075), scaled in two exact steps
    const float r = __uint2float_rn((unsigned)(m & 0x1fffffffULL));
    const float s1 = __uint_as_float((unsigned)(e - 1075 + 64 + 127) << 23);   // 2^(e - 1011)
    const float lo = __fmul_rn(__fmul_rn(r, 0x1p-64f), s1);     // stays inside FP32's range
    return {hi, sign ? -lo : lo};
}

__device__ __forceinline__ dfc to_dfc(double2 v) {
    return dfc{split_double(v.x), split_double(v.y)};
}

// Exponent scaling of the double-single passes.  FP32 covers 2^-126 .. 2^128
// and split_double keeps a low part only inside [2^-100, 2^100), while a
// caller's FP64 coefficients may sit anywhere in FP64's range.  So every line
// (member x field) is carried as c 2^-s, with s = emax - 1023 and emax the
// largest biased FP64 exponent among the coefficients the theta pass reads:
// the largest coefficient then lies in [1, 2) whatever the caller's units, and
// the interpolated values are multiplied back by 2^s.  Both scalings are exact
// (powers of two), so a field and the same field times 2^k give values that
// differ by exactly 2^k.  A line of zeros or subnormals (emax = 0), or one
// holding a non-finite value (emax = 0x7ff), keeps s = 0.
__device__ __forceinline__ int df_line_shift(int emax) {
    return (emax <= 0 || emax >= 0x7ff) ? 0 : emax - 1023;
}

// v 2^-s: the exponent field lowered by integer arithmetic when the result is
// a normal number (every value within 2^1022 of the line's largest), else a
// multiplication by the power of two (zeros, subnormals, non-finite values and
// results below the normal range).  s in [-1022, 1023].
__device__ __forceinline__ double df_scale_down(double v, int s) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e >= 1 && e < 0x7ff && e - s >= 1 && e - s < 0x7ff)
        return __longlong_as_double(b - ((long long)s << 52));
    return scalbn(v, -s);
}

// 2^s as a double, s in [-1022, 1023].
__device__ __forceinline__ double df_pow2(int s) {
    return __longlong_as_double((long long)(s + 1023) << 52);
}

// A complex FP64 coefficient of a line with shift s, as double-single.
__device__ __forceinline__ dfc to_dfc_scaled(double2 v, int s) {
    return dfc{split_double(df_scale_down(v.x, s)), split_double(df_scale_down(v.y, s))};
}

template <> struct CxT<df32> { typedef dfc type; };
