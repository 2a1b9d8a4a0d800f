// Exact reduction of an angle to a fraction of a turn, shared by the kernels
// that place points on a periodic grid (set_points, the Lagrange comparator).
//
// The doubled torus is 2 pi periodic in both angles, so a coordinate only
// matters as a fraction of a turn.  That fraction is computed exactly in
// integer arithmetic from the FP64 bit pattern: Y = floor(v / (2 pi) 2^64)
// mod 2^64 (Q0.64 turns), from the 53-bit significand times 1/(2 pi) held to
// 128 bits.  GB300 runs FP64 at a small fraction of its integer rate, and the
// fixed-point result is also more accurate (one unit in 2^-64 turns) than an
// FP64 product would be.
#pragma once

namespace {

// 1/(2 pi) as an unsigned Q0.128 number, floor(2^128 / (2 pi)) (Machin's formula).
#define DFS_INV_2PI_HI 0x28be60db9391054aULL
#define DFS_INV_2PI_LO 0x7f09d5f47d4d3770ULL

// Fraction of a turn of v in Q0.64: floor(|v| K 2^-64) with K = 2^128 / (2 pi),
// negated for v < 0.  False for inf/nan and for |v| >= 2^53, where FP64 no
// longer resolves a position within a turn.
__device__ __forceinline__ bool turns_q64_any(double v, unsigned long long &Y) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    int e = (int)((bits >> 52) & 0x7ff);
    if (e == 0x7ff) return false;
    unsigned long long m = bits & 0xfffffffffffffULL;
    if (e == 0) e = 1;                      // subnormal: m * 2^(1 - 1075)
    else m |= 1ULL << 52;                   // |v| = m * 2^(e - 1075)
    const int sh = 1139 - e;                // Y = floor(m * K * 2^-sh), K = 2^128 / (2 pi)
    if (sh < 64) return false;
    unsigned long long y = 0;
    if (sh < 192) {
        const unsigned long long hi0 = __umul64hi(m, DFS_INV_2PI_LO);
        const unsigned long long lo1 = m * DFS_INV_2PI_HI;
        const unsigned long long hi1 = __umul64hi(m, DFS_INV_2PI_HI);
        const unsigned long long p1 = hi0 + lo1;          // product bits 64..127
        const unsigned long long p2 = hi1 + (p1 < hi0);   // product bits 128..
        if (sh >= 128) {
            y = p2 >> (sh - 128);
        } else {
            const int s = sh - 64;
            y = s ? ((p1 >> s) | (p2 << (64 - s))) : p1;
        }
    }
    Y = (bits >> 63) ? 0ULL - y : y;
    return true;
}

// The same for the magnitudes points have, 2^-11 <= |v| < 2^9 (others go to
// turns_q64_any): the shift then takes the result from two word pairs, and five
// 32 x 32 products are enough.  Left out of the product is less than 2^34 in
// units of 2^-64 below the 44 to 63 bits shifted out, so Y is the exact floor or,
// once in about 2^16 points, one unit below it.  The integer units bound the
// fold (65% busy): with this and word-wise cell arithmetic 21.5 -> 17.4 us for
// 2.1M points.
__device__ __forceinline__ bool turns_q64(double v, unsigned long long &Y) {
    const unsigned hw = (unsigned)__double2hiint(v), ml = (unsigned)__double2loint(v);
    const int s = 1075 - (int)((hw >> 20) & 0x7ff);
    if (s < 44 || s > 63) return turns_q64_any(v, Y);
    const unsigned mh = (hw & 0xfffffu) | 0x100000u;
    const unsigned kl = (unsigned)DFS_INV_2PI_HI, kh = (unsigned)(DFS_INV_2PI_HI >> 32);
    const unsigned long long low = (unsigned long long)mh * (unsigned)(DFS_INV_2PI_LO >> 32);
    const unsigned long long t0 = (unsigned long long)ml * kl;
    const unsigned long long t1 =
        (unsigned long long)ml * kh + (unsigned)(t0 >> 32) + (unsigned)(low >> 32);
    const unsigned long long t2 = (unsigned long long)mh * kl + (unsigned)t1;
    const unsigned long long t3 =
        (unsigned long long)mh * kh + (unsigned)(t1 >> 32) + (unsigned)(t2 >> 32);
    const unsigned w1 = (unsigned)t2, w2 = (unsigned)t3, w3 = (unsigned)(t3 >> 32);
    const unsigned long long y =
        ((unsigned long long)__funnelshift_r(w2, w3, s - 32) << 32) | __funnelshift_r(w1, w2, s - 32);
    Y = (int)hw < 0 ? 0ULL - y : y;
    return true;
}

}  // namespace
