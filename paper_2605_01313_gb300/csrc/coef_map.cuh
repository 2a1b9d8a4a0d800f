// Coefficient helpers shared by the column passes of the inverse FFT (the
// theta pass and the persistent ensemble step): conjugation, scaling and the
// Hermitian part a real-field plan transforms (Sec. 5 evaluation of Eq. 5.3 for
// real fields, whose values depend on that part only).
#pragma once

#include "common.cuh"
#include "df32.cuh"

namespace dfs_coef {

template <typename C> __device__ __forceinline__ C cconj(C a) { return cmake(a.x, -a.y); }
template <typename C, typename R> __device__ __forceinline__ C cscale(C a, R s) {
    return cmake(a.x * s, a.y * s);
}

// The Hermitian part h_{n,k} = (c_{n,k} + conj c_{-n,-k}) / 2 that a real-field
// plan transforms, for -half <= n <= half and 0 <= k <= N1/2, from a reader
// cf(row, col) of the centred coefficient array that returns zero outside it
// (half = N2/2).  Entries whose mirror lies outside the even-sized array (the
// Nyquist row n = -N2/2 and column m = -N1/2) are split exactly into c/2 at
// (n, m) and conj(c)/2 at (-n, -m); column k = 0 is its own mirror.
template <typename C, class Rd>
__device__ __forceinline__ C herm_coef(int n, int k, int half, int N1, Rd &cf) {
    typedef decltype(C().x) R;
    const int N1h = N1 / 2;
    const int qa = N1h + k;                        // array column of m = k (N1 if k = N1/2)
    if (k == N1h)                                  // mirror of the Nyquist column
        return n == -half ? cmake((R)0, (R)0) : cscale(cconj(cf(half - n, 0)), (R)0.5);
    if (n == half) return cscale(cconj(cf(0, N1 - qa)), (R)0.5);   // mirror of the Nyquist row
    const C c = cf(n + half, qa);
    if (n == -half) return cscale(c, (R)0.5);
    if (k == 0) {
        const C mirror = cf(half - n, qa);
        return cscale(cmake(c.x + mirror.x, c.y - mirror.y), (R)0.5);
    }
    return c;
}

// A coefficient as the pass's complex type: itself, or (double-single passes of
// FP64 plans) the FP64 value times 2^-sh (the line's exponent shift, df32.cuh)
// split into double-single parts.
template <typename C, typename CIn> __device__ __forceinline__ C in_value(CIn v, int) { return v; }
template <> __device__ __forceinline__ dfc in_value<dfc, double2>(double2 v, int sh) {
    return to_dfc_scaled(v, sh);
}
// Complex coefficient c_{n,m} (m >= 0, |n| <= N) of a field given by its
// partial-regularity DFS coefficients (Sec. 4): col[k] = f^c_{k,m} + i f^s_{k,m},
// k = 0..N, for this m.  First the standard coefficient S = f~^c + i f~^s at |n|
// (the product-to-sum stencil of Sec. 4 for the case of m; f~_{0,m} = f_{1,m}/2
// for even m >= 2, which the identity gives in place of the printed 0), then
// Eq. 5.4: c = S/2 (m = 0, n != 0; S for n = 0), conj(S)/2 or /4 (even m), and
// -sign(n) i conj(S)/4 (odd m).  The stencils are linear with real weights, so
// they act on the cosine and sine parts at once.
template <typename C, typename CIn>
__device__ __forceinline__ C pr_coef(int n, int m, int N, const CIn *__restrict__ col,
                                     int sh = 0) {
    typedef decltype(C().x) R;
    const int na = n < 0 ? -n : n;
    // f_{k,m} on the case's index range, zero elsewhere
    auto f = [&](int k, int lo, int hi) -> C {
        return (k >= lo && k <= hi) ? in_value<C>(col[k], sh) : cmake((R)0, (R)0);
    };
    C S;
    if (m == 0) {
        if (na > N) return cmake((R)0, (R)0);
        const R v = in_value<C>(col[na], sh).x;            // no sine part at m = 0
        return cmake(na == 0 ? v : (R)0.5 * v, (R)0);
    } else if (m == 1) {
        if (na == 0) return cmake((R)0, (R)0);
        // sin t cos k t = (sin (k+1) t - sin (k-1) t) / 2, k = 0..N-1
        S = cscale(f(na - 1, 0, N - 1) - f(na + 1, 0, N - 1), (R)0.5);
        if (na == 1) S = S + cscale(f(0, 0, N - 1), (R)0.5);
    } else if ((m & 1) == 0) {
        // sin t sin k t = (cos (k-1) t - cos (k+1) t) / 2, k = 1..N-1
        S = na == 0 ? cscale(f(1, 1, N - 1), (R)0.5)
                    : cscale(f(na + 1, 1, N - 1) - f(na - 1, 1, N - 1), (R)0.5);
    } else {
        if (na == 0) return cmake((R)0, (R)0);
        // sin^2 t sin k t = (2 sin k t - sin (k-2) t - sin (k+2) t) / 4, k = 1..N-2
        S = cscale(cscale(f(na, 1, N - 2), (R)2) - f(na - 2, 1, N - 2) - f(na + 2, 1, N - 2),
                   (R)0.25);
        if (na == 1) S = S + cscale(f(1, 1, N - 2), (R)0.25);
    }
    const C cs = cmake(S.x, -S.y);                         // conj(S) = f~^c - i f~^s
    if ((m & 1) == 0) return cscale(cs, na == 0 ? (R)0.5 : (R)0.25);
    // -sign(n) i conj(S) / 4
    const R g = n > 0 ? (R)-0.25 : (R)0.25;
    return cmake(-g * cs.y, g * cs.x);
}

}  // namespace dfs_coef
