// Interpolation from the fine grid to the departure points: the last stage of
// the type-2 NUFFT evaluating Eq. 5.3 (Sec. 5).  For each point
//
//   Re v_p = sum_{b<w} sum_{a<w} phi(z_b^y) phi(z_a^x) Re G[j0 + b][i0 + a]   (indices mod n)
//
// with phi the exponential-of-semicircle kernel
// phi(z) = exp(beta (sqrt(1 - (2z/w)^2) - 1)) and z_a = (a - c0) - t the
// offsets produced by set_points; the weights come from a per-tap polynomial
// fit of phi in t (see Horner below).
//
// The weights are real, so only the real part of the fine grid is read (the
// phi pass stores nothing else).  Points arrive sorted by bin (tile_x x tile_y
// fine cells); a CTA takes a bin, has the bin's tile plus its halo of every
// field in shared memory, and each thread then evaluates one point at a time
// from shared memory, computing its 2w kernel values once for all fields.
//
// FP32 plans run k_interp_tma: persistent CTAs walk their bins with the next
// bin's tiles arriving by TMA (one 2-D box per field) while the current bin is
// evaluated; the few bins whose tile wraps around the torus seam are staged
// with plain loads instead.  Inside a bin the points come sorted by fine row
// (set_points), so a warp's lanes mostly read consecutive words of one row;
// each stencil row is read with loads as wide as its alignment allows (see
// "Stencil reads" below).  k_interp_f32 (plain loads, paired reads) serves
// plans without a tensor map, and k_interp the FP64 form and wide kernels.
#include <limits.h>

#include "common.cuh"
#include "df32.cuh"
#include "tma.cuh"

namespace {

struct InterpArgs {
    int n1, n2;
    int tile_x, tile_y, lnbx;   // lnbx = log2 of the bins per bin row
    int c0;
    int F, FG;            // fields per member, fields staged per pass
    int NG;               // field groups per bin, ceil(F / FG)
    int BW, box_f;        // TMA box width (cells, multiple of 4), floats per staged box
    int bstride;          // per-member stride of the bin arrays
    int fa, fn;           // fields evaluated: fa .. fa + fn - 1 of each member
    int parts;            // CTAs a bin (k_interp_fx)
};

// Base cell of a point from its record; the first tap sits c0 cells before it.
__device__ __forceinline__ int cell_x(int cell) { return cell & 0xffff; }
__device__ __forceinline__ int cell_y(int cell) { return cell >> 16; }

// A member whose bin scan gave up (n_tasks = -1, points.cu): no list to walk, and
// its n values at `out` become NaN.
template <typename R>
__device__ __forceinline__ bool points_invalid(int ntask, R *out, size_t n) {
    if (ntask >= 0) return false;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = (R)__int_as_float(0x7fc00000);
    return true;
}

// Kernel weights by Horner's rule: for tap a the weight phi((a - c0) - t) is a
// degree-W polynomial in s = t - mid (mid = 0 for odd W, 1/2 for even W),
// fitted on the host (dfsnufft_es_horner) to about e^-beta, the size of the
// kernel's own jump at the edge of its support.  The coefficients ride in the
// kernel's parameter block, so every Horner step is one FMA with a constant
// operand; a NaN offset gives NaN weights.
template <typename R, int W>
struct Horner {
    R c[W][W + 1];
};

template <typename R, int W>
__device__ __forceinline__ void es_weights(R t, const Horner<R, W> &h, R *wv) {
    const R s = t - (W % 2 == 0 ? (R)0.5 : (R)0);
#pragma unroll
    for (int a = 0; a < W; ++a) {
        R acc = h.c[a][W];
#pragma unroll
        for (int k = W - 1; k >= 0; --k) acc = fma(acc, s, h.c[a][k]);
        wv[a] = acc;
    }
}

// The i-th of n claims of the TMA kernel's counter, as a position in the bin
// list: from both ends inward (n - 1 - i/2 for even i, i/2 for odd i, a
// permutation of [0, n)).  The densest bins are those of the first and last
// bin rows, where departure points near the poles crowd, so they start first
// rather than one of them holding up the end of the launch (2048 x 1024 grid,
// three fields: 77.0 -> 75.6 us).  The kernels that walk the list with a fixed stride keep
// the plain order: it was the faster one on the wave-scheduled FP64 grid (3%).
__device__ __forceinline__ int ends_inward(int i, int n) {
    return (i & 1) ? i >> 1 : n - 1 - (i >> 1);
}

template <typename R, int W>
__global__ void __launch_bounds__(256) k_interp(InterpArgs a, const __grid_constant__ Horner<R, W> hw,
                                                const R *__restrict__ grid,
                                                DfsPoints<R> pts,
                                                const int2 *__restrict__ task_all,
                                                const int *__restrict__ n_tasks,
                                                const int *__restrict__ pofs,
                                                R *__restrict__ out_all) {
    dfs_grid_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *tile = reinterpret_cast<R *>(smem_raw);
    const int TH = a.tile_y + W - 1;
    const int TW = a.tile_x + W - 1;
    const int tsz = TH * TW;
    // member k = blockIdx.y: its bins, sorted records [p0, p0 + Pk), F fine grids
    // and F x Pk outputs
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int Pk = pofs[k + 1] - p0;
    const int ntask = n_tasks[k];
    if (points_invalid(ntask, out_all + (size_t)a.F * p0 + (size_t)a.fa * Pk, (size_t)a.fn * Pk))
        return;
    const int2 *tasks = task_all + (size_t)k * a.bstride;
    for (int task = blockIdx.x; task < ntask; task += gridDim.x) {
        const int2 tk = tasks[task];
        const int by = tk.x >> a.lnbx;
        const int bx = tk.x - (by << a.lnbx);
        const int col0 = bx * a.tile_x - a.c0;
        const int row0 = by * a.tile_y - a.c0;
        const int s = p0 + tk.y;
        const int e = p0 + tasks[task + 1].y;
        for (int f0 = a.fa; f0 < a.fa + a.fn; f0 += a.FG) {
            const int fg = min(a.FG, a.fa + a.fn - f0);
            __syncthreads();
            // one warp per tile row: coalesced reads of TW consecutive cells
            for (int rr = threadIdx.x >> 5; rr < fg * TH; rr += blockDim.x >> 5) {
                const int ff = rr / TH;
                const int r = rr - ff * TH;
                const int gr = (row0 + r) & (a.n2 - 1);
                const R *src = grid + ((size_t)(k * a.F + f0 + ff) * a.n2 + gr) * a.n1;
                R *dst = tile + ff * tsz + r * TW;
                for (int cc = threadIdx.x & 31; cc < TW; cc += 32)
                    dst[cc] = src[(col0 + cc) & (a.n1 - 1)];
            }
            __syncthreads();
            for (int pi = s + threadIdx.x; pi < e; pi += blockDim.x) {
                int cell, dst;
                R tx, ty, wx[W], wy[W];
                pts.load(pi, cell, dst, tx, ty);
                es_weights<R, W>(tx, hw, wx);
                es_weights<R, W>(ty, hw, wy);
                const int ox = cell_x(cell) - a.c0 - col0;
                const int oy = cell_y(cell) - a.c0 - row0;
                for (int ff = 0; ff < fg; ++ff) {
                    const R *tp = tile + ff * tsz + oy * TW + ox;
                    R acc = 0;
#pragma unroll
                    for (int bb = 0; bb < W; ++bb) {
                        R rr = 0;
#pragma unroll
                        for (int aa = 0; aa < W; ++aa) rr += wx[aa] * tp[bb * TW + aa];
                        acc += wy[bb] * rr;
                    }
                    out_all[(size_t)a.F * p0 + (size_t)(f0 + ff) * Pk + dst] = acc;
                }
            }
        }
    }
}

// ---- FP64 plans
//
// The fine grid holds (hi, lo) FP32 pairs (written so by the phi pass), and the
// kernel weights are double-single (df32.cuh).  The stencil sums are taken with
// the leading product in fixed point: one 32 x 32 product into a 64-bit sum
// (IMAD.WIDE, about 4 cycles a warp instruction on one of the two FMA pipes,
// measured) adds exactly, and the two cross products, 2^-30 of it, are added in
// FP32.  A tap is then a wide product, a byte permutation and two FMAs, spread
// over the FMA pipes and the ALU, where a compensated floating-point step (Dot2)
// takes 12 instructions and a product of two-limb integers three wide products.
// 2.1M points, three fields, w = 14: 1122 us with Dot2, 836 with two-limb
// integers, 726 in this form (64% of the issue slots; more warps an SM, narrower
// bins and the fields' sums interleaved were no faster).  Of its 8600
// instructions per 32 points the weights take a third and the tiles' staging a
// twelfth.
//
//   tile values  g = S (gh 2^-30 + gl),  |gh| < 2^30, |gl| <= 2^-31, S the power
//                of two above the largest |g| of the staged tile (halo included)
//                of that field; stored as (gl, gh + 2^30);
//   weights      w = wh 2^-30 + wl,  |wl| <= 2^-31.
//
// With sum w <= 3.3 (w <= 16) a row's sum of wh (gh + 2^30) stays below 2^63; it
// starts from -2^30 sum wh, which takes the bias out.  The cross products are
// wl g, whose g comes from the top 23 bits of gh + 2^30 set under the exponent
// of 2^23 (a byte permutation; its bias 1.5 2^23 is taken out by the sum's start),
// and w gl; their rounding stays near 2^-50 S.  A row joins as an integer of units
// 2^-60 S, the rows are summed with the y weights the same way, and the point's
// value is assembled into an FP64 bit pattern by integer operations (GB300's FP64
// units run at 1/64 rate, and the conversions alone took 7% of the kernel).  A
// tile that holds a non-finite value gives NaN.
#define DFS_FX_FG 4            // fields a CTA of k_interp_fx stages at once, at most

template <int W> struct HornerDF {
    float hi[W][W + 1], lo[W][W + 1];
};

// One chain of a weight polynomial in u = s^2, coefficients k0, k0 - 2, .. k1 of
// tap a, by compensated Horner's rule (Graillat, Langlois and Louvet): an FP32
// recurrence whose product and sum errors, with the low parts of the
// coefficients and of u, run through a second one.  The first steps
// (dfs_plain_horner_steps) are plain FP32: on |s| <= 1/2 what they add is smaller
// than the weight by 1e-8 and more.
template <int W>
__device__ __forceinline__ df32 df_chain(const HornerDF<W> &h, int a, int k0, int k1, df32 u) {
    constexpr int TOP = dfs_plain_horner_steps(W);
    float e = h.hi[a][k0];
    float err = TOP ? 0.f : h.lo[a][k0];
#pragma unroll
    for (int k = k0 - 2; k >= k1; k -= 2) {
        if (k0 - k <= 2 * TOP) {
            e = fmaf(e, u.hi, h.hi[a][k]);
            continue;
        }
        const float p = __fmul_rn(e, u.hi);
        float c = fmaf(e, u.hi, -p);
        const df32 t = two_sum(p, h.hi[a][k]);
        c = __fadd_rn(__fadd_rn(c, t.lo), h.lo[a][k]);
        err = fmaf(err, u.hi, fmaf(e, u.lo, c));
        e = t.hi;
    }
    return quick_two_sum(e, err);
}

// The kernel is even, so tap W-1-a at s is tap a at -s: with tap a's
// polynomial split into even and odd parts in u = s^2, P_a(+-s) = E(u) +- s O(u)
// gives both weights of the mirror pair from two Horner chains of half length.
template <int W>
__device__ __forceinline__ void df_pair(const HornerDF<W> &h, int a, df32 s, df32 u, df32 &lo,
                                        df32 &hi) {
    const df32 e = df_chain<W>(h, a, W - (W & 1), 0, u);
    const df32 o = df_chain<W>(h, a, W - 1 + (W & 1), 1, u);
    const df32 so = s * o;
    lo = e + so;                               // tap a
    hi = e - so;                               // tap W-1-a
}

template <int W>
__device__ __forceinline__ df32 df_offset(double t) {
    return split_double(t - (W % 2 == 0 ? 0.5 : 0.0));
}

// v = (hi, lo) times k as an integer, and the fraction f left, |f| <= 1/2: the
// integer part of hi k, then that of what is left with lo k (at most 65).
__device__ __forceinline__ int fix_split(df32 v, float k, float &f) {
    const float x = __fmul_rn(v.hi, k);
    const int h = __float2int_rn(x);
    const float y = fmaf(v.lo, k, __fsub_rn(x, __int2float_rn(h)));
    const float m = __fadd_rn(y, 12582912.f);            // 1.5 2^23: y to an integer
    f = __fsub_rn(y, __fsub_rn(m, 12582912.f));
    return h + (__float_as_int(m) - 0x4b400000);
}

// A tile value as (gl, gh + 2^30), k = 2^30 / S.
__device__ __forceinline__ int2 fix_cell(float2 g, float k) {
    float f;
    const int h = fix_split(df32{g.x, g.y}, k, f);
    return make_int2(__float_as_int(__fmul_rn(f, 0x1p-30f)), h + (1 << 30));
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    return (long long)a * b + c;
}

// v 2^ex as an FP64 number (rounded half up) by integer operations; results
// outside the normal range by scalbn.
__device__ __forceinline__ double fix_value(long long v, int ex) {
    if (v == 0) return 0.0;
    unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)a);
    const int e = 1023 + 63 - lz + ex;
    if (e < 1 || e > 2045) return scalbn((double)v, ex);
    a <<= lz;
    const unsigned long long bits =
        ((unsigned long long)(e - 1) << 52) + (a >> 11) + ((a >> 10) & 1);
    return __longlong_as_double((long long)(bits | ((unsigned long long)v & (1ull << 63))));
}

// One CTA a bin: the tile and its halo of up to DFS_FX_FG fields arrive by
// 16-byte asynchronous copies (rows start on an even column), each thread finds
// the largest magnitude of the cells it copied and, once the CTA knows the
// tile's, converts those cells in place.  Then a thread a point: the x weights
// once, the y weights by mirror pairs of stencil rows, all fields per row.  A row
// of W cells is read as aligned pairs and one or two single cells at its ends by
// the parity of its first column, so no cell outside the stencil is read and a
// quarter-warp's 16-byte reads of neighbouring points do not conflict.
// Two CTAs an SM (98 KB of tiles for three fields at w = 14, 128-cell bins).
template <int W>
__global__ void __launch_bounds__(256, 2) k_interp_fx(InterpArgs a,
                                                      const __grid_constant__ HornerDF<W> hw,
                                                      const float2 *__restrict__ grid,
                                                      DfsPoints<double> pts,
                                                      const int2 *__restrict__ task_all,
                                                      const int *__restrict__ n_tasks,
                                                      const int *__restrict__ pofs,
                                                      double *__restrict__ out_all,
                                                      const int *__restrict__ emax) {
    dfs_grid_wait();
    constexpr int NS = W % 2 == 0 ? 2 : 1;     // single cells a row
    constexpr int NP = (W - NS) / 2;           // pairs a row
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int2 *tile = reinterpret_cast<int2 *>(smem_raw);
    __shared__ unsigned s_max[DFS_FX_FG];
    const int TH = a.tile_y + W - 1;
    const int TW = (a.tile_x + W + 1) & ~1;
    const int Q = TW / 2;                      // 16-byte chunks a row
    const int nq = TH * Q;
    const int tsz = TH * TW;
    // this thread's first chunk of a tile, and the step to its next one
    const int r_first = threadIdx.x / Q, c_first = threadIdx.x - r_first * Q;
    const int r_step = blockDim.x / Q, c_step = blockDim.x - r_step * Q;
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int Pk = pofs[k + 1] - p0;
    const int ntask = n_tasks[k];
    if (points_invalid(ntask, out_all + (size_t)a.F * p0 + (size_t)a.fa * Pk, (size_t)a.fn * Pk))
        return;
    const int2 *tasks = task_all + (size_t)k * a.bstride;
    for (int sub = blockIdx.x; sub < ntask * a.parts; sub += gridDim.x) {
        const int task = sub / a.parts;
        const int2 tk = tasks[task];
        const int by = tk.x >> a.lnbx;
        const int bx = tk.x - (by << a.lnbx);
        const int col0 = (bx * a.tile_x - a.c0) & ~1;
        const int row0 = by * a.tile_y - a.c0;
        // this part's points: whole warps of the bin's
        int s = p0 + tk.y, e = p0 + tasks[task + 1].y;
        if (a.parts > 1) {
            const int share = ((e - s + a.parts - 1) / a.parts + 31) & ~31;
            s += (sub - task * a.parts) * share;
            e = min(e, s + share);
            if (s >= e) continue;
        }
        for (int f0 = a.fa; f0 < a.fa + a.fn; f0 += a.FG) {
            const int fg = min(a.FG, a.fa + a.fn - f0);
            __syncthreads();                   // the tiles of the pass before are consumed
            if (threadIdx.x < DFS_FX_FG) s_max[threadIdx.x] = 0;
            for (int ff = 0; ff < fg; ++ff) {
                const float2 *g = grid + (size_t)(k * a.F + f0 + ff) * a.n2 * a.n1;
                int r = r_first, c = c_first;
                for (int i = threadIdx.x; i < nq; i += blockDim.x) {
                    const int gr = (row0 + r) & (a.n2 - 1);
                    const int gc = (col0 + 2 * c) & (a.n1 - 1);
                    cp_async_16(tile + ff * tsz + 2 * i, g + (size_t)gr * a.n1 + gc);
                    r += r_step;
                    c += c_step;
                    if (c >= Q) {
                        c -= Q;
                        ++r;
                    }
                }
            }
            cp_async_wait_all();
            __syncthreads();                   // s_max is zero
            for (int ff = 0; ff < fg; ++ff) {
                const float4 *t4 = reinterpret_cast<const float4 *>(tile + ff * tsz);
                unsigned m = 0;                // as bits: NaN above infinity above all else
                for (int i = threadIdx.x; i < nq; i += blockDim.x) {
                    const float4 v = t4[i];
                    m = max(m, max(__float_as_uint(v.x) & 0x7fffffffu,
                                   __float_as_uint(v.z) & 0x7fffffffu));
                }
                m = __reduce_max_sync(0xffffffffu, m);
                if ((threadIdx.x & 31) == 0) atomicMax(&s_max[ff], m);
            }
            __syncthreads();
            for (int ff = 0; ff < fg; ++ff) {
                // S = 2^(ue - 126), the power of two above the largest magnitude (at
                // least 2^-90: below it the field is zero next to the line's largest
                // coefficient, which is in [1, 2))
                const int ue = max((int)(s_max[ff] >> 23), 36);
                if (ue >= 255) continue;
                const float kf = __int_as_float((127 + 30 + 126 - ue) << 23);
                int4 *t4 = reinterpret_cast<int4 *>(tile + ff * tsz);
                for (int i = threadIdx.x; i < nq; i += blockDim.x) {
                    const float4 v = *reinterpret_cast<const float4 *>(t4 + i);
                    const int2 x = fix_cell(make_float2(v.x, v.y), kf);
                    const int2 y = fix_cell(make_float2(v.z, v.w), kf);
                    t4[i] = make_int4(x.x, x.y, y.x, y.y);
                }
            }
            __syncthreads();
            for (int pi = s + threadIdx.x; pi < e; pi += blockDim.x) {
                int cell, dst;
                double tx, ty;
                pts.load(pi, cell, dst, tx, ty);
                const int ox = cell_x(cell) - a.c0 - col0;
                const int oy = cell_y(cell) - a.c0 - row0;
                const int odd = ox & 1;
                // x weights in read order: pairs from tap `odd` on, then the singles
                // (tap 0 or the last but one of an even W; the last tap); wh, and
                // (w, wl 2^-22)
                int ph[2 * NP + 1], sh[NS];
                float2 pw[2 * NP + 1], sw[NS];
                long long h0 = 0;              // the starts of a row's sums
                float c0 = 0.f;
                {
                    const df32 sx = df_offset<W>(tx);
                    const df32 ux = sx * sx;
                    int wh[W];
                    float wf[W], wl[W];
                    auto put = [&](int t, df32 w) {
                        float f;
                        wh[t] = fix_split(w, 0x1p30f, f);
                        wf[t] = w.hi;
                        wl[t] = __fmul_rn(f, 0x1p-52f);
                        h0 -= wh[t];
                        c0 = fmaf(-12582912.f, wl[t], c0);
                    };
#pragma unroll
                    for (int t = 0; t < (W + 1) / 2; ++t) {
                        df32 lo, hi;
                        df_pair<W>(hw, t, sx, ux, lo, hi);
                        put(t, lo);
                        if (W - 1 - t != t) put(W - 1 - t, hi);
                    }
                    h0 <<= 30;
                    auto pick = [&](int t1, int t0, int &h, float2 &p) {
                        h = odd ? wh[t1] : wh[t0];
                        p = make_float2(odd ? wf[t1] : wf[t0], odd ? wl[t1] : wl[t0]);
                    };
#pragma unroll
                    for (int i = 0; i < 2 * NP; ++i) pick(i + 1, i, ph[i], pw[i]);
                    pick(0, W - NS, sh[0], sw[0]);
                    if (NS == 2) pick(W - 1, W - 1, sh[NS - 1], sw[NS - 1]);
                }
                const df32 sy = df_offset<W>(ty);
                const df32 uy = sy * sy;
                const int2 *tp0 = tile + oy * TW + ox;
                const int o1 = odd ? 0 : W - NS;
                // the values: yh 2^-58 S + yc S
                long long yh[DFS_FX_FG];
                float yc[DFS_FX_FG];
#pragma unroll
                for (int ff = 0; ff < DFS_FX_FG; ++ff) {
                    yh[ff] = 0;
                    yc[ff] = 0.f;
                }
                auto row = [&](int bb, df32 wy) {
                    float f;
                    const int vh = fix_split(wy, 0x1p30f, f);
                    const float vl = __fmul_rn(f, 0x1p-58f);       // times r 2^-32
                    const float vf = __fmul_rn(wy.hi, 0x1p-60f);   // times r mod 2^32
#pragma unroll
                    for (int ff = 0; ff < DFS_FX_FG; ++ff) {
                        if (ff >= fg) break;
                        const int2 *tp = tp0 + ff * tsz + bb * TW;
                        const int4 *tq = reinterpret_cast<const int4 *>(tp + odd);
                        long long h = h0;
                        float cx = 0.f, cy = c0;
                        auto tap = [&](int xh, float2 xw, int gl, int gh) {
                            h = mad_wide(xh, gh, h);
                            const int t = (int)__byte_perm(gh, 0x4b, 0x4321);
                            cx = fmaf(xw.x, __int_as_float(gl), cx);
                            cy = fmaf(xw.y, __int_as_float(t), cy);
                        };
#pragma unroll
                        for (int i = 0; i < NP; ++i) {
                            const int4 g = tq[i];
                            tap(ph[2 * i], pw[2 * i], g.x, g.y);
                            tap(ph[2 * i + 1], pw[2 * i + 1], g.z, g.w);
                        }
                        const int2 g0 = tp[o1];
                        tap(sh[0], sw[0], g0.x, g0.y);
                        if (NS == 2) {
                            const int2 g1 = tp[W - 1];
                            tap(sh[NS - 1], sw[NS - 1], g1.x, g1.y);
                        }
                        // the row as r = rh 2^32 + rl in units of 2^-60 S (the cross
                        // products, below 2^-27 S, to 2^-57 S)
                        const float2 cc = make_float2(cx, cy);
                        const int ci = __float2int_rn(__fmul_rn(__fadd_rn(cc.x, cc.y), 0x1p57f));
                        const long long r = mad_wide(ci, 8, h);
                        const int rh = (int)(r >> 32);
                        const unsigned rl = (unsigned)r;
                        yh[ff] = mad_wide(vh, rh, yh[ff]);
                        yc[ff] = fmaf(vf, __uint2float_rn(rl),
                                      fmaf(vl, __int2float_rn(rh), yc[ff]));
                    }
                };
#pragma unroll 1
                for (int bb = 0; bb < (W + 1) / 2; ++bb) {
                    df32 wlo, whi;
                    df_pair<W>(hw, bb, sy, uy, wlo, whi);
                    row(bb, wlo);
                    if (W - 1 - bb != bb) row(W - 1 - bb, whi);
                }
                const bool bad = !(tx == tx);          // an unfoldable point: NaN offsets
                double *out = out_all + (size_t)a.F * p0 + (size_t)f0 * Pk + dst;
#pragma unroll
                for (int ff = 0; ff < DFS_FX_FG; ++ff)
                    if (ff < fg) {
                        const int ue = max((int)(s_max[ff] >> 23), 36);
                        // units of 2^-58 S, back to the caller's scale: the line was
                        // carried as c 2^-s; a tile of zeros gives zero (the biases
                        // cancel to rounding only)
                        const long long v =
                            s_max[ff] ? yh[ff] + __float2ll_rn(__fmul_rn(yc[ff], 0x1p58f)) : 0;
                        const int ex = ue - 126 - 58 + df_line_shift(emax[k * a.F + f0 + ff]);
                        out[(size_t)ff * Pk] = bad || ue >= 255
                                                   ? __longlong_as_double(0x7ff8000000000000LL)
                                                   : fix_value(v, ex);
                    }
            }
        }
    }
}

// FP32 weights by mirror pairs.  The kernel is even and the fit is made on
// nodes symmetric about the centre, so tap W-1-a at s is tap a at -s: with tap
// a's polynomial split into even and odd parts in u = s^2, P_a(+-s) = E(u) +-
// s O(u) gives both weights of the pair from two Horner chains of half length
// (about 36 FMAs instead of 49 for w = 7).
template <int W>
__device__ __forceinline__ void es_weights_mirror(float t, const Horner<float, W> &h, float *wv) {
    constexpr int KE = W - (W & 1);           // highest even power
    constexpr int KO = W - 1 + (W & 1);       // highest odd power
    const float s = t - (W % 2 == 0 ? 0.5f : 0.f);
    const float u = s * s;
#pragma unroll
    for (int a = 0; a < (W + 1) / 2; ++a) {
        float e = h.c[a][KE];
#pragma unroll
        for (int k = KE - 2; k >= 0; k -= 2) e = fmaf(e, u, h.c[a][k]);
        float o = h.c[a][KO];
#pragma unroll
        for (int k = KO - 2; k >= 1; k -= 2) o = fmaf(o, u, h.c[a][k]);
        wv[a] = fmaf(s, o, e);
        if (W - 1 - a != a) wv[W - 1 - a] = fmaf(-s, o, e);
    }
}

// Weights of one FP32 point for the paired reads: wy[W] and the x weights
// shifted by the parity of the first tap into a zero-padded vector w8[WP].
template <int W>
__device__ __forceinline__ void paired_weights(float tx, float ty, int odd,
                                               const Horner<float, W> &hw, float *w8,
                                               float *wy) {
    constexpr int WP = (W + 2) & ~1;
    float wx[W];
    es_weights_mirror<W>(tx, hw, wx);
    es_weights_mirror<W>(ty, hw, wy);
#pragma unroll
    for (int k = 0; k < WP; ++k) {
        const float lo = k < W ? wx[k] : 0.f;
        const float hi = (k >= 1 && k - 1 < W) ? wx[k - 1] : 0.f;
        w8[k] = odd ? hi : lo;
    }
}

// Stencil reads of the FP32 TMA kernel.  A tile row holds BW cells (a multiple
// of 4) and starts on a 16-byte boundary; the point's W taps start at column
// ox of its row.  Three read patterns, chosen by W:
//
// Exact-width reads, W = 4q + 3 (w = 7 on 32-cell bins, whose row stride is a
// compile-time constant): the row's W cells are one 8-byte pair, one single
// cell and q aligned 16-byte quads, in an order fixed by m = ox mod 4.
// Offsets from the first tap:
//   m = 0: quads at 0,  pair at 4q,     single at 4q + 2
//   m = 1: single at 0, pair at 1,      quads at 3
//   m = 2: pair at 0,   quads at 2,     single at 4q + 2
//   m = 3: single at 0, quads at 1,     pair at 4q + 1
// Every access is aligned to its width and no cell outside the stencil is
// read: 2 + q loads a row instead of (W + 1) / 2 pairs, and fewer bank
// conflicts, since a quarter-warp's 16-byte loads of neighbouring points of
// one row fall on distinct banks.  For 2.1M points and three fields on a
// 2048 x 1024 grid (w = 7) this took the kernel from 86 to 77 us.
//
// Split reads, other odd W (and w = 7 on other bin widths): (W - 1) / 2
// aligned pairs and one single cell (first when ox is odd, last when it is
// even); 80 us on the same case.  Launches of one field (the host-buffer
// pipeline) would run faster in this form (fewer registers, and the per-point
// set-up of the exact-width weights is not shared by several fields), but the
// two forms add a row's products in different orders, and every launch of a
// plan keeps one form so that all its entry points give the same bits.
//
// Paired reads, even W: WP / 2 aligned pairs from the even column at or
// below ox, the point's weights shifted by the parity of ox (paired_weights).
template <int W> struct ExactRow {
    static constexpr int Q4 = W / 4;          // 16-byte quads a row
    int o4, o2, o1;                           // offsets of the quads, the pair, the single cell
    float w4[Q4 > 0 ? 4 * Q4 : 1], w2[2], w1; // the x weights in that order
};

template <int W>
__device__ __forceinline__ void exact_weights(float tx, float ty, int m,
                                              const Horner<float, W> &hw, ExactRow<W> &er,
                                              float *wy) {
    static_assert(W % 4 == 3, "exact-width reads need W = 4q + 3");
    constexpr int Q4 = ExactRow<W>::Q4;
    float wx[W];
    es_weights_mirror<W>(tx, hw, wx);
    es_weights_mirror<W>(ty, hw, wy);
    er.o4 = (4 - m) & 3;
    er.o2 = m == 0 ? 4 * Q4 : m == 1 ? 1 : m == 2 ? 0 : 4 * Q4 + 1;
    er.o1 = (m & 1) ? 0 : W - 1;
#pragma unroll
    for (int i = 0; i < 4 * Q4; ++i)
        er.w4[i] = m == 0 ? wx[i] : m == 1 ? wx[3 + i] : m == 2 ? wx[2 + i] : wx[1 + i];
#pragma unroll
    for (int i = 0; i < 2; ++i)
        er.w2[i] = m == 0 ? wx[4 * Q4 + i] : m == 1 ? wx[1 + i] : m == 2 ? wx[i]
                                                                        : wx[4 * Q4 + 1 + i];
    er.w1 = (m & 1) ? wx[0] : wx[W - 1];
}

// The w x w stencil sum of one field by exact-width reads: tp points at the
// first tap's cell in the tile, rows BWC floats apart (bw_rt when BWC is 0).
template <int W, int BWC>
__device__ __forceinline__ float exact_sum(const float *tp, int bw_rt, const ExactRow<W> &er,
                                           const float *wy) {
    const int bw = BWC ? BWC : bw_rt;
    const float *p1 = tp + er.o1;
    const float2 *p2 = reinterpret_cast<const float2 *>(tp + er.o2);
    const float4 *p4 = reinterpret_cast<const float4 *>(tp + er.o4);
    float acc = 0.f;
#pragma unroll
    for (int bb = 0; bb < W; ++bb) {
        const float2 g2 = p2[bb * (bw / 2)];
        float rr = er.w1 * p1[bb * bw];
        rr = fmaf(er.w2[0], g2.x, rr);
        rr = fmaf(er.w2[1], g2.y, rr);
#pragma unroll
        for (int c = 0; c < ExactRow<W>::Q4; ++c) {
            const float4 g = p4[bb * (bw / 4) + c];
            rr = fmaf(er.w4[4 * c], g.x, rr);
            rr = fmaf(er.w4[4 * c + 1], g.y, rr);
            rr = fmaf(er.w4[4 * c + 2], g.z, rr);
            rr = fmaf(er.w4[4 * c + 3], g.w, rr);
        }
        acc = fmaf(wy[bb], rr, acc);
    }
    return acc;
}

// Split reads (odd W): the x weights in read order, the single cell's last.
template <int W> struct SplitRow {
    int o2, o1;
    float w2[W - 1], w1;
};

template <int W>
__device__ __forceinline__ void split_weights(float tx, float ty, int odd,
                                              const Horner<float, W> &hw, SplitRow<W> &sr,
                                              float *wy) {
    static_assert(W % 2 == 1, "split reads need odd W");
    float wx[W];
    es_weights_mirror<W>(tx, hw, wx);
    es_weights_mirror<W>(ty, hw, wy);
    sr.o2 = odd;
    sr.o1 = odd ? 0 : W - 1;
#pragma unroll
    for (int i = 0; i < W - 1; ++i) sr.w2[i] = odd ? wx[1 + i] : wx[i];
    sr.w1 = odd ? wx[0] : wx[W - 1];
}

template <int W>
__device__ __forceinline__ float split_sum(const float *tp, int bw, const SplitRow<W> &sr,
                                           const float *wy) {
    const float *p1 = tp + sr.o1;
    const float2 *p2 = reinterpret_cast<const float2 *>(tp + sr.o2);
    float acc = 0.f;
#pragma unroll
    for (int bb = 0; bb < W; ++bb) {
        float rr = sr.w1 * p1[bb * bw];
#pragma unroll
        for (int k = 0; k < (W - 1) / 2; ++k) {
            const float2 g = p2[bb * (bw / 2) + k];
            rr = fmaf(sr.w2[2 * k], g.x, rr);
            rr = fmaf(sr.w2[2 * k + 1], g.y, rr);
        }
        acc = fmaf(wy[bb], rr, acc);
    }
    return acc;
}

// FP32 form: the tile starts at an even column and each stencil row is read as
// WP/2 aligned pairs of cells (8-byte shared loads).  Neighbouring points of
// the departure grid sit about two cells apart, so a warp's loads fall on
// consecutive 8-byte words and do not conflict in the shared-memory banks.
// The point's parity within its pair shifts its w weights into a zero-padded
// vector of WP weights.
template <int W>
__global__ void __launch_bounds__(128) k_interp_f32(InterpArgs a,
                                                    const __grid_constant__ Horner<float, W> hw,
                                                    const float *__restrict__ grid,
                                                    DfsPoints<float> pts,
                                                    const int2 *__restrict__ task_all,
                                                    const int *__restrict__ n_tasks,
                                                    const int *__restrict__ pofs,
                                                    float *__restrict__ out_all) {
    constexpr int WP = (W + 2) & ~1;          // taps read per row, even
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *tile = reinterpret_cast<float *>(smem_raw);
    const int TH = a.tile_y + W - 1;
    const int TW = a.tile_x + WP;             // even: rows stay 8-byte aligned
    const int Q = TW / 2;                     // pairs per tile row
    const int tsz = TH * TW;
    // member k = blockIdx.y: its bins, sorted records [p0, p0 + Pk), F fine grids
    // and F x Pk outputs
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int Pk = pofs[k + 1] - p0;
    const int ntask = n_tasks[k];
    if (points_invalid(ntask, out_all + (size_t)a.F * p0 + (size_t)a.fa * Pk, (size_t)a.fn * Pk))
        return;
    const int2 *tasks = task_all + (size_t)k * a.bstride;
    for (int task = blockIdx.x; task < ntask; task += gridDim.x) {
        const int2 tk = tasks[task];
        const int by = tk.x >> a.lnbx;
        const int bx = tk.x - (by << a.lnbx);
        const int col0 = (bx * a.tile_x - a.c0) & ~1;
        const int row0 = by * a.tile_y - a.c0;
        const int s = p0 + tk.y;
        const int e = p0 + tasks[task + 1].y;
        for (int f0 = a.fa; f0 < a.fa + a.fn; f0 += a.FG) {
            const int fg = min(a.FG, a.fa + a.fn - f0);
            __syncthreads();
            // one warp per tile row, a lane per pair of cells (Q <= 32); each warp
            // issues the loads of 4 rows before storing any, to keep them in flight
            {
                const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
                const int nrows = fg * TH;
                const int gc = (col0 + 2 * lane) & (a.n1 - 1);
                for (int r0 = threadIdx.x >> 5; r0 < nrows; r0 += 4 * nwarp) {
                    float2 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int rr = r0 + u * nwarp;
                        if (rr < nrows && lane < Q) {
                            const int ff = rr / TH;
                            const int gr = (row0 + rr - ff * TH) & (a.n2 - 1);
                            v[u] = *reinterpret_cast<const float2 *>(
                                grid + ((size_t)(k * a.F + f0 + ff) * a.n2 + gr) * a.n1 + gc);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int rr = r0 + u * nwarp;
                        if (rr < nrows && lane < Q) {
                            const int ff = rr / TH;
                            *reinterpret_cast<float2 *>(tile + ff * tsz + (rr - ff * TH) * TW +
                                                        2 * lane) = v[u];
                        }
                    }
                }
            }
            __syncthreads();
            for (int pi = s + threadIdx.x; pi < e; pi += blockDim.x) {
                int cell, dst;
                float tx, ty;
                pts.load(pi, cell, dst, tx, ty);
                const int ox = cell_x(cell) - a.c0 - col0;
                const int odd = ox & 1;
                float wy[W], w8[WP];
                paired_weights<W>(tx, ty, odd, hw, w8, wy);
                const int oy = cell_y(cell) - a.c0 - row0;
                for (int ff = 0; ff < fg; ++ff) {
                    const float2 *tp = reinterpret_cast<const float2 *>(
                        tile + ff * tsz + oy * TW + (ox - odd));
                    float acc = 0.f;
#pragma unroll
                    for (int bb = 0; bb < W; ++bb) {
                        float rr = 0.f;
#pragma unroll
                        for (int k = 0; k < WP / 2; ++k) {
                            const float2 g = tp[bb * Q + k];
                            rr += w8[2 * k] * g.x + w8[2 * k + 1] * g.y;
                        }
                        acc += wy[bb] * rr;
                    }
                    out_all[(size_t)a.F * p0 + (size_t)(f0 + ff) * Pk + dst] = acc;
                }
            }
        }
    }
}

// FP32 with TMA staging.  grid (CTAs per member, members); the CTAs of member
// k claim its sub-tasks from the member's counter work[2k] (one atomic a
// claim), a sub-task being one non-empty bin and one group of FG fields, so
// that SMs whose bins hold fewer points take more of them and all finish
// together.  Claims take the sub-tasks from both ends of the bin list inward
// (ends_inward): the bins of the first and last bin rows, where departure
// points near the poles crowd (up to six times a bin's median count on a
// 2048 x 1024 grid), start first instead of one of them holding up the end of
// the launch.  The last CTA of the member to finish (counter work[2k + 1])
// sets both counters back to zero for the next launch.
//
// Two stages: while a CTA evaluates its sub-task from stage j & 1, the boxes
// of the next one it claimed land in the other stage (claimed and issued after
// the barrier that ends the reads of that stage).  The chain claim -> task entry
// -> boxes is walked by the first thread of the last warp, which has no points
// of the remainder when a bin holds a few more than a multiple of the CTA's 128
// (a bin of a regular grid's departure points holds about 128), and the
// geometry reaches the other threads through shared memory (68 -> 65 us on 2.1M
// points and three fields against thread 0 and geometry loaded by every thread;
// claiming one sub-task further ahead measured 77 us).  A box starts
// at the bin's first stencil column rounded down to 4 cells (16 bytes, the TMA
// alignment rule), so a point's first tap sits at column ox in [0, tile_x + 2]
// of the box and its reads end below tile_x + 2 + WP <= BW.  BWC, when
// nonzero, is BW as a compile-time constant (the exact-width reads).  A box
// that would leave [0, n1) x [0, n2) (a bin at the torus seam) is not copied
// by TMA: its barrier phase completes on the issuing thread's arrival alone,
// and the CTA stages the tile with wrapped plain loads.  A wait that runs out
// (about a second) sets the status word to DFS_STATUS_TIMEOUT and ends the
// CTA's loop after its copies land.
template <int W, int BWC>
__global__ void __launch_bounds__(128) k_interp_tma(InterpArgs a,
                                                    const __grid_constant__ Horner<float, W> hw,
                                                    const __grid_constant__ CUtensorMap gmap,
                                                    const float *__restrict__ grid,
                                                    DfsPoints<float> pts,
                                                    const int2 *__restrict__ task_all,
                                                    const int *__restrict__ n_tasks,
                                                    const int *__restrict__ pofs,
                                                    float *__restrict__ out_all,
                                                    int *__restrict__ status,
                                                    int *__restrict__ work) {
    dfs_grid_wait();
    constexpr int WP = (W + 2) & ~1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *sb = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sb);
    // per stage: first column and row of the box, sorted points [z, w) (z < 0:
    // no more sub-tasks), and the fields staged (first, count)
    int4 *s_geo = reinterpret_cast<int4 *>(sb + 16);
    int2 *s_fld = reinterpret_cast<int2 *>(sb + 48);
    float *stage = reinterpret_cast<float *>(sb + 128);
    const int TH = a.tile_y + W - 1;
    const int BWr = BWC ? BWC : a.BW;         // floats per box row
    const int Q = BWr / 2;                    // pairs per box row
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int Pk = pofs[k + 1] - p0;
    const int ntask = n_tasks[k], total = ntask * a.NG;
    if (points_invalid(ntask, out_all + (size_t)a.F * p0 + (size_t)a.fa * Pk, (size_t)a.fn * Pk))
        return;
    const int2 *tasks = task_all + (size_t)k * a.bstride;
    int *wk = work + 2 * k;
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    const unsigned box_bytes = (unsigned)(a.BW * TH * 4);
    auto wraps = [&](int col0, int row0) {
        return col0 < 0 || col0 + a.BW > a.n1 || row0 < 0 || row0 + TH > a.n2;
    };
    const bool producer = threadIdx.x == blockDim.x - 32;
    // Take a sub-task for stage b and start its boxes; false if none is left.  A
    // CTA's first one is its own index (a thousand claims of one counter at once
    // took 2 us of a small grid's step), the others are claimed.
    auto stage_next = [&](int b, bool first) -> bool {
        int sub = first ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(&wk[0], 1);
        if (sub >= total) {
            s_geo[b] = make_int4(0, 0, -1, 0);
            return false;
        }
        sub = ends_inward(sub, total);
        const int task = sub / a.NG;
        const int2 tk = tasks[task], tn = tasks[task + 1];
        const int by = tk.x >> a.lnbx;
        const int bx = tk.x - (by << a.lnbx);
        const int col0 = (bx * a.tile_x - a.c0) & ~3;
        const int row0 = by * a.tile_y - a.c0;
        const int f0 = a.fa + (sub - task * a.NG) * a.FG;
        const int fg = min(a.FG, a.fa + a.fn - f0);
        s_geo[b] = make_int4(col0, row0, p0 + tk.y, p0 + tn.y);
        s_fld[b] = make_int2(f0, fg);
        if (wraps(col0, row0)) {
            mbar_arrive_expect_tx(&bar[b], 0);
            return true;
        }
        float *dst = stage + (size_t)b * a.FG * a.box_f;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&bar[b], box_bytes * fg);
        for (int ff = 0; ff < fg; ++ff)
            tma_load_2d(dst + (size_t)ff * a.box_f, &gmap, col0 >> 1,   // 8-byte units
                        (k * a.F + f0 + ff) * a.n2 + row0, &bar[b]);
        return true;
    };
    uint32_t ph0 = 0, ph1 = 0;
    if (producer) stage_next(0, true);
    __syncthreads();
    for (int it = 0;; ++it) {
        const int cur = it & 1;
        const int4 geo = s_geo[cur];
        if (geo.z < 0) break;
        const int2 fld = s_fld[cur];
        const bool staged_next = producer && stage_next(cur ^ 1, false);
        // the first point's record, fetched while the boxes land
        const int col0 = geo.x, row0 = geo.y, e = geo.w;
        const int f0 = fld.x, fg = fld.y;
        int pi = geo.z + threadIdx.x;
        int cell = 0, dst = 0;
        float2 t = make_float2(0.f, 0.f);
        if (pi < e) pts.load(pi, cell, dst, t.x, t.y);
        float *out = out_all + (size_t)a.F * p0 + (size_t)f0 * Pk;
        const bool ok = mbar_wait_bounded(&bar[cur], cur ? ph1 : ph0);
        if (cur) ph1 ^= 1;
        else ph0 ^= 1;
        if (__syncthreads_or(!ok)) {
            if (producer) {
                atomicExch(status, DFS_STATUS_TIMEOUT);
                mbar_wait_bounded(&bar[cur], cur ? ph1 ^ 1 : ph0 ^ 1);
                if (staged_next) mbar_wait_bounded(&bar[cur ^ 1], cur ? ph0 : ph1);
            }
            __syncthreads();
            break;
        }
        float *tile = stage + (size_t)cur * a.FG * a.box_f;
        if (wraps(col0, row0)) {
            // seam bin: the same box, gathered with indices taken mod n
            const int nq = fg * TH * Q;
            for (int i = threadIdx.x; i < nq; i += blockDim.x) {
                const int rr = i / Q;
                const int qq = i - rr * Q;
                const int ff = rr / TH;
                const int r = rr - ff * TH;
                const int gr = (row0 + r) & (a.n2 - 1);
                const int gc = (col0 + 2 * qq) & (a.n1 - 1);
                *reinterpret_cast<float2 *>(tile + (size_t)ff * a.box_f + r * BWr + 2 * qq) =
                    *reinterpret_cast<const float2 *>(
                        grid + ((size_t)(k * a.F + f0 + ff) * a.n2 + gr) * a.n1 + gc);
            }
            __syncthreads();
        }
        while (pi < e) {
            const int ox = cell_x(cell) - a.c0 - col0;
            const int oy = cell_y(cell) - a.c0 - row0;
            float *o = out + dst;
            auto next_record = [&]() {         // in flight during this point's sums
                pi += blockDim.x;
                if (pi < e) pts.load(pi, cell, dst, t.x, t.y);
            };
            if constexpr (BWC != 0 && W % 4 == 3) {
                ExactRow<W> er;
                float wy[W];
                exact_weights<W>(t.x, t.y, ox & 3, hw, er, wy);
                next_record();
                for (int ff = 0; ff < fg; ++ff) {
                    const float *tp = tile + (size_t)ff * a.box_f + oy * BWr + ox;
                    o[(size_t)ff * Pk] = exact_sum<W, BWC>(tp, BWr, er, wy);
                }
                continue;
            }
            if constexpr (W % 2 == 1) {
                SplitRow<W> sr;
                float wy[W];
                split_weights<W>(t.x, t.y, ox & 1, hw, sr, wy);
                next_record();
                for (int ff = 0; ff < fg; ++ff) {
                    const float *tp = tile + (size_t)ff * a.box_f + oy * BWr + ox;
                    o[(size_t)ff * Pk] = split_sum<W>(tp, BWr, sr, wy);
                }
                continue;
            }
            const int odd = ox & 1;
            float w8[WP], wy[W];
            paired_weights<W>(t.x, t.y, odd, hw, w8, wy);
            next_record();
            for (int ff = 0; ff < fg; ++ff) {
                const float2 *tp = reinterpret_cast<const float2 *>(
                    tile + (size_t)ff * a.box_f + oy * BWr + (ox - odd));
                float acc = 0.f;
#pragma unroll
                for (int bb = 0; bb < W; ++bb) {
                    float rr = 0.f;
#pragma unroll
                    for (int kk = 0; kk < WP / 2; ++kk) {
                        const float2 g = tp[bb * Q + kk];
                        rr += w8[2 * kk] * g.x + w8[2 * kk + 1] * g.y;
                    }
                    acc += wy[bb] * rr;
                }
                o[(size_t)ff * Pk] = acc;
            }
        }
        __syncthreads();                       // stage cur is free for the boxes after next
    }
    // the member's last CTA to finish resets its counters for the next launch
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&wk[1], 1) == (int)gridDim.x - 1) {
            wk[0] = 0;
            wk[1] = 0;
            __threadfence();
        }
    }
}

// Points in the caller's order (DFSNUFFT_KEEP_ORDER): one thread per point,
// member k = blockIdx.y; the stencil rows are read from the fine grid through
// the L1 cache (neighbouring points of a grid-ordered set share rows), indices
// taken mod n.  FP32 reads each row as WP/2 aligned pairs (paired_weights).
template <typename R, int W>
__global__ void __launch_bounds__(256) k_interp_direct(InterpArgs a,
                                                       const __grid_constant__ Horner<R, W> hw,
                                                       const R *__restrict__ grid,
                                                       DfsPoints<R> pts,
                                                       const int *__restrict__ pofs,
                                                       R *__restrict__ out_all) {
    constexpr bool PAIR = sizeof(R) == 4 && W <= 8;
    constexpr int WP = (W + 2) & ~1;
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int Pk = pofs[k + 1] - p0;
    const int m1 = a.n1 - 1, m2 = a.n2 - 1;
    for (int pl = blockIdx.x * blockDim.x + threadIdx.x; pl < Pk; pl += gridDim.x * blockDim.x) {
        int cell, own;
        R tx, ty;
        pts.load((size_t)p0 + pl, cell, own, tx, ty);
        const int2 b = make_int2(cell_x(cell) - a.c0, cell_y(cell) - a.c0);
        R *out = out_all + (size_t)a.F * p0 + pl;
        if constexpr (PAIR) {
            const int odd = b.x & 1;
            const int cx = b.x - odd;                  // even: pairs never straddle a row end
            float w8[WP], wy[W];
            paired_weights<W>(tx, ty, odd, hw, w8, wy);
            for (int f = a.fa; f < a.fa + a.fn; ++f) {
                const float *g = grid + (size_t)(k * a.F + f) * a.n2 * a.n1;
                float acc = 0.f;
#pragma unroll
                for (int bb = 0; bb < W; ++bb) {
                    const float *gr = g + (size_t)((b.y + bb) & m2) * a.n1;
                    float rr = 0.f;
#pragma unroll
                    for (int kk = 0; kk < WP / 2; ++kk) {
                        const float2 v = __ldg(reinterpret_cast<const float2 *>(
                            gr + ((cx + 2 * kk) & m1)));
                        rr += w8[2 * kk] * v.x + w8[2 * kk + 1] * v.y;
                    }
                    acc += wy[bb] * rr;
                }
                out[(size_t)f * Pk] = acc;
            }
        } else {
            R wx[W], wy[W];
            es_weights<R, W>(tx, hw, wx);
            es_weights<R, W>(ty, hw, wy);
            for (int f = a.fa; f < a.fa + a.fn; ++f) {
                const R *g = grid + (size_t)(k * a.F + f) * a.n2 * a.n1;
                R acc = 0;
#pragma unroll
                for (int bb = 0; bb < W; ++bb) {
                    const R *gr = g + (size_t)((b.y + bb) & m2) * a.n1;
                    R rr = 0;
#pragma unroll
                    for (int aa = 0; aa < W; ++aa) rr += wx[aa] * __ldg(gr + ((b.x + aa) & m1));
                    acc += wy[bb] * rr;
                }
                out[(size_t)f * Pk] = acc;
            }
        }
    }
}

// Points in the caller's order, FP32: each warp takes 32 consecutive points of
// a member, finds their stencils' bounding box (coordinates unwrapped around
// lane 0's, so a chunk across the torus seam stays compact) and, when the box
// fits half of its shared-memory slice of WT_CAP floats, stages the fields'
// boxes by asynchronous 8-byte copies (cp.async, indices taken mod n), field
// f + 1 landing in one half while field f is evaluated from the other; a chunk
// whose box does not fit reads its stencils from the fine grid directly.  Points of one arrival row sit about two cells apart, so
// the warp's pair reads fall on consecutive words.  grid (CTAs, members).
#define WT_CAP 1536
template <int W>
__global__ void __launch_bounds__(256) k_interp_wtile(InterpArgs a,
                                                      const __grid_constant__ Horner<float, W> hw,
                                                      const float *__restrict__ grid,
                                                      DfsPoints<float> pts,
                                                      const int *__restrict__ pofs,
                                                      float *__restrict__ out_all) {
    constexpr int WP = (W + 2) & ~1;
    __shared__ __align__(16) float tiles[8][WT_CAP];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float *tile = tiles[wid];
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int Pk = pofs[k + 1] - p0;
    const int m1 = a.n1 - 1, m2 = a.n2 - 1;
    const int nchunk = (Pk + 31) >> 5;
    const int wstride = gridDim.x * (blockDim.x >> 5);
    for (int ch = blockIdx.x * (blockDim.x >> 5) + wid; ch < nchunk; ch += wstride) {
        const int pl = (ch << 5) + lane;
        const bool live = pl < Pk;
        int2 b = make_int2(0, 0);
        float2 t = make_float2(0.f, 0.f);
        if (live) {
            int cell, own;
            pts.load((size_t)p0 + pl, cell, own, t.x, t.y);
            b = make_int2(cell_x(cell) - a.c0, cell_y(cell) - a.c0);
        }
        // unwrap around lane 0's cell, then the chunk's box
        const int bx0 = __shfl_sync(0xffffffffu, b.x, 0), by0 = __shfl_sync(0xffffffffu, b.y, 0);
        const int ux = bx0 + ((((b.x - bx0) + (a.n1 >> 1)) & m1) - (a.n1 >> 1));
        const int uy = by0 + ((((b.y - by0) + (a.n2 >> 1)) & m2) - (a.n2 >> 1));
        const int xmin = __reduce_min_sync(0xffffffffu, live ? ux : INT_MAX);
        const int xmax = __reduce_max_sync(0xffffffffu, live ? ux : INT_MIN);
        const int ymin = __reduce_min_sync(0xffffffffu, live ? uy : INT_MAX);
        const int ymax = __reduce_max_sync(0xffffffffu, live ? uy : INT_MIN);
        const int col0 = xmin & ~1;                        // even: pairs stay aligned
        const int TW = ((xmax - col0) + WP + 1) & ~1;      // pair reads end below TW
        const int TH = ymax - ymin + W;
        const int Q = TW >> 1;
        const bool fits = 2 * TW * TH <= WT_CAP;
        // lanes past the member's last point read the box's first cells
        const int ox = live ? ux - col0 : 0, odd = ox & 1, oy = live ? uy - ymin : 0;
        float w8[WP], wy[W];
        paired_weights<W>(t.x, t.y, odd, hw, w8, wy);
        float *out = out_all + (size_t)a.F * p0 + pl;
        // asynchronous copies of field f's box into half f & 1 of the slice
        auto stage = [&](int f) {
            const float *g = grid + (size_t)(k * a.F + f) * a.n2 * a.n1;
            float *dst = tile + (f & 1) * (WT_CAP / 2);
            for (int r = 0; r < TH; ++r) {
                const float *gr = g + (size_t)((ymin + r) & m2) * a.n1;
                for (int q = lane; q < Q; q += 32)
                    cp_async_8(dst + r * TW + 2 * q, gr + ((col0 + 2 * q) & m1));
            }
            cp_async_commit();
        };
        __syncwarp();                                      // the previous chunk's boxes are consumed
        if (fits) stage(a.fa);
        for (int f = a.fa; f < a.fa + a.fn; ++f) {
            const float *g = grid + (size_t)(k * a.F + f) * a.n2 * a.n1;
            float acc = 0.f;
            if (fits) {
                if (f + 1 < a.fa + a.fn) {
                    __syncwarp();                          // half (f + 1) & 1 was read at f - 1
                    stage(f + 1);
                    cp_async_wait_group<1>();
                } else {
                    cp_async_wait_group<0>();
                }
                __syncwarp();
                const float2 *tp = reinterpret_cast<const float2 *>(
                    tile + (f & 1) * (WT_CAP / 2) + oy * TW + (ox - odd));
#pragma unroll
                for (int bb = 0; bb < W; ++bb) {
                    float rr = 0.f;
#pragma unroll
                    for (int kk = 0; kk < WP / 2; ++kk) {
                        const float2 v = tp[bb * Q + kk];
                        rr += w8[2 * kk] * v.x + w8[2 * kk + 1] * v.y;
                    }
                    acc += wy[bb] * rr;
                }
            } else {
                const int cx = b.x - odd;
#pragma unroll
                for (int bb = 0; bb < W; ++bb) {
                    const float *gr = g + (size_t)((b.y + bb) & m2) * a.n1;
                    float rr = 0.f;
#pragma unroll
                    for (int kk = 0; kk < WP / 2; ++kk) {
                        const float2 v = __ldg(reinterpret_cast<const float2 *>(
                            gr + ((cx + 2 * kk) & m1)));
                        rr += w8[2 * kk] * v.x + w8[2 * kk + 1] * v.y;
                    }
                    acc += wy[bb] * rr;
                }
            }
            if (live) out[(size_t)f * Pk] = acc;
        }
    }
}

template <typename R, int W>
cudaError_t launch_w(dfsnufft_plan p, void *values) {
    const dfsnufft_params &q = p->prm;
    InterpArgs a;
    a.n1 = q.n1;
    a.n2 = q.n2;
    a.tile_x = q.tile_x;
    a.tile_y = q.tile_y;
    a.lnbx = 0;
    while ((1 << a.lnbx) < p->nbx) ++a.lnbx;
    a.c0 = p->c0;
    a.F = p->n_fields;
    a.bstride = p->bstride;
    // a line window (one-member plans) selects fields
    a.fa = p->nwin ? p->win0 : 0;
    a.fn = p->nwin ? p->nwin : a.F;
    a.NG = 1;
    a.parts = 1;
    a.BW = 0;
    a.box_f = 0;
    // the plan's fitted weight polynomials (fitting them costs the host 10 us at
    // w = 7 and 35 us at w = 14, more than the launches of a small step)
    Horner<R, W> hw;
    for (int i = 0; i < W; ++i)
        for (int k = 0; k <= W; ++k) hw.c[i][k] = (R)p->horner[i * (W + 1) + k];
    const int M = p->n_members;
    constexpr int WP = (W + 2) & ~1;
    if (p->keep_order) {
        int64_t blocks = (p->max_member_points + 255) / 256;
        if (blocks < 1) blocks = 1;
        if constexpr (sizeof(R) == 4 && W <= 8) {
            Horner<float, W> hf;
            for (int i = 0; i < W; ++i)
                for (int kk = 0; kk <= W; ++kk) hf.c[i][kk] = (float)hw.c[i][kk];
            k_interp_wtile<W><<<dim3((unsigned)blocks, M), 256, 0, p->stream>>>(
                a, hf, (const float *)p->d_G, dfs_points<float>(p), p->d_pofs, (float *)values);
            return cudaGetLastError();
        }
        k_interp_direct<R, W><<<dim3((unsigned)blocks, M), 256, 0, p->stream>>>(
            a, hw, (const R *)p->d_G, dfs_points<R>(p), p->d_pofs, (R *)values);
        return cudaGetLastError();
    }
    if constexpr (sizeof(R) == 4 && W <= 8) {
        Horner<float, W> hf;
        for (int i = 0; i < W; ++i)
            for (int k = 0; k <= W; ++k) hf.c[i][k] = (float)hw.c[i][k];
        // TMA form: plans that own their buffers (status word, fixed d_G)
        const int TH = q.tile_y + W - 1;
        const int BW = (q.tile_x + WP + 2 + 3) & ~3;
        if (p->d_status && p->d_work && BW / 2 <= 256 && TH <= 256) {
            if (!p->tmap_G_ok) {
                if (dfs_encode_tensor_map_2d(&p->tmap_G, p->d_G, (uint64_t)(q.n1 / 2),
                                             (uint64_t)M * a.F * q.n2,
                                             (uint64_t)q.n1 * sizeof(float), (uint32_t)(BW / 2),
                                             (uint32_t)TH) == cudaSuccess)
                    p->tmap_G_ok = 1;
            }
            if (p->tmap_G_ok) {
                a.BW = BW;
                a.box_f = (BW * TH + 31) & ~31;           // 128-byte aligned boxes
                // fields per stage: two stages within about 26 KB
                int fg = (13 * 1024) / (a.box_f * 4);
                if (fg < 1) fg = 1;
                if (fg > a.F) fg = a.F;
                a.FG = fg;
                a.NG = (a.fn + fg - 1) / fg;
                const size_t smem = 128 + 128 + 2 * (size_t)fg * a.box_f * sizeof(float);
                // w = 7 on 32-cell bins (BW = 44): the exact-width reads, in
                // every launch of the plan, so that launches of one field (the
                // host-buffer pipeline) and of all fields give the same bits
                auto kern = k_interp_tma<W, 0>;
                if constexpr (W == 7)
                    if (BW == 44) kern = k_interp_tma<W, 44>;
                cudaError_t e = dfs_allow_smem((const void *)kern, smem);
                if (e) return e;
                if (p->interp_ctas_per_sm <= 0) {
                    int occ = 0;
                    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 128,
                                                                      smem) != cudaSuccess ||
                        occ < 1)
                        occ = 1;
                    p->interp_ctas_per_sm = occ;
                }
                int64_t want = ((int64_t)p->num_sms * p->interp_ctas_per_sm + M - 1) / M;
                const int64_t cap = (int64_t)p->nbins * a.NG;
                if (want > cap) want = cap;
                if (want < 1) want = 1;
                return dfs_launch_dependent(
                    kern, dim3((unsigned)want, M), dim3(128), smem, p->stream, a, hf,
                    p->tmap_G, (const float *)p->d_G, dfs_points<float>(p),
                    (const int2 *)p->d_task_bin, (const int *)p->d_n_tasks,
                    (const int *)p->d_pofs, (float *)values, p->d_status, p->d_work);
            }
        }
        // plain loads: tile rows of at most 32 pairs
        if ((q.tile_x + WP) / 2 <= 32) {
            const int tw = q.tile_x + WP;
            const size_t per_field = sizeof(float) * (size_t)TH * tw;
            int fg = (int)((96 * 1024) / per_field);
            if (fg < 1) fg = 1;
            if (fg > a.F) fg = a.F;
            a.FG = fg;
            const size_t smem = per_field * fg;
            int per = (152 * 16 + M - 1) / M;
            if (per > p->nbins) per = p->nbins;
            if (per < 1) per = 1;
            cudaError_t e = dfs_allow_smem((const void *)k_interp_f32<W>, smem);
            if (e) return e;
            k_interp_f32<W><<<dim3(per, M), 128, smem, p->stream>>>(
                a, hf, (const float *)p->d_G, dfs_points<float>(p), p->d_task_bin, p->d_n_tasks,
                p->d_pofs, (float *)values);
            return cudaGetLastError();
        }
    }
    const int tw = q.tile_x + W - 1;
    const size_t per_field = sizeof(R) * (size_t)(q.tile_y + W - 1) * tw;
    int fg = (int)((96 * 1024) / per_field);
    if (fg < 1) fg = 1;
    if (fg > a.F) fg = a.F;
    a.FG = fg;
    const size_t smem = per_field * fg;
    // blocks per member: enough to fill the GPU across all members
    int per = (152 * 16 + M - 1) / M;
    if (per > p->nbins) per = p->nbins;
    if (per < 1) per = 1;
    if constexpr (sizeof(R) == 8) {
        if (p->gdf) {
            HornerDF<W> hd;
            for (int i = 0; i < W; ++i)
                for (int kk = 0; kk <= W; ++kk) {
                    const double c = (double)hw.c[i][kk];
                    hd.hi[i][kk] = (float)c;
                    hd.lo[i][kk] = (float)(c - (double)hd.hi[i][kk]);
                }
            const size_t tile =
                sizeof(int2) * (size_t)(q.tile_y + W - 1) * ((q.tile_x + W + 1) & ~1);
            // fields a CTA holds at once: as many as leave two CTAs an SM (one if
            // none does), the passes over the fields evened out
            a.FG = (int)(112 * 1024 / tile);
            if (a.FG < 1) a.FG = 1;
            if (a.FG > DFS_FX_FG) a.FG = DFS_FX_FG;
            const int passes = (a.fn + a.FG - 1) / a.FG;
            a.FG = (a.fn + passes - 1) / passes;
            const size_t smem_fx = tile * a.FG;
            // few bins: several CTAs a bin, each staging the tile for whole warps of
            // its points, until the SMs have a CTA each (64 x 32: 5 of 8 bins hold
            // points, 20 -> 12 us in 40 CTAs)
            a.parts = p->num_sms / (p->nbins * M);
            if (a.parts > 8) a.parts = 8;
            if (a.parts < 1) a.parts = 1;
            per = per * a.parts;
            cudaError_t e = dfs_allow_smem((const void *)k_interp_fx<W>, smem_fx);
            if (e) return e;
            return dfs_launch_dependent(
                k_interp_fx<W>, dim3(per, M), dim3(256), smem_fx, p->stream, a, hd,
                (const float2 *)p->d_G, dfs_points<double>(p), (const int2 *)p->d_task_bin,
                (const int *)p->d_n_tasks, (const int *)p->d_pofs, (double *)values,
                (const int *)p->d_emax);
        }
    }
    cudaError_t e = dfs_allow_smem((const void *)k_interp<R, W>, smem);
    if (e) return e;
    const int threads = sizeof(R) == 4 ? 128 : 256;
    return dfs_launch_dependent(k_interp<R, W>, dim3(per, M), dim3(threads), smem, p->stream, a,
                                hw, (const R *)p->d_G, dfs_points<R>(p),
                                (const int2 *)p->d_task_bin, (const int *)p->d_n_tasks,
                                (const int *)p->d_pofs, (R *)values);
}

template <typename R, int W>
cudaError_t dispatch(dfsnufft_plan p, void *values, int w) {
    if constexpr (W > 16) {
        return cudaErrorInvalidValue;
    } else {
        if (w == W) return launch_w<R, W>(p, values);
        return dispatch<R, W + 1>(p, values, w);
    }
}

}  // namespace

cudaError_t dfs_launch_interp(dfsnufft_plan p, void *values) {
    if (p->prm.dtype == DFSNUFFT_F64) return dispatch<double, 2>(p, values, p->prm.w);
    return dispatch<float, 2>(p, values, p->prm.w);
}
