// FFT engine of the FP32 theta and phi passes: two transforms carried together
// through the packed FP32 instructions of sm_100 and later (add / mul / fma on
// a 64-bit register pair, .f32x2).
//
// Packing halves the issue slots the arithmetic takes (f32x2.cuh), which is what
// bounded the two passes (58% of the issue slots busy, FP32 and index
// arithmetic, shared-memory exchanges and table loads competing for them).  The
// exchanges move one 16-byte element (both transforms' complex values) where two
// 8-byte ones moved before.  Against the
// scalar two-line form (2048 x 1024 grid, three fields): theta pass 65 -> 57 us,
// phi pass 58 -> 40 us.
//
// A PairC holds z0 and z1 as (re0, re1), (im0, im1).  Sign changes are not
// packed instructions, so the butterflies are written without them: a
// multiplication by +-i swaps the operands of a subtraction.
#pragma once

#include "f32x2.cuh"
#include "fft_core.cuh"

namespace dfs_fft {

struct __align__(16) PairC {
    f32x2 x, y;
};

__device__ __forceinline__ PairC pair_of(float2 z0, float2 z1) {
    return PairC{pk(z0.x, z1.x), pk(z0.y, z1.y)};
}
__device__ __forceinline__ PairC operator+(PairC a, PairC b) {
    return PairC{padd(a.x, b.x), padd(a.y, b.y)};
}
__device__ __forceinline__ PairC operator-(PairC a, PairC b) {
    return PairC{psub(a.x, b.x), psub(a.y, b.y)};
}
// Both values times one complex number.
__device__ __forceinline__ PairC cmul(PairC a, float2 w) {
    const f32x2 wx = pk(w.x, w.x), wy = pk(w.y, w.y), my = pk(-w.y, -w.y);
    return PairC{pfma(a.x, wx, pmul(a.y, my)), pfma(a.x, wy, pmul(a.y, wx))};
}

// (a - c) e^{+2 pi i K / 16} for even K below 8.
template <int K>
__device__ __forceinline__ PairC rot_diff(PairC a, PairC c) {
    static_assert(K == 0 || K == 2 || K == 4 || K == 6, "radix-8 rotations");
    if constexpr (K == 0) {
        return a - c;
    } else if constexpr (K == 4) {                       // i d
        return PairC{psub(c.y, a.y), psub(a.x, c.x)};
    } else {
        constexpr float h = (float)c16(2);
        const f32x2 ph = pk(h, h), mh = pk(-h, -h);
        const PairC d = a - c;
        if constexpr (K == 2) return PairC{pmul(psub(d.x, d.y), ph), pmul(padd(d.x, d.y), ph)};
        else return PairC{pmul(padd(d.x, d.y), mh), pmul(psub(d.x, d.y), ph)};
    }
}

// Exchange layout: element i of a column's region at i ^ ((i >> 3) & 7), which
// XORs the 16-byte bank group with the 8-element group: the unit-stride reads
// and the Ns-strided writes of a quarter-warp (8 lanes of 16 bytes) each cover
// the eight bank groups once.  With cb columns interleaved in the lanes, column
// c's region starts c (n + 8 / cb) elements in, which keeps that true.
__device__ __forceinline__ int pair_pad(int i) { return i ^ ((i >> 3) & 7); }
__host__ __device__ constexpr int pair_region_stride(int n, int cb) {
    return cb == 1 ? n : n + (cb >= 8 ? 1 : 8 / cb);
}

template <int R, int K, int S, int H, int B, int P>
__device__ __forceinline__ void pair_dif_step(PairC *v) {
    if constexpr (B < R / (2 * H)) {
        if constexpr (P < H) {
            constexpr int i = K + (B * 2 * H + P) * S;
            constexpr int j = i + H * S;
            const PairC a = v[i], c = v[j];
            v[i] = a + c;
            v[j] = rot_diff<P * (8 / H)>(a, c);
            pair_dif_step<R, K, S, H, B, P + 1>(v);
        } else {
            pair_dif_step<R, K, S, H, B + 1, 0>(v);
        }
    }
}

template <int R, int K, int S, int H>
__device__ __forceinline__ void pair_dif_levels(PairC *v) {
    if constexpr (H >= 1) {
        pair_dif_step<R, K, S, H, 0, 0>(v);
        pair_dif_levels<R, K, S, H / 2>(v);
    }
}

template <int R, int K, int NS, int OFF, int T, bool LAST, class St>
__device__ __forceinline__ void pair_butterfly(PairC *v, int t, const float2 *__restrict__ stw,
                                               PairC *sm, St &st) {
    constexpr int E = DFS_FFT_E, G = E / R;
    if constexpr (K < G) {
        const int j = t + K * T;
        const int jm = j & (NS - 1);
        if constexpr (NS > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r)
                v[K + r * G] = cmul(v[K + r * G], ldt(&stw[OFF + (r - 1) * NS + jm]));
        }
        pair_dif_levels<R, K, G, R / 2>(v);
        const int base = (j - jm) * R + jm;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int o = base + bitrev(r, R) * NS;
            if constexpr (LAST) st(o, v[K + r * G]);
            else sm[pair_pad(o)] = v[K + r * G];
        }
        pair_butterfly<R, K + 1, NS, OFF, T, LAST>(v, t, stw, sm, st);
    }
}

// Barrier of the T threads of one transform group.  SPLIT: the group has whole
// warps to itself and waits for its own threads only (hardware barrier id, 1 ..
// 8), so that the groups of a CTA drift apart, one's exchange under another's
// butterflies (phi pass, 48 lines: rows of 2048 cells 138 -> 136 us, 1024 36 -> 33
// us).  The theta pass interleaves its columns in the lanes instead, for the sake
// of its stores: columns apart (16 bytes of a sector each) 56 -> 66 us.
template <int T, bool SPLIT>
__device__ __forceinline__ void group_sync(int id) {
    if constexpr (!SPLIT) __syncthreads();
    else if constexpr (T == 32) __syncwarp();
    else if constexpr (T > 32) asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(T) : "memory");
    else __syncthreads();
}

template <int LOGN, int LNS, bool SPLIT, class St, class Hook>
__device__ __forceinline__ void pair_stages(PairC *v, int t, int id,
                                            const float2 *__restrict__ stw, PairC *sm, St &st,
                                            Hook &after_first_barrier) {
    constexpr int E = DFS_FFT_E, LE = 3;
    constexpr int REM = LOGN - LNS;
    if constexpr (REM > 0) {
        constexpr int LR = REM >= LE ? LE : REM;
        constexpr int T = (1 << LOGN) / E;
        if constexpr (LNS > 0) {
            group_sync<T, SPLIT>(id);
            if constexpr (LNS == LE) after_first_barrier();
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = sm[pair_pad(t + e * T)];
            if constexpr (REM > LR) group_sync<T, SPLIT>(id);   // the last stage writes no exchange
        }
        pair_butterfly<(1 << LR), 0, (1 << LNS), stage_table_offset(LOGN, E, LNS), T, REM == LR>(
            v, t, stw, sm, st);
        pair_stages<LOGN, LNS + LR, SPLIT>(v, t, id, stw, sm, st, after_first_barrier);
    }
}

// Two length-2^LOGN inverse FFTs (LOGN > 3) of the 2^LOGN / 8 threads t, every
// thread of the CTA calling: v[e] holds input t + e 2^LOGN / 8 of both, st(i, v)
// receives output i, stw is the stage-ordered twiddle table of this length, id the
// group's barrier (group_sync).  after_first_barrier() runs on every thread when
// no thread of its group reads the inputs any more; the caller synchronises before
// it reuses the exchange region.
template <int LOGN, bool SPLIT, class St, class Hook>
__device__ __forceinline__ void pair_fft(const float2 *__restrict__ stw, PairC *sm, int t, int id,
                                         PairC *v, St &st, Hook &after_first_barrier) {
    static_assert(LOGN > 3, "at least two stages");
    pair_stages<LOGN, 0, SPLIT>(v, t, id, stw, sm, st, after_first_barrier);
}

// Lengths the pair kernels are compiled for.
#define DFS_PAIR_MIN_LOG 6
#define DFS_PAIR_MAX_LOG 12

}  // namespace dfs_fft
