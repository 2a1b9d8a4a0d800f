// set_points: fold the departure points onto the fine-grid torus, sort them by
// interpolation bin with a counting sort, and find the range of fine rows their
// stencils touch.
//
// The doubled torus is 2 pi periodic in both angles (Sec. 4-5), so a coordinate
// only matters as a fraction of a turn.  That fraction is computed exactly in
// integer arithmetic from the FP64 bit pattern: Y = floor(v / (2 pi) 2^64)
// mod 2^64 (Q0.64 turns, or one unit below), from the 53-bit significand times
// 1/(2 pi) held to 128 bits.  GB300 runs FP64 at a small fraction of its integer rate, and the
// fixed-point result is also more accurate (one unit in 2^-64 turns) than an
// FP64 product would be.  For a fine grid of n = 2^L cells the point sits at
// x = Y / 2^(64-L) cells; it gets an integer base cell b and an offset t = x - b:
//   even w: b = floor(x),       t in [0, 1)
//   odd  w: b = floor(x + 1/2), t in [-1/2, 1/2)
// The w taps sit at cells b - c0 .. b - c0 + w - 1 (c0 = w/2 - 1 or (w-1)/2),
// at kernel arguments z_a = (a - c0) - t, all inside [-w/2, w/2].  Only the
// offset t leaves this file in plan precision (FP32 or FP64), so the FP32 form
// keeps its kernel arguments accurate to ~1e-9 cells at any grid size.
#include "common.cuh"
#include "tma.cuh"
#include "turns.cuh"

namespace {

struct FoldParams {
    int L1, L2;         // log2 of the fine sizes
    int odd_w;
    int c0, w;
    int ltx, lty, nbx;  // log2 of the bin size (powers of two), bins per bin row
};

// Base cell and offset of one coordinate on a fine grid of 2^L cells (4 <= L <=
// 13).  tq is the offset t in units of 2^-64 cells (signed for odd w).  Word by
// word: the cell is the top L bits, and half a cell is a bit of the high word.
__device__ __forceinline__ void split_cell(unsigned long long Y, int L, int odd_w, int &b,
                                           unsigned long long &tq) {
    const unsigned lo = (unsigned)Y;
    const unsigned hi = (unsigned)(Y >> 32) + (odd_w ? 1u << (31 - L) : 0u);
    b = (int)(hi >> (32 - L));
    const unsigned th = __funnelshift_l(lo, hi, L) ^ (odd_w ? 0x80000000u : 0u);
    tq = ((unsigned long long)th << 32) | (lo << L);
}

template <typename R> __device__ __forceinline__ R offset_value(unsigned long long tq, int odd_w);
template <> __device__ __forceinline__ float offset_value<float>(unsigned long long tq, int odd_w) {
    return odd_w ? (float)(int)(tq >> 32) * 0x1p-32f : (float)(unsigned)(tq >> 32) * 0x1p-32f;
}
template <>
__device__ __forceinline__ double offset_value<double>(unsigned long long tq, int odd_w) {
    return odd_w ? (double)((long long)tq >> 11) * 0x1p-53
                 : (double)(long long)(tq >> 11) * 0x1p-53;
}

// A coordinate that cannot be folded (non-finite, or beyond 2^53 rad) is placed
// at cell 0; its offset becomes NaN so that its value comes out NaN.
__device__ __forceinline__ bool fold_point(const FoldParams &f, double lon, double colat,
                                           int &bx, int &by, unsigned long long &tx,
                                           unsigned long long &ty) {
    unsigned long long yx = 0, yy = 0;
    const bool ok = turns_q64(lon, yx) & turns_q64(colat, yy);
    split_cell(ok ? yx : 0ULL, f.L1, f.odd_w, bx, tx);
    split_cell(ok ? yy : 0ULL, f.L2, f.odd_w, by, ty);
    return ok;
}

__device__ __forceinline__ int bin_of(const FoldParams &f, int bx, int by) {
    return (by >> f.lty) * f.nbx + (bx >> f.ltx);
}

// Unsorted record of a folded point, written by k_fold_count and moved to its
// sorted place by k_scatter: base cell (bx | by << 16, both below 2^13), the
// point's rank inside its bin (input order) and its offsets in plan precision.
// 16 bytes in FP32 (one vector store and load), 24 in FP64.
template <typename R> struct FoldRec;
template <> struct __align__(16) FoldRec<float> {
    int base, rank;
    float tx, ty;
};
template <> struct __align__(8) FoldRec<double> {
    int base, rank;
    double tx, ty;
};
static_assert(sizeof(FoldRec<float>) == 16 && sizeof(FoldRec<double>) == 24,
              "record sizes of dfs_fold_rec_bytes");

// Sort key of a point: its bin, then its base cell's row inside the bin (the
// rank within a bin follows fine rows, so that the points of one warp share
// stencil rows and read consecutive shared-memory words).
__device__ __forceinline__ int rowkey_of(const FoldParams &f, int bx, int by) {
    return (bin_of(f, bx, by) << f.lty) | (by & ((1 << f.lty) - 1));
}

// grid (ceil(max member points / 256), members): member k = blockIdx.y.  Folds
// every point once (kept in its unsorted record) and counts the points of each
// row of each bin (the row counts at rowoff in the member's count slice); the
// rank of a point is its position among its row's points, in input order.
template <typename R>
__global__ void __launch_bounds__(256) k_fold_count(const double *__restrict__ lon,
                                                    const double *__restrict__ colat,
                                                    FoldParams f, const int *__restrict__ pofs,
                                                    int cstride, int rowoff,
                                                    int *__restrict__ bin_count,
                                                    FoldRec<R> *__restrict__ urec) {
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int pl = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = pl < pofs[k + 1] - p0;
    int bin = -1;                               // the row key
    FoldRec<R> rec;
    if (live) {
        int bx, by;
        unsigned long long tx, ty;
        const bool ok = fold_point(f, lon[p0 + pl], colat[p0 + pl], bx, by, tx, ty);
        bin = rowkey_of(f, bx, by);
        rec.base = bx | (by << 16);
        rec.tx = offset_value<R>(tx, f.odd_w);
        rec.ty = offset_value<R>(ty, f.odd_w);
        if (!ok) rec.tx = rec.ty = (R)__int_as_float(0x7fc00000);
    }
    // warp aggregation over runs of equal bins (points arrive nearly sorted):
    // the first lane of each run takes the run's ranks with one atomicAdd
    const int lane = threadIdx.x & 31;
    const int prev = __shfl_up_sync(0xffffffffu, bin, 1);
    const bool head = live && (lane == 0 || prev != bin);
    const unsigned heads = __ballot_sync(0xffffffffu, head);
    const unsigned live_mask = __ballot_sync(0xffffffffu, live);
    // this lane's run: from its head to the lane before the next head (or the
    // last live lane)
    const int my_head = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
    const unsigned later = heads & ~(0xffffffffu >> (31 - lane));   // heads after this lane
    const int run_end = later ? __ffs(later) - 1 : 32 - __clz(live_mask);
    int base = 0;
    if (head) base = atomicAdd(&bin_count[(size_t)k * cstride + rowoff + bin], run_end - lane);
    base = __shfl_sync(0xffffffffu, base, my_head);
    if (live) {
        rec.rank = base + lane - my_head;
        urec[p0 + pl] = rec;
    }
}

// Smallest index i in [from, from + nb) (circular over nb bits) whose bit in
// `bits` equals `value`; from + nb if there is none.
__device__ int next_bit(const unsigned *bits, int nb, int from, int value) {
    int i = from;
    const int end = from + nb;
    while (i < end) {
        const int k = i < nb ? i : i - nb;
        unsigned w = bits[k >> 5];
        if (!value) w = ~w;
        w >>= (k & 31);
        // bits past nb in the last word do not count
        const int avail = min(32 - (k & 31), nb - k);
        if (avail < 32) w &= (1u << avail) - 1u;
        if (w) {
            const int hit = i + __ffs(w) - 1;
            return hit < end ? hit : end;
        }
        i += avail;
    }
    return end;
}

struct ScanParams {
    int nbins, lnbx, nbr;     // bins, log2 of the bins per bin row, bin rows (n2 / tile_y)
    int bstride;              // per-member stride of the start and task arrays (multiple of 4)
    int cstride;              // per-member stride of the count slice (scan workspace + counts)
    int nch;                  // chunks of DFS_SCAN_CHUNK bins
    int tile_y, c0, w, n2;
    long long budget;         // SM cycles the look-back waits at most (self-test)
};

// Layout of a member's count slice (cstride ints, zeroed before each
// set_points): the scan's ticket and completion counters, the bin-row flags
// (bytes), one 64-bit word a chunk, then the row counts.
__device__ __forceinline__ int *ws_ticket(int *slice) { return slice; }
__device__ __forceinline__ int *ws_done(int *slice) { return slice + 1; }
__device__ __forceinline__ unsigned char *ws_rows(int *slice) {
    return reinterpret_cast<unsigned char *>(slice + 4);
}
__device__ __forceinline__ unsigned long long *ws_chunks(int *slice) {
    return reinterpret_cast<unsigned long long *>(slice + 4 + DFS_MAX_ROW_BLOCKS / 4);
}

// Exclusive block-wide scan of (a, b) over the CTA's threads; returns the
// thread's prefixes and the totals.  blockDim.x <= 1024.
__device__ __forceinline__ void block_scan2(int a, int b, int &pa, int &pb, int &ta, int &tb) {
    __shared__ int s_a[32], s_b[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int xa = a, xb = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int ya = __shfl_up_sync(0xffffffffu, xa, o);
        const int yb = __shfl_up_sync(0xffffffffu, xb, o);
        if (lane >= o) {
            xa += ya;
            xb += yb;
        }
    }
    if (lane == 31) {
        s_a[wid] = xa;
        s_b[wid] = xb;
    }
    __syncthreads();
    if (wid == 0) {
        int va = lane < nw ? s_a[lane] : 0;
        int vb = lane < nw ? s_b[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ya = __shfl_up_sync(0xffffffffu, va, o);
            const int yb = __shfl_up_sync(0xffffffffu, vb, o);
            if (lane >= o) {
                va += ya;
                vb += yb;
            }
        }
        if (lane < nw) {
            s_a[lane] = va;
            s_b[lane] = vb;
        }
    }
    __syncthreads();
    pa = xa - a + (wid > 0 ? s_a[wid - 1] : 0);
    pb = xb - b + (wid > 0 ? s_b[wid - 1] : 0);
    ta = s_a[nw - 1];
    tb = s_b[nw - 1];
    __syncthreads();
}

// Run by every thread of the last CTA of a member once all its bin-row flags
// are published: the circular range of fine rows the stencils touch.  The
// points of bin row by use rows by*tile_y - c0 .. (by+1)*tile_y - c0 + w - 2,
// so the range is the complement of the longest circular run of empty bin
// rows (the first one in row order, of several), widened by the stencil and
// rounded out to whole row blocks.  Each thread measures the gaps after its
// bin rows; the longest wins a shared-memory maximum.
__device__ void rowrange_of_bits(const ScanParams &sp, const unsigned *s_bits, int *s_best,
                                 int2 *range_out) {
    const int tid = threadIdx.x, nb = sp.nbr;
    __syncthreads();                           // the bits, and *s_best = -1
    for (int i = tid; i < nb; i += blockDim.x) {
        if (!(s_bits[i >> 5] >> (i & 31) & 1)) continue;
        const int from = i + 1 == nb ? 0 : i + 1;
        const int gap = next_bit(s_bits, nb, from, 1) - from;    // i itself if it is alone
        atomicMax(s_best, (gap << 16) | (0xffff - i));
    }
    __syncthreads();
    if (tid == 0) {
        int2 range = make_int2(0, 0);
        if (*s_best >= 0) {
            const int best = *s_best >> 16;
            const int best_at = best ? 0xffff - (*s_best & 0xffff) + 1 : 0;
            // needed rows: after the gap, through the last non-empty bin row's stencil
            int first = ((best_at + best) % nb) * sp.tile_y - sp.c0;
            int cnt = (nb - best) * sp.tile_y + sp.w - 1;
            first &= sp.n2 - 1;
            const int fb = first & ~(DFS_ROW_BLOCK - 1);
            cnt = ((cnt + (first - fb) + DFS_ROW_BLOCK - 1) / DFS_ROW_BLOCK) * DFS_ROW_BLOCK;
            range = make_int2(fb, cnt < sp.n2 ? cnt : sp.n2);
        }
        *range_out = range;
    }
}

__device__ void finish_rowrange(const ScanParams &sp, const unsigned char *rows,
                                unsigned *s_bits, int *s_best, int2 *range_out) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    if (tid == 0) *s_best = -1;
    for (int k = wid; k * 32 < sp.nbr; k += nw) {
        const int i = k * 32 + lane;
        const unsigned b = __ballot_sync(0xffffffffu, i < sp.nbr && __ldcg(rows + i) != 0);
        if (lane == 0) s_bits[k] = b;
    }
    rowrange_of_bits(sp, s_bits, s_best, range_out);
}

// One chunk's word of the bin scan: 2 flag bits (0 not yet, 1 the chunk's own
// totals, 2 the totals through it, 3 the chunk gave up), 31 bits of non-empty
// bins, 31 of points.
__device__ __forceinline__ unsigned long long chunk_word(int flag, int ne, int sum) {
    return ((unsigned long long)flag << 62) | ((unsigned long long)ne << 31) |
           (unsigned long long)sum;
}

// The bin scan in one pass.  grid (nch, members), a thread a bin: the exclusive
// prefix of the bin's row counts (in place: the offset of each row inside the
// bin), its start, the list of non-empty bins in bin order and the bin-row
// flags.  A chunk's offsets come from the chunks before it by looking back
// (decoupled look-back, Merrill and Garland 2016): each publishes its own totals,
// then the totals through it, and warp 0 reads 32 words at a time until it meets
// one of the latter.  Chunks are taken by ticket, so every word waited for belongs
// to a CTA that is already running.  The last CTA of a member to finish finds the
// needed row range.
//
// The wait is bounded (DFS_WAIT_CYCLES, about a second).  A chunk that gives up
// sets DFS_STATUS_TIMEOUT, counts itself as failed in the upper half of the
// completion counter and tells the chunks after it; its starts are sums of fewer
// counts, so the scatter stays inside the member's slice, but the list and the
// records have gaps.  The last CTA then leaves n_tasks = -1 and an empty row range,
// whatever the chunks stored: no pass reads the list or the records, and the
// interpolation writes NaN.  SELFTEST: the same with a limit of the caller's, and
// chunk 0 publishes nothing, so that every other chunk gives up (a form of its own,
// since both as kernel parameters cost 1 us of the 42 of set_points).
//
// Bound by latency: a chain of a ticket, the row counts, two block scans and the
// words before it.  One kernel in place of a row prefix, chunk sums and a second
// scan pass whose last CTA searched the row gaps serially: 17 us in three
// launches -> 9.8 us (32768 bins), 13 -> 8 us (2048 bins).
template <bool SELFTEST>
__global__ void __launch_bounds__(DFS_SCAN_CHUNK) k_scan(ScanParams sp,
                                                         int *__restrict__ count_all,
                                                         int *__restrict__ start_all,
                                                         int2 *__restrict__ task_all,
                                                         int *__restrict__ n_tasks,
                                                         int2 *__restrict__ rowrange,
                                                         int *__restrict__ status) {
    dfs_grid_wait();
    __shared__ unsigned s_bits[(DFS_MAX_ROW_BLOCKS + 31) / 32];
    __shared__ int s_chunk, s_last, s_best, s_pre[2];
    bool failed = false;                       // warp 0's
    const int member = blockIdx.y, tid = threadIdx.x;
    int *slice = count_all + (size_t)member * sp.cstride;
    int *start = start_all + (size_t)member * sp.bstride;
    int2 *task = task_all + (size_t)member * sp.bstride;
    unsigned long long *words = ws_chunks(slice);
    unsigned char *rows = ws_rows(slice);
    if (tid == 0) s_chunk = atomicAdd(ws_ticket(slice), 1);
    __syncthreads();
    const int chunk = s_chunk;
    const int bin = chunk * DFS_SCAN_CHUNK + tid;
    int c = 0;
    if (bin < sp.nbins) {
        int *rc = slice + dfs_rowcount_offset(sp.nbins) + (size_t)bin * sp.tile_y;
        if ((sp.tile_y & 3) == 0 && sp.tile_y <= 32) {
            // all of the bin's row counts in flight at once (16-byte loads; the
            // slices keep 16-byte alignment), then the offsets stored over them
            const int nq = sp.tile_y >> 2;
            int4 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < nq) v[q] = reinterpret_cast<const int4 *>(rc)[q];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < nq) {
                    int4 o;
                    o.x = c;
                    o.y = o.x + v[q].x;
                    o.z = o.y + v[q].y;
                    o.w = o.z + v[q].z;
                    c = o.w + v[q].w;
                    reinterpret_cast<int4 *>(rc)[q] = o;
                }
        } else {
            for (int r = 0; r < sp.tile_y; ++r) {
                const int n = rc[r];
                rc[r] = c;
                c += n;
            }
        }
    }
    int ps, pn, ts, tn;
    block_scan2(c, c > 0, ps, pn, ts, tn);
    if (tid < 32) {
        int bs = 0, bn = 0;
        if (tid == 0 && !(SELFTEST && chunk == 0))
            *(volatile unsigned long long *)&words[chunk] = chunk_word(chunk ? 1 : 2, tn, ts);
        const long long budget = SELFTEST ? sp.budget : DFS_WAIT_CYCLES;
        const long long t0 = clock64();
        for (int base = chunk - 1; base >= 0; base -= 32) {
            const int idx = base - tid;
            unsigned long long w = chunk_word(2, 0, 0);
            bool late = false;
            if (idx >= 0) {
                volatile unsigned long long *p = &words[idx];
                while (((w = *p) >> 62) == 0 && !late) late = clock64() - t0 > budget;
                late |= (w >> 62) == 3;
            }
            failed = __any_sync(0xffffffffu, late);
            if (failed) break;
            const unsigned through = __ballot_sync(0xffffffffu, (w >> 62) == 2);
            const bool use = !through || tid <= __ffs(through) - 1;
            bs += __reduce_add_sync(0xffffffffu, use ? (int)(w & 0x7fffffff) : 0);
            bn += __reduce_add_sync(0xffffffffu, use ? (int)((w >> 31) & 0x7fffffff) : 0);
            if (through) break;
        }
        if (tid == 0) {
            if (failed && status) atomicExch(status, DFS_STATUS_TIMEOUT);
            if (chunk)
                *(volatile unsigned long long *)&words[chunk] =
                    chunk_word(failed ? 3 : 2, bn + tn, bs + ts);
            s_pre[0] = bs;
            s_pre[1] = bn;
        }
    }
    __syncthreads();
    const int base_s = s_pre[0], base_n = s_pre[1];
    if (bin < sp.nbins) {
        start[bin] = base_s + ps;
        if (c > 0) {
            task[base_n + pn] = make_int2(bin, base_s + ps);
            rows[bin >> sp.lnbx] = 1;
        }
    }
    if (chunk == sp.nch - 1 && tid == 0) {
        start[sp.nbins] = base_s + ts;
        task[base_n + tn] = make_int2(sp.nbins, base_s + ts);
        n_tasks[member] = base_n + tn;
    }
    // publish the flags, then count this CTA done
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const int add = failed ? 0x10001 : 1;              // at most 1024 chunks
        const int done = atomicAdd(ws_done(slice), add) + add;
        s_last = (done & 0xffff) == sp.nch ? done : 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    finish_rowrange(sp, rows, s_bits, &s_best, rowrange + member);
    if (tid == 0 && s_last > 0xffff) {
        n_tasks[member] = -1;
        rowrange[member] = make_int2(0, 0);
    }
}

// Points kept in the caller's order (DFSNUFFT_KEEP_ORDER): fold every point to
// its record at its own index, flag the bin rows it touches, and let the last
// CTA of the member find the needed row range.  grid (ceil(max member points /
// 256), members).
template <typename R>
__global__ void __launch_bounds__(256) k_fold_direct(const double *__restrict__ lon,
                                                     const double *__restrict__ colat,
                                                     FoldParams f, ScanParams sp,
                                                     const int *__restrict__ pofs,
                                                     int *__restrict__ count_all,
                                                     DfsPoints<R> pts,
                                                     int2 *__restrict__ rowrange) {
    __shared__ unsigned char s_row[DFS_MAX_ROW_BLOCKS];
    __shared__ unsigned s_bits[(DFS_MAX_ROW_BLOCKS + 31) / 32];
    __shared__ int s_last, s_best;
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int pl = blockIdx.x * blockDim.x + threadIdx.x;
    int *slice = count_all + (size_t)k * sp.cstride;
    unsigned char *rows = ws_rows(slice);
    for (int i = threadIdx.x; i < sp.nbr; i += blockDim.x) s_row[i] = 0;
    __syncthreads();
    if (pl < pofs[k + 1] - p0) {
        int bx, by;
        unsigned long long tx, ty;
        const bool ok = fold_point(f, lon[p0 + pl], colat[p0 + pl], bx, by, tx, ty);
        R ox = offset_value<R>(tx, f.odd_w), oy = offset_value<R>(ty, f.odd_w);
        if (!ok) ox = oy = (R)__int_as_float(0x7fc00000);
        pts.store((size_t)p0 + pl, bx | (by << 16), pl, ox, oy);
        s_row[by >> f.lty] = 1;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < sp.nbr; i += blockDim.x)
        if (s_row[i]) rows[i] = 1;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ws_done(slice), 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    finish_rowrange(sp, rows, s_bits, &s_best, rowrange + k);
}

// grid (ceil(max member points / 256), members): member k = blockIdx.y.  Each
// point's unsorted record goes to its sorted place in the member's slice
// [pofs[k], pofs[k+1]): bin start plus row offset plus rank.  The stored index
// is the member-local one.  One 16-byte store a point in FP32 (three stores of 8,
// 8 and 4 bytes before: 14.9 -> 13.6 us for 2.1M points).
template <typename R>
__global__ void __launch_bounds__(256) k_scatter(const FoldRec<R> *__restrict__ urec,
                                                 FoldParams f, const int *__restrict__ pofs,
                                                 int bstride, const int *__restrict__ start_all,
                                                 int cstride, int rowoff,
                                                 const int *__restrict__ count_all,
                                                 DfsPoints<R> pts) {
    dfs_grid_wait();
    const int k = blockIdx.y;
    const int p0 = pofs[k];
    const int pl = blockIdx.x * blockDim.x + threadIdx.x;
    if (pl >= pofs[k + 1] - p0) return;
    const FoldRec<R> rec = urec[p0 + pl];
    const int bx = rec.base & 0xffff, by = rec.base >> 16;
    const int pos = p0 + start_all[(size_t)k * bstride + bin_of(f, bx, by)] +
                    count_all[(size_t)k * cstride + rowoff + rowkey_of(f, bx, by)] + rec.rank;
    pts.store(pos, rec.base, pl, rec.tx, rec.ty);
}

// set_points of small members in one launch: a CTA a member, its row counts and
// their prefixes in shared memory, its points (at most SMALL_PPT a thread) in
// registers between the count and the store.  A step of a few thousand points is
// a chain of launches of 2 to 4 us each: 64 x 32 in FP64 (2048 points), a
// counter clear and three kernels of 14 us together before, 9.5 us in this form.
// Up to SMALL_POINTS points and SMALL_KEYS rows of bins: beyond, one SM's fold
// costs more than the launches.
constexpr int SMALL_PPT = 4, SMALL_POINTS = 1024 * SMALL_PPT, SMALL_KEYS = 8192;

template <typename R>
__global__ void __launch_bounds__(1024) k_points_small(const double *__restrict__ lon,
                                                       const double *__restrict__ colat,
                                                       FoldParams f, ScanParams sp,
                                                       const int *__restrict__ pofs,
                                                       DfsPoints<R> pts,
                                                       int2 *__restrict__ task_all,
                                                       int *__restrict__ n_tasks,
                                                       int2 *__restrict__ rowrange) {
    extern __shared__ int s_cnt[];                     // nbins x tile_y row counts
    __shared__ unsigned s_bits[(DFS_MAX_ROW_BLOCKS + 31) / 32];
    __shared__ int s_best;
    const int k = blockIdx.y, tid = threadIdx.x;
    const int p0 = pofs[k], n = pofs[k + 1] - p0;
    const int nkeys = sp.nbins * sp.tile_y;
    for (int i = tid; i < nkeys; i += blockDim.x) s_cnt[i] = 0;
    if (tid < (DFS_MAX_ROW_BLOCKS + 31) / 32) s_bits[tid] = 0;
    if (tid == 0) s_best = -1;
    __syncthreads();
    int base[SMALL_PPT], key[SMALL_PPT], rank[SMALL_PPT];
    R ox[SMALL_PPT], oy[SMALL_PPT];
#pragma unroll
    for (int u = 0; u < SMALL_PPT; ++u) {
        const int pl = tid + u * 1024;
        if (pl >= n) break;
        int bx, by;
        unsigned long long tx, ty;
        const bool ok = fold_point(f, lon[p0 + pl], colat[p0 + pl], bx, by, tx, ty);
        base[u] = bx | (by << 16);
        key[u] = rowkey_of(f, bx, by);
        ox[u] = offset_value<R>(tx, f.odd_w);
        oy[u] = offset_value<R>(ty, f.odd_w);
        if (!ok) ox[u] = oy[u] = (R)__int_as_float(0x7fc00000);
        rank[u] = atomicAdd(&s_cnt[key[u]], 1);
    }
    __syncthreads();
    // each bin's start and its rows' places, the list of non-empty bins
    int2 *task = task_all + (size_t)k * sp.bstride;
    int base_s = 0, base_n = 0;
    for (int b0 = 0; b0 < sp.nbins; b0 += blockDim.x) {
        const int bin = b0 + tid;
        int *rc = s_cnt + bin * sp.tile_y;
        int c = 0;
        if (bin < sp.nbins)
            for (int r = 0; r < sp.tile_y; ++r) c += rc[r];
        int ps, pn, ts, tn;
        block_scan2(c, c > 0, ps, pn, ts, tn);
        if (c > 0) {
            task[base_n + pn] = make_int2(bin, base_s + ps);
            atomicOr(&s_bits[(bin >> sp.lnbx) >> 5], 1u << ((bin >> sp.lnbx) & 31));
            int at = base_s + ps;
            for (int r = 0; r < sp.tile_y; ++r) {
                const int m = rc[r];
                rc[r] = at;
                at += m;
            }
        }
        base_s += ts;
        base_n += tn;
    }
    if (tid == 0) {
        task[base_n] = make_int2(sp.nbins, base_s);
        n_tasks[k] = base_n;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < SMALL_PPT; ++u) {
        const int pl = tid + u * 1024;
        if (pl >= n) break;
        pts.store((size_t)p0 + s_cnt[key[u]] + rank[u], base[u], pl, ox[u], oy[u]);
    }
    rowrange_of_bits(sp, s_bits, &s_best, rowrange + k);
}

template <typename R>
cudaError_t launch_points_small(dfsnufft_plan p, const double *lon, const double *colat,
                                const FoldParams &f, const ScanParams &sp) {
    const size_t smem = sizeof(int) * (size_t)sp.nbins * sp.tile_y;     // at most 32 KB
    k_points_small<R><<<dim3(1, p->n_members), 1024, smem, p->stream>>>(
        lon, colat, f, sp, p->d_pofs, dfs_points<R>(p), p->d_task_bin, p->d_n_tasks,
        p->d_rowrange);
    return cudaGetLastError();
}

int ilog2(int n) {
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

}  // namespace

cudaError_t dfs_launch_set_points(dfsnufft_plan p, const double *lon, const double *colat) {
    const dfsnufft_params &q = p->prm;
    FoldParams f;
    f.L1 = ilog2(q.n1);
    f.L2 = ilog2(q.n2);
    f.odd_w = q.w & 1;
    f.c0 = p->c0;
    f.w = q.w;
    f.ltx = ilog2(q.tile_x);
    f.lty = ilog2(q.tile_y);
    f.nbx = p->nbx;
    const int M = p->n_members;
    cudaError_t e;
    const int tpb = 256;
    const dim3 grid((unsigned)((p->max_member_points + tpb - 1) / tpb), M);
    ScanParams sp;
    sp.nbins = p->nbins;
    sp.bstride = p->bstride;
    sp.cstride = p->cstride;
    sp.nch = p->nch;
    sp.lnbx = ilog2(p->nbx);
    sp.nbr = q.n2 / q.tile_y;
    sp.tile_y = q.tile_y;
    sp.c0 = p->c0;
    sp.w = q.w;
    sp.n2 = q.n2;
    sp.budget = p->scan_budget;
    if (!p->keep_order && p->max_member_points <= SMALL_POINTS &&
        p->nbins * q.tile_y <= SMALL_KEYS)
        return q.dtype == DFSNUFFT_F64 ? launch_points_small<double>(p, lon, colat, f, sp)
                                       : launch_points_small<float>(p, lon, colat, f, sp);
    if ((e = cudaMemsetAsync(p->d_bin_count, 0, sizeof(int) * (size_t)M * p->cstride, p->stream)))
        return e;
    if (p->keep_order) {
        if (q.dtype == DFSNUFFT_F64)
            k_fold_direct<double><<<grid, tpb, 0, p->stream>>>(lon, colat, f, sp, p->d_pofs,
                                                              p->d_bin_count,
                                                              dfs_points<double>(p),
                                                              p->d_rowrange);
        else
            k_fold_direct<float><<<grid, tpb, 0, p->stream>>>(lon, colat, f, sp, p->d_pofs,
                                                             p->d_bin_count, dfs_points<float>(p),
                                                             p->d_rowrange);
        return cudaGetLastError();
    }
    const int rowoff = dfs_rowcount_offset(p->nbins);
    if (q.dtype == DFSNUFFT_F64)
        k_fold_count<double><<<grid, tpb, 0, p->stream>>>(lon, colat, f, p->d_pofs, p->cstride,
                                                          rowoff, p->d_bin_count,
                                                          (FoldRec<double> *)p->d_urec);
    else
        k_fold_count<float><<<grid, tpb, 0, p->stream>>>(lon, colat, f, p->d_pofs, p->cstride,
                                                         rowoff, p->d_bin_count,
                                                         (FoldRec<float> *)p->d_urec);
    // the kernels after the fold start launching while their predecessor drains
    if ((e = dfs_launch_dependent(sp.budget ? k_scan<true> : k_scan<false>, dim3(p->nch, M),
                                  dim3(DFS_SCAN_CHUNK), 0, p->stream, sp, p->d_bin_count,
                                  p->d_bin_start, p->d_task_bin, p->d_n_tasks, p->d_rowrange,
                                  p->d_status)))
        return e;
    if (q.dtype == DFSNUFFT_F64)
        return dfs_launch_dependent(k_scatter<double>, grid, dim3(tpb), 0, p->stream,
                                    (const FoldRec<double> *)p->d_urec, f, p->d_pofs, p->bstride,
                                    (const int *)p->d_bin_start, p->cstride, rowoff,
                                    (const int *)p->d_bin_count, dfs_points<double>(p));
    return dfs_launch_dependent(k_scatter<float>, grid, dim3(tpb), 0, p->stream,
                                (const FoldRec<float> *)p->d_urec, f, p->d_pofs, p->bstride,
                                (const int *)p->d_bin_start, p->cstride, rowoff,
                                (const int *)p->d_bin_count, dfs_points<float>(p));
}
