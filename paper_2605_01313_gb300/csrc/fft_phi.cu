// phi pass: the row FFTs of the oversampled 2-D inverse FFT (sign +1), the
// last FFT stage of the type-2 NUFFT evaluating Eq. 5.3 (Sec. 5).
//
// Only the real part of the fine grid is needed (the interpolation weights are
// real and the values are Re v), so each row is a complex-to-real transform:
// Re g(j) = sum_k H_k e^{2 pi i k j / n1} with H_k = (T_k + conj T_{-k}) / 2
// Hermitian.  With M = n1 / 2 and Z_k = (H_k + H_{k+M}) + i e^{2 pi i k / n1}
// (H_k - H_{k+M}), the length-M inverse FFT z of Z gives
// Re g(2j) = Re z_j and Re g(2j+1) = Im z_j.  T_k is the theta-pass value at
// phi-mode k mod n1 (zero outside the N1 modes).  A real-field plan's theta
// pass already transformed the Hermitian part of the coefficients, so its row
// holds H_k itself for k = 0..N1/2, and H_{-k} = conj H_k.  Each CTA handles CB
// rows inside the plan's needed row range; the row's values are staged in
// shared memory first, since every one of them enters two Z_k.  FP32 plans with
// fine rows of 2^7 to 2^13 cells run k_phi_pair (fft_phi_pair.cu) instead.
#include <type_traits>

#include "fft_core.cuh"
#include "df32.cuh"

using namespace dfs_fft;

namespace {

struct PhiArgs {
    int N1, n1, logm, n2;     // logm = log2(n1 / 2)
    int CB;                   // rows per CTA (divides DFS_ROW_BLOCK)
    int F;                    // fields per member (line f belongs to member f / F)
    int tcols, tpitch;        // theta-pass columns per row and row pitch
    int line0;                // first line (blockIdx.y = line - line0)
};

// grid (n2 / CB, lines); block CB * M/E threads, thread = (t, c) with t fastest.
// LOGM > 0 fixes the transform length at compile time; 0 takes it from a.logm.
// DF (FP64 plans): each fine-grid value is written as the double-single pair
// (hi, lo) of df32.cuh, the input of the double-single interpolation.
template <typename R, int E, int MAXT, int MINB, int LOGM, bool HERM, bool DF = false>
__global__ void __launch_bounds__(MAXT, MINB)
    k_phi_pass(PhiArgs a, const typename CxT<R>::type *__restrict__ in,
               const typename CxT<R>::type *__restrict__ tw,
               const typename CxT<R>::type *__restrict__ stw, const int2 *__restrict__ rowrange,
               R *__restrict__ grid, const int *__restrict__ cexp, int *__restrict__ emax) {
    dfs_grid_wait();
    typedef typename CxT<R>::type C;
    const int row0 = blockIdx.x * a.CB;
    const int2 rr = rowrange[(a.line0 + blockIdx.y) / a.F];
    // whole CTA (within one row block): no stencil touches these rows
    if (((row0 - rr.x) & (a.n2 - 1)) >= rr.y) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *smem = reinterpret_cast<C *>(smem_raw);
    const int M = LOGM ? (1 << LOGM) : (1 << a.logm);
    const int T = M / E;
    const int t = threadIdx.x % T;
    const int c = threadIdx.x / T;
    const int row = row0 + c;
    const int f = a.line0 + blockIdx.y;
    const C *src = in + (size_t)f * a.n2 * a.tpitch;
    R *dst = grid + ((size_t)f * a.n2 + row) * a.n1;
    const int half = a.N1 / 2;
    const int nmask = a.n1 - 1;
    C *sm = smem + (size_t)c * region_len<C>(M);
    C *srow = smem + (size_t)a.CB * region_len<C>(M) + (size_t)c * a.tcols;
    bool scaled = false;
    if constexpr (std::is_same<R, df32>::value) {
        // T's columns each carry their own power of two (cexp): the line's is the
        // largest, and each column is brought to it as it is staged
        scaled = cexp != nullptr;
        if (scaled) {
            __shared__ int s_emax;
            const int *ce = cexp + (size_t)f * a.tpitch;
            if (threadIdx.x == 0) s_emax = 0;
            int m = 0;
            for (int i = threadIdx.x; i < a.tcols; i += blockDim.x) m = max(m, ce[i]);
            // every thread of the warp is named (a CTA may have 8 or 16 threads), so the
            // lanes that took one column more join the others here
            m = __reduce_max_sync(blockDim.x >= 32 ? 0xffffffffu : (1u << blockDim.x) - 1, m);
            __syncthreads();
            if ((threadIdx.x & 31) == 0) atomicMax(&s_emax, m);
            __syncthreads();
            const int em = s_emax;
            if (threadIdx.x == 0) emax[f] = em;             // every CTA writes the same
            const int sl = df_line_shift(em);
            for (int i = t; i < a.tcols; i += T) {
                // at most 0 for finite lines; ce = 0 is a column of zeros
                const int d = df_line_shift(ce[i]) - sl;
                const float k = em >= 0x7ff ? 1.f
                                : ce[i] == 0 || d < -126 ? 0.f
                                                         : __int_as_float((127 + d) << 23);
                C v = t_load(src, row, i, a.tpitch);
                v.x = df32(v.x.hi * k, v.x.lo * k);
                v.y = df32(v.y.hi * k, v.y.lo * k);
                srow[i] = v;
            }
        }
    }
    if (!scaled)
        for (int i = t; i < a.tcols; i += T) srow[i] = t_load(src, row, i, a.tpitch);
    __syncthreads();
    auto hval = [&](int k) -> C {              // real-field rows: H_k, k taken mod n1
        k &= nmask;
        if (k <= half) return srow[k];
        if (k >= a.n1 - half) {
            const C v = srow[a.n1 - k];
            return cmake(v.x, -v.y);
        }
        return cmake((R)0, (R)0);
    };
    auto tval = [&](int k) -> C {              // T_k, k taken mod n1
        k &= nmask;
        int m;
        if (k < half) m = k;
        else if (k >= a.n1 - half) m = k - a.n1;
        else return cmake((R)0, (R)0);
        return srow[m + half];
    };
    auto ld = [&](int k) -> C {
        if constexpr (HERM) {
            const C h0 = hval(k), h1 = hval(k + M);
            const C d = cmul(cmake(h0.x - h1.x, h0.y - h1.y), ldt(&tw[k]));
            return cmake(h0.x + h1.x - d.y, h0.y + h1.y + d.x);
        }
        const C t0 = tval(k), t1 = tval(-k), t2 = tval(k + M), t3 = tval(M - k);
        // 2 H_k = T_k + conj T_{-k},  2 H_{k+M} = T_{k+M} + conj T_{M-k}
        const C h0 = cmake(t0.x + t1.x, t0.y - t1.y);
        const C h1 = cmake(t2.x + t3.x, t2.y - t3.y);
        const C d = cmul(cmake(h0.x - h1.x, h0.y - h1.y), ldt(&tw[k]));
        // (h0 + h1 + i d) / 2
        return cmake((R)0.5 * (h0.x + h1.x - d.y), (R)0.5 * (h0.y + h1.y + d.x));
    };
    auto st = [&](int j, C z) {
        if constexpr (std::is_same<R, df32>::value) {       // already double-single
            reinterpret_cast<float4 *>(dst)[j] = make_float4(z.x.hi, z.x.lo, z.y.hi, z.y.lo);
        } else if constexpr (DF) {
            const df32 h0 = split_double(z.x), h1 = split_double(z.y);
            reinterpret_cast<float4 *>(dst)[j] = make_float4(h0.hi, h0.lo, h1.hi, h1.lo);
        } else {
            reinterpret_cast<C *>(dst)[j] = z;
        }
    };
    if constexpr (LOGM > 0) line_fft_ct<LOGM, E>(stw, sm, t, ld, st);
    else line_fft<E>(a.logm, tw, 1, sm, t, ld, st);
}

// Per precision: elements per thread E, threads per CTA at most MAXT with MINB
// resident CTAs (MINBH for the rows of real-field plans); rows longer than
// E x MAXT complex values (FP32 fine grids of 8192 columns) use the wide form of
// MAXTW threads.  Double-single rows of real-field plans run with 64
// registers a thread, so that two CTAs share an SM (2048 x 1024 in FP64: 305 -> 256
// us): at most 8 bytes of spills at the compile-time lengths, 64 at the run-time
// one.  The general rows keep one CTA (117 registers; 40 bytes at the run-time
// length).
template <typename R> struct PhiCfg;
template <> struct PhiCfg<float> {
    static const int E = DFS_FFT_E, MAXT = 256, MINB = 3, MINBH = 3, MAXTW = 512;
};
template <> struct PhiCfg<double> {
    static const int E = DFS_FFT_E, MAXT = 512, MINB = 1, MINBH = 1, MAXTW = 512;
};
template <> struct PhiCfg<df32> {
    static const int E = DFS_FFT_E, MAXT = 512, MINB = 1, MINBH = 2, MAXTW = 512;
};

template <typename R, int MAXT, int MINB, int LOGM, bool HERM, bool DF>
cudaError_t run_phi_df(dfsnufft_plan p, const PhiArgs &a, size_t smem, dim3 grid, int threads) {
    typedef typename CxT<R>::type C;
    constexpr int E = PhiCfg<R>::E;
    cudaError_t e = allow_smem(k_phi_pass<R, E, MAXT, MINB, LOGM, HERM, DF>, smem);
    if (e) return e;
    const bool dfr = std::is_same<R, df32>::value;     // double-single tables
    return dfs_launch_dependent(k_phi_pass<R, E, MAXT, MINB, LOGM, HERM, DF>, grid,
                                dim3(threads), smem, p->stream, a, (const C *)p->d_T,
                                (const C *)(dfr ? p->d_df_tw1 : p->d_tw1),
                                (const C *)(dfr ? p->d_df_stw_phi : p->d_stw_phi),
                                (const int2 *)p->d_rowrange, (R *)p->d_G,
                                (const int *)(dfr && p->colscale ? p->d_cexp : nullptr),
                                p->d_emax);
}

// FP64 plans whose interpolation runs in double-single (p->gdf) take the DF form.
template <typename R, int MAXT, int MINB, int LOGM, bool HERM>
cudaError_t run_phi(dfsnufft_plan p, const PhiArgs &a, size_t smem, dim3 grid, int threads) {
    if constexpr (std::is_same<R, double>::value) {
        if (p->gdf) return run_phi_df<R, MAXT, MINB, LOGM, HERM, true>(p, a, smem, grid, threads);
    }
    return run_phi_df<R, MAXT, MINB, LOGM, HERM, false>(p, a, smem, grid, threads);
}

template <typename R, bool HERM>
cudaError_t dispatch_phi(dfsnufft_plan p, const PhiArgs &a, size_t smem, dim3 grid, int threads) {
    constexpr int MAXT = PhiCfg<R>::MAXT, MAXTW = PhiCfg<R>::MAXTW;
    constexpr int MINB = HERM ? PhiCfg<R>::MINBH : PhiCfg<R>::MINB;
    if (threads > MAXT) return run_phi<R, MAXTW, 1, 0, HERM>(p, a, smem, grid, threads);
    // compile-time lengths need the plan's stage-ordered table (double-single
    // for df32)
    if constexpr (!std::is_same<R, float>::value) {
        switch ((std::is_same<R, df32>::value ? p->d_df_stw_phi : p->d_stw_phi) ? a.logm : 0) {
            case 9: return run_phi<R, MAXT, MINB, 9, HERM>(p, a, smem, grid, threads);
            case 10: return run_phi<R, MAXT, MINB, 10, HERM>(p, a, smem, grid, threads);
            case 11: return run_phi<R, MAXT, MINB, 11, HERM>(p, a, smem, grid, threads);
            default: break;
        }
    }
    return run_phi<R, MAXT, MINB, 0, HERM>(p, a, smem, grid, threads);
}

template <typename R>
cudaError_t launch_phi(dfsnufft_plan p) {
    typedef typename CxT<R>::type C;
    constexpr int E = PhiCfg<R>::E, MAXT = PhiCfg<R>::MAXT;
    const dfsnufft_params &q = p->prm;
    PhiArgs a;
    a.N1 = q.N1;
    a.n1 = q.n1;
    a.logm = ilog2(q.n1) - 1;
    a.n2 = q.n2;
    a.F = p->n_fields;
    a.tcols = dfs_tcols(p->herm, q.N1);
    a.tpitch = dfs_tpitch(p->herm, q.N1);
    int lines;
    dfs_lines(p, a.line0, lines);
    const int M = q.n1 / 2;
    const int T = M / E;
    int cb = MAXT / T;
    if (cb < 1) cb = 1;
    if (cb > DFS_ROW_BLOCK) cb = DFS_ROW_BLOCK;
    const size_t per_row = sizeof(C) * (size_t)(region_len<C>(M) + a.tcols);
    while (cb > 1 && per_row * cb > 160 * 1024) cb >>= 1;
    // few rows: fewer a CTA (down to a warp), so that they spread over the SMs
    while (cb > 1 && cb * T > 32 && (q.n2 / cb) * lines < p->num_sms) cb >>= 1;
    a.CB = cb;
    const size_t smem = per_row * cb;
    const dim3 grid(q.n2 / cb, lines);
    if (p->herm) return dispatch_phi<R, true>(p, a, smem, grid, cb * T);
    return dispatch_phi<R, false>(p, a, smem, grid, cb * T);
}

}  // namespace

cudaError_t dfs_launch_phi_pass(dfsnufft_plan p) {
    if (p->gdf) return launch_phi<df32>(p);           // FP64 plans in double-single
    if (p->prm.dtype == DFSNUFFT_F64) return launch_phi<double>(p);
    const cudaError_t e = dfs_launch_phi_pair(p);
    return e == cudaErrorNotSupported ? launch_phi<float>(p) : e;
}
