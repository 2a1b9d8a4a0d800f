// theta pass of FP64 plans in double-single arithmetic (deconvolve, pad and the
// column FFTs; see fft_theta.cu for the input forms).
//
// Persistent CTAs take blocks of CB columns, whose N2 FP64 coefficient rows
// arrive in shared memory by 2-D TMA boxes while the block before is
// transformed.  A column is carried at its own power of two: the largest
// exponent of its coefficients (cexp, read back by the phi pass, which brings the
// columns of a line to one scale as it stages them), found in shared memory, so
// that no pass over the coefficients comes first.  The transform has length n2 with
// the modes in its first and last quarter: the first radix-8 stage adds nothing
// to the zeros between.
//
// Bound by FP32 instructions and the exchanges (49% of the issue slots).  2048 x
// 1024, three fields: an exponent pass of 40 us and a plain-load theta pass of 388
// us (16-byte strided loads) before, 344 us in this form with the butterflies'
// earlier arithmetic; 64 x 32: 39 us in two launches (two CTAs of 512 threads) to
// 20 us.
#include <string.h>

#include "coef_map.cuh"
#include "fft_core.cuh"
#include "tma.cuh"

using namespace dfs_fft;
using namespace dfs_coef;

namespace {

struct ThetaDfArgs {
    int N1, N2, n2;
    int nbq;                  // column blocks per line, ceil(tcols / CB)
    int total;                // nbq * lines (members x fields)
    int F;                    // fields per member (line f belongs to member f / F)
    int nbox, box_rows;       // TMA boxes per block and rows per box
    int in_elems;             // complex elements delivered per block
    unsigned tx_bytes;        // bytes delivered per block
    int tcols, tpitch;        // transformed columns, row pitch of T
    int col_base;             // array column of transformed column 0
    int line0;                // first line of the launch
};

// Columns a block: two (32-byte sectors of the coefficients and of T) where they
// leave CTAs of at most 512 threads; small CTAs, so that small grids spread over
// the SMs.
template <int LOGN> struct ThetaDfCfg {
    static constexpr int T = 1 << (LOGN - 3);                    // threads a column
    static constexpr int CB = T >= 512 ? 1 : T >= 16 ? 2 : 4;
    static constexpr int THREADS = CB * T;
    // resident CTAs the register budget (64 a thread) is set for
    static constexpr int MINB = 1024 / THREADS > 16 ? 16 : 1024 / THREADS;
};

// Biased exponent for the column scale.  A subnormal number counts as exponent 1
// (scale 2^1022), so that a column of them keeps its digits beside the line's
// other columns; 0 is left for zeros.
__device__ __forceinline__ int exp_of(double v) {
    const unsigned h = (unsigned)__double2hiint(v) & 0x7fffffffu;
    const int e = (int)(h >> 20);
    return e ? e : (h | (unsigned)__double2loint(v)) != 0;
}
__device__ __forceinline__ int exp_of(double2 v) { return max(exp_of(v.x), exp_of(v.y)); }

template <int LOGN, bool HERM>
__global__ void __launch_bounds__(ThetaDfCfg<LOGN>::THREADS, ThetaDfCfg<LOGN>::MINB)
    k_theta_df(ThetaDfArgs a, const __grid_constant__ CUtensorMap tmap,
               const double2 *__restrict__ coef, const df32 *__restrict__ inv1,
               const df32 *__restrict__ inv2, const dfc *__restrict__ stw,
               const int2 *__restrict__ rowrange, dfc *__restrict__ out,
               int *__restrict__ cexp, int *__restrict__ status) {
    dfs_grid_wait();
    constexpr int E = DFS_FFT_E, n2 = 1 << LOGN, T = n2 / E, CB = ThetaDfCfg<LOGN>::CB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    uint64_t *bar = reinterpret_cast<uint64_t *>(base);
    int *s_exp = reinterpret_cast<int *>(base + 16);         // 2 x CB, by block parity
    double2 *nyq = reinterpret_cast<double2 *>(base + 64);   // CB (at most 4) values
    double2 *in = reinterpret_cast<double2 *>(base + 128);
    dfc *ex = reinterpret_cast<dfc *>(in + a.in_elems);
    const int c = threadIdx.x % CB;
    const int t = threadIdx.x / CB;
    const int half = a.N2 / 2;                     // at most n2 / 4
    dfc *sm = ex + (size_t)c * region_stride<dfc>(n2, CB);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    if (threadIdx.x < 2 * CB) s_exp[threadIdx.x] = 0;
    __syncthreads();
    auto issue = [&](int blk) {                    // thread 0
        const int f = a.line0 + blk / a.nbq;
        const int qb = blk - (f - a.line0) * a.nbq;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(bar, a.tx_bytes);
        const int x = (a.col_base + qb * CB) * 2;  // 8-byte units
        for (int i = 0; i < a.nbox; ++i)
            tma_load_2d(in + (size_t)i * a.box_rows * CB, &tmap, x, f * a.N2 + i * a.box_rows, bar);
    };
    uint32_t phase = 0;
    if (threadIdx.x == 0 && (int)blockIdx.x < a.total) issue(blockIdx.x);
    for (int blk = blockIdx.x; blk < a.total; blk += gridDim.x) {
        const int nxt = blk + gridDim.x;
        const int f = a.line0 + blk / a.nbq;
        const int qb = blk - (f - a.line0) * a.nbq;
        if (HERM && threadIdx.x < CB) {
            // c_{-N2/2,-m} of each column (the mirror of the Nyquist row)
            const int q = qb * CB + threadIdx.x;
            nyq[threadIdx.x] = q < a.tcols ? coef[(size_t)f * a.N2 * a.N1 + (a.N1 - a.col_base - q)]
                                           : make_double2(0.0, 0.0);
        }
        const int q = qb * CB + c;                 // column of T
        const int qa = a.col_base + q;             // array column
        const bool col_ok = q < a.tcols;
        const df32 sq = col_ok ? inv1[qa < a.N1 ? qa : 0] : df32(0.f, 0.f);
        const int2 rr = rowrange[f / a.F];
        const bool ok = mbar_wait_bounded(bar, phase);
        if (__syncthreads_or(!ok)) {
            // give up on this launch; let copies still in flight land first
            if (threadIdx.x == 0) {
                atomicExch(status, DFS_STATUS_TIMEOUT);
                mbar_wait_bounded(bar, phase);
            }
            __syncthreads();
            return;
        }
        phase ^= 1;
        const double2 *cf0 = coef + (size_t)f * a.N2 * a.N1;
        const bool k_zero = HERM && q == 0;        // m = 0: its own mirror
        const bool k_nyq = HERM && qa == a.N1;     // m = N1/2: mirror of the Nyquist column
        // array entry of mode n, -half <= n < half (column m = N1/2: of its mirror)
        auto raw = [&](int n) -> double2 {
            if (HERM && k_nyq) return cf0[(size_t)(n == -half ? 0 : half - n) * a.N1];
            return in[(n + half) * CB + c];
        };
        // the column's largest exponent; s_exp of the other parity is reset for the
        // next block
        int *se = s_exp + (phase ? CB : 0);
        {
            int m = 0;
            if (col_ok) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int i = t + e * T;
                    if (e < 2 && i < half) m = max(m, exp_of(raw(i)));
                    if (e >= 6 && i >= n2 - half) m = max(m, exp_of(raw(i - n2)));
                }
                if (HERM && t == 0) m = max(m, exp_of(nyq[c]));
            }
#pragma unroll
            for (int o = 16; o >= CB; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            if ((threadIdx.x & 31) < CB) atomicMax(&se[c], m);
            if (threadIdx.x < CB) s_exp[(phase ? 0 : CB) + threadIdx.x] = 0;
        }
        __syncthreads();
        const int ce = se[c];
        const int sh = df_line_shift(ce);
        if (t == 0 && col_ok) cexp[(size_t)f * a.tpitch + q] = ce;
        // h_{n,m} (real-field plans, see herm_coef) or c_{n,m}, deconvolved
        auto coef_nm = [&](int n) -> dfc {
            dfc v;
            if (HERM && n == half) {
                if (k_nyq) v = cconj(to_dfc_scaled(cf0[0], sh));
                else v = cconj(to_dfc_scaled(nyq[c], sh));
                v = cscale(v, df32(0.5f, 0.f));
            } else {
                v = to_dfc_scaled(raw(n), sh);
                if constexpr (HERM) {
                    if (k_nyq) {
                        if (n == -half) v = cmake(df32(0.f, 0.f), df32(0.f, 0.f));
                        else v = cscale(cconj(v), df32(0.5f, 0.f));
                    } else if (n == -half) {
                        v = cscale(v, df32(0.5f, 0.f));
                    } else if (k_zero) {
                        v = cscale(v + cconj(to_dfc_scaled(raw(-n), sh)), df32(0.5f, 0.f));
                    }
                }
            }
            const int r = n + half;
            return cscale(v, sq * inv2[r < a.N2 ? r : 0]);
        };
        const dfc zero = cmake(df32(0.f, 0.f), df32(0.f, 0.f));
        auto input = [&](int i, int n) -> dfc {
            if (!col_ok || n < -half || n > half || (!HERM && n == half)) return zero;
            return coef_nm(n);
        };
        // first stage: inputs t + e T, the modes n >= 0 at e = 0, 1 and n < 0 at
        // e = 6, 7 (half <= 2 T); v2 .. v5 are zero but for the mode n = +half of a
        // real-field plan, at e = 2 of thread 0 when half = 2 T
        dfc v[E];
        {
            const dfc a0 = input(t, t), a1 = input(t + T, t + T);
            const dfc a6 = input(t + 6 * T, t - 2 * T), a7 = input(t + 7 * T, t - T);
            v[0] = a0;
            v[4] = a0;
            v[1] = a1;
            v[5] = tw16<2>(a1);
            v[2] = a6;
            v[6] = tw16<12>(a6);                   // i (0 - a6)
            v[3] = a7;
            v[7] = tw16<14>(a7);                   // e^{3 pi i / 4} (0 - a7)
            if (HERM && col_ok && t == 0 && half == 2 * T) {
                const dfc y = coef_nm(half);
                v[2] = v[2] + y;
                v[6] = v[6] + tw16<4>(y);
            }
        }
        dif_levels<8, 0, 1, 2>(v);
#pragma unroll
        for (int r = 0; r < 8; ++r) sm[spad<dfc>(t * 8 + bitrev(r, 8))] = v[r];
        dfc *dst = out + (size_t)f * n2 * a.tpitch + q;
        auto st = [&](int i, dfc z) {
            if (col_ok && ((i - rr.x) & (n2 - 1)) < rr.y) dst[(size_t)i * a.tpitch] = z;
        };
        auto refill = [&]() {
            if (threadIdx.x == 0 && nxt < a.total) issue(nxt);
        };
        ct_stages<LOGN, E, 3>(v, t, stw, sm, st, refill);
    }
}

template <int LOGN, bool HERM>
cudaError_t run(dfsnufft_plan p, ThetaDfArgs &a, const void *coeffs) {
    typedef ThetaDfCfg<LOGN> Cfg;
    const dfsnufft_params &q = p->prm;
    constexpr int CB = Cfg::CB, n2 = 1 << LOGN;
    a.nbq = (a.tcols + CB - 1) / CB;
    int line0, lines;
    dfs_lines(p, line0, lines);
    a.line0 = line0;
    a.total = a.nbq * lines;
    constexpr int ra = 128 / (CB * (int)sizeof(double2));      // box rows of 128 bytes
    a.box_rows = q.N2 < 256 ? ((q.N2 + ra - 1) / ra * ra) : 256;
    a.nbox = (q.N2 + a.box_rows - 1) / a.box_rows;
    a.in_elems = a.nbox * a.box_rows * CB;
    a.tx_bytes = (unsigned)(sizeof(double2) * a.in_elems);
    const size_t smem = 256 + sizeof(double2) * (size_t)a.in_elems +
                        sizeof(dfc) * (size_t)CB * region_len<dfc>(n2);
    if (smem > 226 * 1024) return cudaErrorNotSupported;
    CUtensorMap tmap;
    if (dfs_encode_tensor_map_2d(&tmap, coeffs, (uint64_t)q.N1 * 2,
                                 (uint64_t)q.N2 * (line0 + lines), sizeof(double2) * (uint64_t)q.N1,
                                 (uint32_t)(CB * 2), (uint32_t)a.box_rows))
        return cudaErrorNotSupported;              // no encoder: the plain-load pass
    auto kern = k_theta_df<LOGN, HERM>;
    cudaError_t e = allow_smem(kern, smem);
    if (e) return e;
    int per_sm = (int)(226 * 1024 / (smem + 1024));
    if (per_sm > Cfg::MINB) per_sm = Cfg::MINB;
    if (per_sm < 1) per_sm = 1;
    int grid = (p->num_sms > 0 ? p->num_sms : 1) * per_sm;
    if (grid > a.total) grid = a.total;
    e = dfs_launch_dependent(kern, dim3(grid), dim3(Cfg::THREADS), smem, p->stream, a, tmap,
                             (const double2 *)coeffs, (const df32 *)p->d_df_inv1,
                             (const df32 *)p->d_df_inv2, (const dfc *)p->d_df_stw_theta,
                             (const int2 *)p->d_rowrange, (dfc *)p->d_T, p->d_cexp, p->d_status);
    if (!e) p->colscale = 1;
    return e;
}

template <int LOGN>
cudaError_t dispatch(dfsnufft_plan p, ThetaDfArgs &a, const void *coeffs, int logn) {
    if constexpr (LOGN > 12) {
        return cudaErrorNotSupported;
    } else {
        if (logn != LOGN) return dispatch<LOGN + 1>(p, a, coeffs, logn);
        return p->herm ? run<LOGN, true>(p, a, coeffs) : run<LOGN, false>(p, a, coeffs);
    }
}

}  // namespace

// Plans with double-single tables, 2^6 to 2^12 fine rows (longer columns do not
// fit 512 threads), coefficients on a 16-byte boundary.
cudaError_t dfs_launch_theta_df(dfsnufft_plan p, const void *coeffs) {
    const dfsnufft_params &q = p->prm;
    const int logn = ilog2(q.n2);
    if (logn < 6 || !p->d_status || !p->d_df_stw_theta || !p->d_cexp ||
        ((uintptr_t)coeffs & 15) != 0)
        return cudaErrorNotSupported;
    ThetaDfArgs a;
    memset(&a, 0, sizeof(a));
    a.N1 = q.N1;
    a.N2 = q.N2;
    a.n2 = q.n2;
    a.F = p->n_fields;
    a.tcols = dfs_tcols(p->herm, q.N1);
    a.tpitch = dfs_tpitch(p->herm, q.N1);
    a.col_base = p->herm ? q.N1 / 2 : 0;
    return dispatch<6>(p, a, coeffs, logn);
}
