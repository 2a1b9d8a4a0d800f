// theta pass of FP32 plans (deconvolve, pad and the column FFTs of the
// oversampled 2-D inverse FFT, a middle stage of the type-2 NUFFT evaluating
// Eq. 5.3, Sec. 5; see fft_theta.cu for the input forms and the Hermitian part
// a real-field plan transforms).
//
// Persistent CTAs take blocks of CB columns.  The block's N2 coefficient rows
// arrive in shared memory by 2-D TMA boxes (rows of CB x 8 bytes).  Each
// column's length-n2 transform is two length-n2/2 transforms, output rows 2q
// and 2q + 1 (the modes fit in n2/2; when n2 = 2 N2 the two Nyquist modes
// n = -N2/2 and n = +N2/2 of a real-field plan share index N2/2 and are added
// there).  They run packed in the same threads (fft_pair.cuh): twiddles, index
// arithmetic, barriers and the stores of T serve both.  One input buffer is
// enough: the next block's boxes are issued once every thread has read its
// inputs (after the transforms' first barrier) and land meanwhile.
#include <string.h>

#include "coef_map.cuh"
#include "fft_pair.cuh"

using namespace dfs_fft;
using namespace dfs_coef;

namespace {

struct ThetaPairArgs {
    int N1, N2, n2;
    int nbq;                  // column blocks per line, ceil(tcols / CB)
    int total;                // nbq * lines (members x fields)
    int F;                    // fields per member (line f belongs to member f / F)
    int nbox, box_rows;       // TMA boxes per block and rows per box
    int in_elems;             // complex elements delivered per block
    unsigned tx_bytes;        // bytes delivered per block
    int tcols, tpitch;        // transformed columns, row pitch of T
    int col_base;             // array column of transformed column 0
    int prM, prN;             // partial-regularity input: truncation (prM < 0: complex input)
    int line0;                // first line of the launch (blocks cover lines line0 ..)
};

// Columns a block: CTAs of 256 threads where a column takes fewer (more columns
// also make longer box rows and longer runs of stores), two columns (16-byte
// boxes, the TMA minimum; 32-byte stores) where it takes 128 or more.  Two
// columns a CTA at every length, with a run-time-length transform below 2^10
// and above 2^12 fine rows, left the short columns with 32 to 128 threads a CTA
// and two CTAs an SM; measured before and after, 48 lines of real fields:
// 128 fine rows' half length 82 -> 11 us, 256 147 -> 19, 512 99 -> 43, 1024
// 262 -> 169, and three lines of 4096 678 -> 229 us.
template <int LOGH> struct ThetaPairCfg {
    static constexpr int T = 1 << (LOGH - 3);                    // threads a column
    static constexpr int CB = T >= 128 ? 2 : T >= 16 ? 256 / T : 16;
    static constexpr int THREADS = CB * T;
    // resident CTAs the register budget (64 a thread) is set for
    static constexpr int MINB = THREADS >= 1024 ? 1 : THREADS >= 256 ? 1024 / THREADS : 6;
};

// PRIN (real-field plans): the input is partial-regularity DFS coefficients,
// lines x (prM + 1) x (prN + 1) complex, whose column m is contiguous; a block's
// CB columns are staged by 8-byte asynchronous copies of every thread instead of
// TMA boxes (the columns are not 16-byte aligned), completing on the same
// mbarrier, and converted on the fly by pr_coef.
template <int LOGH, bool HERM, bool PRIN>
__global__ void __launch_bounds__(ThetaPairCfg<LOGH>::THREADS, ThetaPairCfg<LOGH>::MINB)
    k_theta_pair(ThetaPairArgs a, const __grid_constant__ CUtensorMap tmap,
                 const float2 *__restrict__ coef, const float *__restrict__ inv1,
                 const float *__restrict__ inv2, const float2 *__restrict__ tw,
                 const float2 *__restrict__ stw, const int2 *__restrict__ rowrange,
                 PairC *__restrict__ out, int *__restrict__ status) {
    dfs_grid_wait();
    typedef float2 C;
    constexpr int E = DFS_FFT_E, H = 1 << LOGH, T = H / E, CB = ThetaPairCfg<LOGH>::CB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // TMA destinations start on 128-byte boundaries (base rounded up here; box
    // sizes are multiples of 128 bytes by construction)
    unsigned char *base = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);
    uint64_t *bar = reinterpret_cast<uint64_t *>(base);
    C *in = reinterpret_cast<C *>(base + 128);
    PairC *ex = reinterpret_cast<PairC *>(in + a.in_elems);
    C *nyq = reinterpret_cast<C *>(ex + (size_t)CB * pair_region_stride(H, CB));
    float *f2 = reinterpret_cast<float *>(nyq + CB);                 // 1 / phihat2
    const int c = threadIdx.x % CB;
    const int t = threadIdx.x / CB;
    const int half = a.N2 / 2;                     // at most H / 2
    PairC *sm = ex + (size_t)c * pair_region_stride(H, CB);
    for (int i = threadIdx.x; i < a.N2; i += blockDim.x) f2[i] = inv2[i];
    if (threadIdx.x == 0) {
        // PRIN: every thread arrives once a phase, when its copies have landed
        mbar_init(bar, PRIN ? blockDim.x : 1);
        fence_mbar_init();
    }
    __syncthreads();
    const int prs = a.prN + 1;                     // PRIN: staged elements a column
    // issued by thread 0 (TMA boxes), or by every thread (PRIN)
    auto issue = [&](int blk) {
        const int f = a.line0 + blk / a.nbq;
        const int qb = blk - (f - a.line0) * a.nbq;
        if constexpr (PRIN) {
            for (int cc = 0; cc < CB; ++cc) {
                const int q = qb * CB + cc;
                if (q > a.prM) break;
                const C *src = coef + ((size_t)f * (a.prM + 1) + q) * prs;
                for (int k = threadIdx.x; k < prs; k += blockDim.x)
                    cp_async_8(in + (size_t)cc * prs + k, src + k);
            }
            cp_async_mbar_arrive_noinc(bar);
        } else {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(bar, a.tx_bytes);
            const int x = a.col_base + qb * CB;
            for (int i = 0; i < a.nbox; ++i)
                tma_load_2d(in + (size_t)i * a.box_rows * CB, &tmap, x, f * a.N2 + i * a.box_rows,
                            bar);
        }
    };
    uint32_t phase = 0;
    const bool issuer = PRIN || threadIdx.x == 0;
    if (issuer && (int)blockIdx.x < a.total) issue(blockIdx.x);
    const C wt = ldt(&tw[t]);
    for (int blk = blockIdx.x; blk < a.total; blk += gridDim.x) {
        const int nxt = blk + gridDim.x;
        const int f = a.line0 + blk / a.nbq;
        const int qb = blk - (f - a.line0) * a.nbq;
        if (HERM && !PRIN && threadIdx.x < CB) {
            // conj c_{-N2/2,-m} of each column (the mirror of the Nyquist row),
            // fetched while the block's boxes land
            const int q = qb * CB + threadIdx.x;
            C v = cmake(0.f, 0.f);
            if (q < a.tcols) v = coef[(size_t)f * a.N2 * a.N1 + (a.N1 - a.col_base - q)];
            nyq[threadIdx.x] = cconj(v);
        }
        const int q = qb * CB + c;                     // column of T
        const int qa = a.col_base + q;                 // array column
        const bool col_ok = q < a.tcols;
        const float sq = col_ok ? inv1[qa < a.N1 ? qa : 0] : 0.f;
        const int2 rr = rowrange[f / a.F];
        const bool ok = mbar_wait_bounded(bar, phase);
        phase ^= 1;
        if (__syncthreads_or(!ok)) {
            // give up on this launch; let copies still in flight land first
            if constexpr (PRIN) {
                cp_async_wait_all();
                if (threadIdx.x == 0) atomicExch(status, DFS_STATUS_TIMEOUT);
            } else if (threadIdx.x == 0) {
                atomicExch(status, DFS_STATUS_TIMEOUT);
                mbar_wait_bounded(bar, phase ^ 1);
            }
            __syncthreads();
            return;
        }
        const C *cf0 = coef + (size_t)f * a.N2 * a.N1;
        PairC *dst = out + (size_t)f * (a.n2 >> 1) * a.tpitch + q;
        const bool k_zero = HERM && q == 0;            // m = 0: its own mirror
        const bool k_nyq = HERM && qa == a.N1;         // m = N1/2: mirror of the Nyquist column
        // h_{n,m} (real-field plans, see herm_coef) or c_{n,m}, deconvolved
        auto coef_nm = [&](int n) -> C {
            const int r = n + half;
            if constexpr (PRIN) {
                if (q > a.prM || n > a.prN || n < -a.prN) return cmake(0.f, 0.f);
                return cscale(pr_coef<C>(n, q, a.prN, in + (size_t)c * prs), sq * f2[r]);
            }
            C v;
            if constexpr (HERM) {
                if (k_nyq) {                           // one column per line: global loads
                    v = n == -half ? cmake(0.f, 0.f)
                                   : cscale(cconj(cf0[(size_t)(half - n) * a.N1]), 0.5f);
                } else if (n == half) {
                    v = cscale(nyq[c], 0.5f);
                } else {
                    v = in[r * CB + c];
                    if (n == -half) {
                        v = cscale(v, 0.5f);
                    } else if (k_zero) {
                        const C mirror = in[(a.N2 - r) * CB + c];
                        v = cscale(cmake(v.x + mirror.x, v.y - mirror.y), 0.5f);
                    }
                }
            } else {
                v = in[r * CB + c];
            }
            return cscale(v, sq * f2[r < a.N2 ? r : 0]);
        };
        // Inputs i = t + e T of both transforms: y_n and y_n e^{2 pi i n / n2}.
        // The twiddle is e^{2 pi i t / n2} e^{i pi e / 8}, negated for n = i - H:
        // one table read a thread, the rest rotations by constants.  The modes
        // n >= 0 sit in the first half of the inputs (half <= H / 2), n < 0 in
        // the second.
        PairC v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int i = t + e * T;
            C y0 = cmake(0.f, 0.f), y1 = y0;
            const C wi = cmul(wt, cmake((float)c16(e), (float)s16(e)));
            if (e < E / 2) {
                if (col_ok && i < half) {
                    y0 = coef_nm(i);
                    y1 = cmul(y0, wi);
                }
            } else if (col_ok && i >= H - half) {
                y0 = coef_nm(i - H);
                const C z = cmul(y0, wi);
                y1 = cmake(-z.x, -z.y);
            }
            v[e] = pair_of(y0, y1);
        }
        if (HERM && col_ok && t == (half & (T - 1))) {     // the mode n = +half
            const C y = coef_nm(half);
            const PairC z = pair_of(y, cmul(y, ldt(&tw[half])));
            const int eh = half / T;
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (e == eh) v[e] = v[e] + z;
        }
        // the needed rows come in blocks of 16: both rows of a pair or neither
        auto st = [&](int qq, PairC z) {
            if (col_ok && ((2 * qq - rr.x) & (a.n2 - 1)) < rr.y)
                dst[(size_t)qq * a.tpitch] = z;
        };
        auto refill = [&]() {
            if (issuer && nxt < a.total) issue(nxt);
        };
        pair_fft<LOGH, false>(stw, sm, t, 0, v, st, refill);
        __syncthreads();
    }
}

template <int LOGH, bool HERM, bool PRIN>
cudaError_t run(dfsnufft_plan p, ThetaPairArgs &a, const void *coeffs) {
    typedef ThetaPairCfg<LOGH> Cfg;
    const dfsnufft_params &q = p->prm;
    constexpr int CB = Cfg::CB, H = 1 << LOGH;
    a.nbq = (a.tcols + CB - 1) / CB;
    int line0, lines;
    dfs_lines(p, line0, lines);
    a.line0 = line0;
    a.total = a.nbq * lines;
    // boxes of CB columns x box_rows rows, each a multiple of 128 bytes (box
    // destinations stay 128-byte aligned): box_rows a multiple of ra rows
    constexpr int ra = CB * (int)sizeof(float2) >= 128 ? 1 : 128 / (CB * (int)sizeof(float2));
    a.box_rows = q.N2 < 256 ? ((q.N2 + ra - 1) / ra * ra) : 256;
    a.nbox = (q.N2 + a.box_rows - 1) / a.box_rows;
    a.in_elems = a.nbox * a.box_rows * CB;
    a.tx_bytes = (unsigned)(sizeof(float2) * a.in_elems);
    if (PRIN && (long long)CB * (a.prN + 1) > a.in_elems) return cudaErrorNotSupported;
    const size_t smem = 256 + sizeof(float2) * (size_t)a.in_elems +
                        sizeof(PairC) * (size_t)CB * pair_region_stride(H, CB) +
                        sizeof(float2) * CB + sizeof(float) * (size_t)q.N2;
    if (smem > 226 * 1024) return cudaErrorNotSupported;
    CUtensorMap tmap;
    memset(&tmap, 0, sizeof(tmap));             // unused by the partial-regularity form
    if (!PRIN) {
        cudaError_t e = dfs_encode_tensor_map_2d(&tmap, coeffs, (uint64_t)q.N1,
                                                 (uint64_t)q.N2 * (line0 + lines),
                                                 sizeof(float2) * (uint64_t)q.N1, (uint32_t)CB,
                                                 (uint32_t)a.box_rows);
        if (e) return cudaErrorNotSupported;   // no encoder: the plain-load pass
    }
    auto kern = k_theta_pair<LOGH, HERM, PRIN>;
    cudaError_t e = allow_smem(kern, smem);
    if (e) return e;
    int per_sm = (int)(226 * 1024 / (smem + 1024));
    if (per_sm > Cfg::MINB) per_sm = Cfg::MINB;
    if (per_sm < 1) per_sm = 1;
    int grid = (p->num_sms > 0 ? p->num_sms : 1) * per_sm;
    if (grid > a.total) grid = a.total;
    return dfs_launch_dependent(kern, dim3(grid), dim3(Cfg::THREADS), smem, p->stream, a, tmap,
                                (const float2 *)coeffs, (const float *)p->d_inv1,
                                (const float *)p->d_inv2, (const float2 *)p->d_tw2,
                                (const float2 *)p->d_stw_theta, (const int2 *)p->d_rowrange,
                                (PairC *)p->d_T, p->d_status);
}

template <int LOGH>
cudaError_t dispatch(dfsnufft_plan p, ThetaPairArgs &a, const void *coeffs, int logh) {
    if constexpr (LOGH > DFS_PAIR_MAX_LOG) {
        return cudaErrorNotSupported;
    } else {
        if (logh != LOGH) return dispatch<LOGH + 1>(p, a, coeffs, logh);
        if (a.prM >= 0) return run<LOGH, true, true>(p, a, coeffs);
        return p->herm ? run<LOGH, true, false>(p, a, coeffs)
                       : run<LOGH, false, false>(p, a, coeffs);
    }
}

}  // namespace

// prM >= 0: partial-regularity input (real-field plans).  Taken by plans that
// own their tables (status word, stage-ordered twiddles) at fine sizes of
// 2^(DFS_PAIR_MIN_LOG + 1) .. 2^(DFS_PAIR_MAX_LOG + 1) rows; complex input must
// start on 16 bytes and its first box column too.
cudaError_t dfs_launch_theta_pair(dfsnufft_plan p, const void *coeffs, int prM, int prN) {
    const dfsnufft_params &q = p->prm;
    const int logh = ilog2(q.n2) - 1;
    if (logh < DFS_PAIR_MIN_LOG || !p->d_status || !p->d_stw_theta) return cudaErrorNotSupported;
    ThetaPairArgs a;
    memset(&a, 0, sizeof(a));
    a.N1 = q.N1;
    a.N2 = q.N2;
    a.n2 = q.n2;
    a.F = p->n_fields;
    a.tcols = dfs_tcols(p->herm, q.N1);
    a.tpitch = dfs_tpitch(p->herm, q.N1);
    a.col_base = p->herm ? q.N1 / 2 : 0;
    a.prM = prM;
    a.prN = prN;
    if (prM >= 0) {
        if (!p->herm || ((uintptr_t)coeffs & (sizeof(float2) - 1)) != 0)
            return cudaErrorNotSupported;
    } else if (((uintptr_t)coeffs & 15) != 0 || (a.col_base * sizeof(float2)) % 16 != 0) {
        return cudaErrorNotSupported;
    }
    return dispatch<DFS_PAIR_MIN_LOG>(p, a, coeffs, logh);
}
