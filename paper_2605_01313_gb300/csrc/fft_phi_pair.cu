// phi pass of FP32 plans: the row FFTs of the oversampled 2-D inverse FFT, each
// row a complex-to-real transform done as a half-length complex one (see
// fft_phi.cu for the algebra), two rows packed in the same threads
// (fft_pair.cuh).
//
// A CTA takes NP row pairs.  With M = n1 / 2 and N1 <= M, input k of the
// length-M transform is Z_k = (1 + i w_k) H_k for k <= N1/2 and
// Z_k = (1 - i w_k) conj H_{M-k} for k >= M - N1/2 (zero between; both are
// added at k = M/2 when N1 = M), w_k = e^{2 pi i k / n1}.  Each thread reads its
// eight inputs straight from the theta pass's output, all in flight at once and
// each value twice (the second read hits the L1 cache): no staging pass over
// shared memory and no barrier before the transform.  Bound by the shared-memory
// and global-access wavefronts (79% of the L1 data pipe at 2048 x 1024).
// Measured against the staged, scalar form: three lines of 2080 rows x 4096
// cells 58 -> 40 us, of 4112 x 8192 (run-time length before) 488 -> 165 us, 48
// lines of 2048 cells 212 -> 139 us.
#include "fft_pair.cuh"

using namespace dfs_fft;

namespace {

struct PhiPairArgs {
    int N1, n1, n2;
    int F;                    // fields per member (line f belongs to member f / F)
    int tpitch;               // row pitch of T
    int line0;                // first line (blockIdx.y = line - line0)
};

// Row pairs a CTA: 256 threads where a row takes fewer, at most the 8 pairs of
// a needed-row block of 16 (so that a whole CTA is needed or not).
template <int LOGM> struct PhiPairCfg {
    static constexpr int T = 1 << (LOGM - 3);                    // threads a row pair
    static constexpr int NP = T >= 256 ? 1 : 256 / T > 8 ? 8 : 256 / T;
    static constexpr int THREADS = NP * T;
    // resident CTAs the register budget (64 a thread) is set for
    static constexpr int MINB = 1024 / THREADS > 8 ? 8 : 1024 / THREADS;
};
static_assert(DFS_ROW_BLOCK == 16, "a CTA's rows lie in one block of needed rows");

// grid (n2 / (2 NP), lines), thread = (t, pair) with t fastest.
template <int LOGM, bool HERM>
__global__ void __launch_bounds__(PhiPairCfg<LOGM>::THREADS, PhiPairCfg<LOGM>::MINB)
    k_phi_pair(PhiPairArgs a, const PairC *__restrict__ in, const float2 *__restrict__ tw,
               const float2 *__restrict__ stw, const int2 *__restrict__ rowrange,
               float *__restrict__ grid) {
    dfs_grid_wait();
    constexpr int E = DFS_FFT_E, M = 1 << LOGM, T = M / E, NP = PhiPairCfg<LOGM>::NP;
    const int f = a.line0 + blockIdx.y;
    const int2 rr = rowrange[f / a.F];
    // whole CTA (within one row block): no stencil touches these rows
    if (((2 * NP * (int)blockIdx.x - rr.x) & (a.n2 - 1)) >= rr.y) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int t = threadIdx.x % T;
    const int c = threadIdx.x / T;                 // row pair
    PairC *sm = reinterpret_cast<PairC *>(smem_raw) + (size_t)c * M;
    const int pr = blockIdx.x * NP + c;
    const PairC *src = in + ((size_t)f * (a.n2 >> 1) + pr) * a.tpitch;
    float2 *dst0 = reinterpret_cast<float2 *>(grid + ((size_t)f * a.n2 + 2 * pr) * a.n1);
    float2 *dst1 = dst0 + M;
    const int half = a.N1 / 2;                     // at most M / 2
    // H_j, 0 <= j <= N1/2: real-field rows hold it, general rows hold T_m (m =
    // -N1/2 .. N1/2 - 1) and H_j = (T_j + conj T_{-j}) / 2
    auto hval = [&](int j) -> PairC {
        if constexpr (HERM) {
            return src[j];
        } else {
            const PairC n = src[half - j];
            const PairC q = j < half ? src[half + j] : PairC{0ull, 0ull};
            const f32x2 h = pk(0.5f, 0.5f);
            return PairC{pmul(padd(q.x, n.x), h), pmul(psub(q.y, n.y), h)};
        }
    };
    auto lower = [&](PairC h, float2 w) -> PairC {        // (1 + i w) h
        const PairC d = cmul(h, w);
        return PairC{psub(h.x, d.y), padd(h.y, d.x)};
    };
    auto upper = [&](PairC h, float2 w) -> PairC {        // (1 - i w) conj h
        // d = w conj(h) up to signs: the sum's parts are h.x + d_y and -(h.y + d_x)
        const f32x2 mx = pk(-w.x, -w.x), wy = pk(w.y, w.y), my = pk(-w.y, -w.y);
        return PairC{padd(h.x, pfma(h.x, wy, pmul(h.y, mx))),
                     psub(pfma(h.x, mx, pmul(h.y, my)), h.y)};
    };
    PairC v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int k = t + e * T;
        const int j = e < E / 2 ? k : M - k;
        v[e] = j <= half ? hval(j) : PairC{0ull, 0ull};
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const float2 w = ldt(&tw[t + e * T]);
        if (e < E / 2) {
            v[e] = lower(v[e], w);
        } else {
            const PairC h = v[e];
            v[e] = upper(h, w);
            if (e == E / 2 && t == 0 && half == M / 2) v[e] = v[e] + lower(h, w);
        }
    }
    auto st = [&](int j, PairC z) {
        const float2 re = unpk(z.x), im = unpk(z.y);
        dst0[j] = make_float2(re.x, im.x);
        dst1[j] = make_float2(re.y, im.y);
    };
    auto none = [] {};
    pair_fft<LOGM, (T >= 32)>(stw, sm, t, c + 1, v, st, none);
}

template <int LOGM, bool HERM>
cudaError_t run(dfsnufft_plan p, const PhiPairArgs &a, int lines) {
    typedef PhiPairCfg<LOGM> Cfg;
    const size_t smem = sizeof(PairC) * (size_t)Cfg::NP * (1 << LOGM);
    auto kern = k_phi_pair<LOGM, HERM>;
    cudaError_t e = allow_smem(kern, smem);
    if (e) return e;
    return dfs_launch_dependent(kern, dim3(a.n2 / (2 * Cfg::NP), lines), dim3(Cfg::THREADS), smem,
                                p->stream, a, (const PairC *)p->d_T, (const float2 *)p->d_tw1,
                                (const float2 *)p->d_stw_phi, (const int2 *)p->d_rowrange,
                                (float *)p->d_G);
}

template <int LOGM>
cudaError_t dispatch(dfsnufft_plan p, const PhiPairArgs &a, int lines, int logm) {
    if constexpr (LOGM > DFS_PAIR_MAX_LOG) {
        return cudaErrorNotSupported;
    } else {
        if (logm != LOGM) return dispatch<LOGM + 1>(p, a, lines, logm);
        return p->herm ? run<LOGM, true>(p, a, lines) : run<LOGM, false>(p, a, lines);
    }
}

}  // namespace

// Fine rows of 2^(DFS_PAIR_MIN_LOG + 1) .. 2^(DFS_PAIR_MAX_LOG + 1) cells, plans
// that own their stage-ordered twiddles.
cudaError_t dfs_launch_phi_pair(dfsnufft_plan p) {
    const dfsnufft_params &q = p->prm;
    const int logm = ilog2(q.n1) - 1;
    if (logm < DFS_PAIR_MIN_LOG || !p->d_stw_phi) return cudaErrorNotSupported;
    PhiPairArgs a;
    a.N1 = q.N1;
    a.n1 = q.n1;
    a.n2 = q.n2;
    a.F = p->n_fields;
    a.tpitch = dfs_tpitch(p->herm, q.N1);
    int lines;
    dfs_lines(p, a.line0, lines);
    return dispatch<DFS_PAIR_MIN_LOG>(p, a, lines, logm);
}
