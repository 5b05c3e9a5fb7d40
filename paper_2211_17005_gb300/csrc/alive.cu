// Least squares on the hierarchically simulated sample (Sec. "Learning on
// Hierarchically Simulated Paths"): at pricing date i, one row per (outer path k,
// inner draw l) with the features (X_i^{k,l}, Y_i^k), X the default indicators of
// the counterparties and Y the market state (Sec. 4.1), and the per-draw target
//   xi_i^{k,l} = beta_i^{-1} sum_c (1 - R_c) beta_j MtM_c(t_j)^+ 1{i < j <= n},  j = idx_c^{k,l},
// of eq. (eq:CVA_portfolio). The basis is [1, Y - Y^0, X_1..X_C] (Y^0: path 0's state).
//
// The M N rows are never formed. The rows of path k all carry its state and the
// indicators are 0/1, so the normal equations need only these sums over the N draws
// of each path (an exact regrouping of the sum over (k, l)):
//   d_c  = #{l : X_c = 1}            (column sum of X_c, and its products with Y)
//   P_cd = #{l : X_c = X_d = 1}      (c < d: the X_c X_d products)
//   q_c  = sum_l X_c xi^{k,l}        (right-hand side of X_c)
// and N xi_bar^k for the right-hand side of Y. P_cd and q_c enter only through their
// sums over the paths, d_c also through its products with Y.
//
// alive_stats_kernel turns a tile of paths' default steps into d_c per path, the tile's
// sums of P_cd and the sums of q_c over at most eight paths at every date. gram.cuh accumulates sum_k [1, Y - Y^0]^T
// [1, Y - Y^0, d, xi_bar]. alive_pq_kernel adds the P_cd and q_c.
// alive_solve_kernel adds the Gram chunks, assembles the (1 + F + C)-square system and
// solves it by a Jacobi-scaled factorisation L D L^T in FP64, dropping a column whose
// pivot vanishes (a counterparty with no default by t_i anywhere in the sample).
#include <math.h>

#include "cva_internal.h"
#include "gram.cuh"

namespace cva {

namespace {

constexpr int kMaxUnknowns = 40;    // 1 + F + C
constexpr int kMaxAug = 44;         // [1, Y - Y^0, d, xi_bar]
constexpr int kStatDraws = 64;      // draws staged at a time by the statistics kernel

struct AliveArgs {
    uint32_t M, N;
    int n, F, C, mY, NQ;
    const uint8_t *idx;       // [M][N][C] default steps, n+1 = none
    const float *expo;        // [n+1][C][M] of the portfolio
    const float *disc;        // [n+1][M]
    const float *feat;        // [n+1][F][M]
    float *dstat;             // [n][C][M] d_c per path
    float *psum;              // [n][NP][nblk] P_cd summed over a tile's paths
    float *qsum;              // [n][C][nblk << (lg - lq)] q_c summed over at most eight of them
    uint32_t nblk;            // tiles of the statistics kernel
    int lg, lq;               // log2 of its paths per tile, of the paths q_c is summed over in FP32
    int chunks;
    size_t stride;            // doubles of a Gram partial
    double *part;             // [n-1][chunks][stride]
    double *pq;               // [n-1][NQ]
    double *coef;             // [n-1][1+F+C] centred basis
    double *coef_raw;         // [n-1][1+F+C] raw basis
    int *status;              // [n-1] dropped columns
};

// Shared memory of a tile of 2^lg paths, C counterparties, n dates: the changes of q~_c
// and the defaults of c by (date, c, path), the discount factors by (date, path), the
// pair counts by (date, pair), the staged default steps and the draws listed by a thread.
struct StatShape {
    int threads;              // 2^lg C, rounded up to whole warps: the stride of a date
    size_t dq, dn, beta, pair, steps, list, bytes;   // byte offsets
    int row;                  // bytes between two paths' staged steps
};
__host__ __device__ inline StatShape stat_shape(int lg, int C, int n)
{
    StatShape s;
    s.threads = ((C << lg) + 31) / 32 * 32;
    s.row = kStatDraws * C + 8;   // 8 bytes more: consecutive paths start two banks apart
    s.dq = 0;
    s.beta = s.dq + (size_t)n * s.threads * 4;
    s.pair = s.beta + ((size_t)n * 4 << lg);
    s.steps = s.pair + (size_t)n * (C * (C - 1) / 2) * 4;
    s.steps = (s.steps + 15) / 16 * 16;
    s.dn = s.steps + (((size_t)s.row << lg) + 15) / 16 * 16;
    s.list = s.dn + (size_t)n * s.threads * 2;
    s.bytes = s.list + (size_t)kStatDraws * s.threads;
    return s;
}

// One thread per (counterparty c, path): it walks the path's draws in order and, where c
// defaults at step i <= n, counts it at date i; every other counterparty d of the draw
// that defaults later, at step j, moves q~_c(i) by V_d(j) at date i and by -V_d(j) at date
// j, with q_c = beta^{-1} q~_c. The changes live in a column of its own in shared memory
// ([date][thread]: no bank and no word is shared, no atomics, so the sums have one order).
// The pair counts P_cd are integers and go to the tile's table by atomics. A second walk
// over the dates turns the changes into running sums, stores d_c and reduces q_c over the
// tile's paths.
//
// Bound by latency and by shared memory for the columns (6 bytes per date and thread:
// 12 warps a multiprocessor). 2^17 paths, 64 draws, 100 dates: 1.31 ms; a warp per path that
// re-read a draw's table at each of its events, with a block barrier per date, took 3.13 ms,
// and this walk without the list of events 4.5 ms.
template <int C>
__global__ void __launch_bounds__(256) alive_stats_kernel(AliveArgs a)
{
    constexpr int NP = C * (C - 1) / 2;
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = a.n, lg = a.lg, PT = 1 << lg, tid = threadIdx.x, nthr = blockDim.x;
    const StatShape sh = stat_shape(lg, C, n);
    float *dq = reinterpret_cast<float *>(smem + sh.dq) + tid;
    uint16_t *dn = reinterpret_cast<uint16_t *>(smem + sh.dn) + tid;
    float *binv = reinterpret_cast<float *>(smem + sh.beta);   // [n][PT] beta^{-1}
    int *pair = reinterpret_cast<int *>(smem + sh.pair);       // [n][NP]
    uint8_t *steps = smem + sh.steps;                          // [PT][row]
    uint8_t *list = smem + sh.list + tid;                      // [kStatDraws], this thread's column
    const uint32_t M = a.M, N = a.N, tile0 = blockIdx.x << lg;
    const int p = tid & (PT - 1), c = tid >> lg;
    const uint32_t kl = tile0 + (uint32_t)p;
    const bool live = c < C && kl < M;
    for (uint32_t i = tid; i < (uint32_t)(n * nthr * 4) / 16; i += nthr)   // (whole warps: a multiple of 128 bytes a date)
        reinterpret_cast<uint4 *>(smem + sh.dq)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t i = tid; i < (uint32_t)(n * nthr * 2) / 16; i += nthr)
        reinterpret_cast<uint4 *>(smem + sh.dn)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = tid; i < n * NP; i += nthr) pair[i] = 0;
    for (int i = tid; i < n << lg; i += nthr) {
        const uint32_t k = tile0 + (uint32_t)(i & (PT - 1));
        binv[i] = k < M ? expf(__ldg(a.disc + (size_t)(i >> lg) * M + k)) : 0.f;
    }
    const uint32_t paths = min((uint32_t)PT, M - tile0);
    for (uint32_t l0 = 0; l0 < N; l0 += kStatDraws) {
        const uint32_t nl = min((uint32_t)kStatDraws, N - l0), bytes = nl * C;
        __syncthreads();
        if (((N * C) & 7u) == 0) {   // every path's draws start on 8 bytes
            for (uint32_t i = tid; i < paths * (bytes / 8); i += nthr) {
                const uint32_t q = i / (bytes / 8), o = 8 * (i % (bytes / 8));
                *reinterpret_cast<uint2 *>(steps + q * sh.row + o) =
                    __ldg(reinterpret_cast<const uint2 *>(a.idx + ((size_t)(tile0 + q) * N + l0) * C + o));
            }
        } else {
            for (uint32_t i = tid; i < paths * bytes; i += nthr)
                steps[(i / bytes) * sh.row + i % bytes] = __ldg(a.idx + ((size_t)(tile0 + i / bytes) * N + l0) * C + i % bytes);
        }
        __syncthreads();
        if (!live) continue;
        // this thread's draws with a default of c, listed; then their losses, the gathers of a
        // draw's later defaults all in flight
        const uint8_t *row = steps + p * sh.row;
        int found = 0;
#pragma unroll 4
        for (uint32_t l = 0; l < nl; ++l) {
            const int ic = row[l * C + c];
            if (ic <= n) {
                list[found * nthr] = (uint8_t)l;
                ++found;
            }
        }
        for (int t = 0; t < found; ++t) {
            const uint8_t *js = row + list[t * nthr] * C;
            const int ic = js[c];
            float v[C], later = 0.f;
            int jd[C];
            if constexpr (C == 8) {   // the draw's steps in one load
                const uint2 w = *reinterpret_cast<const uint2 *>(js);
#pragma unroll
                for (int d = 0; d < 8; ++d) jd[d] = ((d < 4 ? w.x : w.y) >> (8 * (d & 3))) & 255u;
            } else {
#pragma unroll
                for (int d = 0; d < C; ++d) jd[d] = js[d];
            }
#pragma unroll
            for (int d = 0; d < C; ++d) {
                v[d] = jd[d] > ic && jd[d] <= n ? __ldg(a.expo + ((size_t)jd[d] * C + d) * M + kl) : 0.f;
            }
#pragma unroll
            for (int d = 0; d < C; ++d) {
                const int j = max(ic, jd[d]);
                if (d > c && j < n) atomicAdd(&pair[j * NP + c * (2 * C - c - 1) / 2 + (d - c - 1)], 1);
                later += v[d];
            }
            if (ic < n) {
                dq[ic * nthr] += later;
                dn[ic * nthr] += 1;
            }
#pragma unroll
            for (int d = 0; d < C; ++d)
                if (jd[d] > ic && jd[d] < n) dq[jd[d] * nthr] -= v[d];
        }
    }
    __syncthreads();
    float q = 0.f;
    uint32_t defaults = 0u;
#pragma unroll 4
    for (int i = 1; i < n; ++i) {
        q += dq[i * nthr];
        defaults += dn[i * nthr];
        dq[i * nthr] = live ? q * binv[(i << lg) + p] : 0.f;
        if (live) a.dstat[((size_t)i * C + c) * M + kl] = (float)defaults;
    }
    __syncthreads();
    // q_c over eight of the tile's paths at a time (the sums go on in FP64 from there): a thread
    // per (date, c, eight paths), which starts at a path of its own so that a warp's reads
    // spread over the banks
    const int lr = lg - a.lq, QT = 1 << a.lq;
    for (int t = tid; t < ((n - 1) * C) << lr; t += nthr) {
        const int e = t & ((1 << lr) - 1), i = 1 + (t >> lr) / C, d = (t >> lr) % C;
        const float *src = reinterpret_cast<const float *>(smem + sh.dq) + i * nthr + (d << lg) + (e << a.lq);
        float s = 0.f;
        for (int u = 0; u < QT; ++u) s += src[(u + (tid >> 2)) & (QT - 1)];
        a.qsum[(((size_t)i * C + d) * a.nblk + blockIdx.x << lr) + e] = s;
    }
    for (int t = tid; t < NP; t += nthr) {
        int s = 0;
        for (int i = 1; i < n; ++i) {
            s += pair[i * NP + t];
            a.psum[((size_t)i * NP + t) * a.nblk + blockIdx.x] = (float)s;
        }
    }
}

// P_cd and q_c of a date over all tiles: blockIdx = (statistic, date - 1). The pair counts
// are added exactly as integers, q_c in FP64, in a fixed order.
__global__ void __launch_bounds__(256) alive_pq_kernel(AliveArgs a)
{
    __shared__ double sh[256];
    const int q = blockIdx.x, i = blockIdx.y + 1, tid = threadIdx.x, NP = a.NQ - a.C;
    const int lr = a.lg - a.lq;
    const float *src = q < NP ? a.psum + ((size_t)i * NP + q) * a.nblk
                              : a.qsum + (((size_t)i * a.C + (q - NP)) * a.nblk << lr);
    double s = 0.0;
    if (q < NP) {
        long long t = 0;
#pragma unroll 8
        for (uint32_t b = tid; b < a.nblk; b += 256) t += (long long)__ldg(src + b);
        s = (double)t;
    } else {
#pragma unroll 8
        for (uint32_t b = tid; b < a.nblk << lr; b += 256) s += (double)__ldg(src + b);
    }
    sh[tid] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (tid < o) sh[tid] += sh[tid + o];
        __syncthreads();
    }
    if (tid == 0) a.pq[(size_t)blockIdx.y * a.NQ + q] = sh[0];
}

__global__ void __launch_bounds__(256) alive_solve_kernel(AliveArgs a)
{
    constexpr int LD = 41;
    __shared__ double A[41 * LD], w[40], sc[40];   // m <= 40 unknowns, one right-hand side
    __shared__ int drop[40];
    const int g = blockIdx.x, tid = threadIdx.x, mY = a.mY, C = a.C, m = mY + C, cols = m + 1, NP = a.NQ - C;
    const double Nd = (double)a.N, *pq = a.pq + (size_t)g * a.NQ;
    // row i of [1, Y - Y^0] against column j of [1, Y - Y^0, d, xi_bar]
    for (int i = tid >> 4; i < mY; i += 16)
        for (int j = i + (tid & 15); j < cols; j += 16) {
            const double *p = a.part + (size_t)g * a.chunks * a.stride + tri_index(cols, i, j);
            double s = 0.0;
#pragma unroll 8
            for (int c = 0; c < a.chunks; ++c) s += p[(size_t)c * a.stride];
            A[j * LD + i] = j < mY || j == m ? Nd * s : s;   // (the right-hand side is row m)
            if (i == 0 && j >= mY && j < m) A[j * LD + j] = s;   // X_c^2 = X_c
        }
    for (int c = tid; c < C; c += 256) {
        for (int d = c + 1; d < C; ++d) A[(mY + d) * LD + mY + c] = pq[c * (2 * C - c - 1) / 2 + (d - c - 1)];
        A[m * LD + mY + c] = pq[NP + c];
    }
    __syncthreads();
    const int dropped = solve_normal<LD>(A, m, 1, w, sc, drop);
    if (tid >= 32) return;
    double *co = a.coef + (size_t)g * m, *cr = a.coef_raw + (size_t)g * m;
    const float *feat = a.feat + (size_t)(g + 1) * a.F * a.M;
    double s = 0.0;
    for (int r = tid; r < m; r += 32) {
        co[r] = w[r];
        if (r > 0) cr[r] = w[r];
        if (r >= 1 && r <= a.F) s = fma(w[r], (double)feat[(size_t)(r - 1) * a.M], s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tid == 0) {
        cr[0] = w[0] - s;
        a.status[g] = dropped;
    }
}

constexpr int kStatMaxSmem = 110 * 1024;   // two blocks a multiprocessor

// paths per tile: 32 up to four counterparties, else 16 (128 threads), fewer where the
// dates' columns would not fit shared memory twice over
int stat_lg(int C, int n)
{
    int lg = C <= 4 ? 5 : 4;
    while (lg > 2 && stat_shape(lg, C, n).bytes > kStatMaxSmem) --lg;
    return lg;
}

template <int C>
cva_status launch_stats(const AliveArgs &a, bool capturing, cudaStream_t st)
{
    const StatShape sh = stat_shape(a.lg, C, a.n);
    if (!capturing)   // (the most any date count takes, so that no call lowers another's limit)
        CVA_CUDA_TRY(cudaFuncSetAttribute(alive_stats_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          kStatMaxSmem));
    alive_stats_kernel<C><<<a.nblk, sh.threads, sh.bytes, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    return CVA_OK;
}

}  // namespace

cva_status alive_regress(Sim &s, int pf, float *pred_dev, double *coef_host, int *dropped_host, cudaStream_t st)
{
    if (pf < 0 || pf >= s.NPF) return fail(CVA_EINVAL, "regress_alive: portfolio index out of range");
    if (s.n < 2) return fail(CVA_EINVAL, "regress_alive: need at least two pricing steps");
    if (!s.d_idx) return fail(CVA_EINVAL, "regress_alive: the simulation keeps no default steps (CVA_KEEP_DEFAULTS)");
    if (s.C < 1 || s.C > 8) return fail(CVA_ENOTSUP, "regress_alive: at most 8 counterparties");
    if (s.M > 0x7fffffffull) return fail(CVA_EINVAL, "regress_alive: M too large");
    const int C = s.C, NQ = C * (C - 1) / 2 + C, mY = s.F + 1, m = mY + C;
    if (m > kMaxUnknowns) return fail(CVA_ENOTSUP, "regress_alive: 1 + F + C must be <= 40");
    // the number of draws this call takes: N (5C + 6) within 160 KB (the kernel stages 64 at a time
    // and could take more: up to 65535, which its 16-bit counters hold)
    const size_t draw_floats = ((size_t)s.N * (C + 1) * 4 + 15) / 16 * 16;
    if ((draw_floats + (size_t)s.N * (C + 2) + 15) / 16 * 16 + 64 * (size_t)(2 * C + C * (C - 1) / 2) > (size_t)160 * 1024)
        return fail(CVA_ENOTSUP, "regress_alive: N * C too large for the per-path draw tables");
    const int cols = m + 1;   // Gram columns: [1, Y - Y^0] (mY), d (C), xi_bar
    if (cols > kMaxAug) return fail(CVA_ENOTSUP, "regress_alive: too many Gram columns");
    const size_t M = s.M;
    const int lg = stat_lg(C, s.n);
    const uint32_t nblk = (uint32_t)((M + (1u << lg) - 1) >> lg);
    const int groups = s.n - 1;
    uint64_t rows_per_chunk, chunks;
    gram_chunks(M, groups, s.tune_lsq_chunks > 0 ? s.tune_lsq_chunks : 2432, 1024, &rows_per_chunk, &chunks);
    const size_t stride = (size_t)tri_index(cols, mY - 1, cols - 1) + 1;
    const size_t need = (size_t)groups * (chunks * stride + NQ + 2 * (size_t)m + 1);
    const int lq = lg < 3 ? lg : 3;
    const size_t need_stats = (size_t)s.n * C * M + (size_t)s.n * ((size_t)(NQ - C) * nblk + ((size_t)C * nblk << (lg - lq)));
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CVA_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
    if (s.alive_cap < need || s.alive_stats_cap < need_stats) {
        if (cap != cudaStreamCaptureStatusNone)
            return fail(CVA_EINVAL, "regress_alive: call once before capturing so that the scratch exists");
        CVA_CUDA_TRY(cudaStreamSynchronize(st));
        if (s.alive_cap < need) {
            cudaFree(s.d_alive);
            s.d_alive = nullptr;
            s.alive_cap = 0;
            if (cudaMalloc(&s.d_alive, need * sizeof(double)) != cudaSuccess)
                return fail(CVA_ENOMEM, "regress_alive: scratch allocation failed");
            s.alive_cap = need;
        }
        if (s.alive_stats_cap < need_stats) {
            cudaFree(s.d_alive_stats);
            s.d_alive_stats = nullptr;
            s.alive_stats_cap = 0;
            if (cudaMalloc(&s.d_alive_stats, need_stats * sizeof(float)) != cudaSuccess)
                return fail(CVA_ENOMEM, "regress_alive: statistics allocation failed");
            s.alive_stats_cap = need_stats;
        }
    }
    AliveArgs a;
    a.M = (uint32_t)M;
    a.N = s.N;
    a.n = s.n;
    a.F = s.F;
    a.C = C;
    a.mY = mY;
    a.NQ = NQ;
    a.idx = s.d_idx;
    a.expo = s.d_expo + (size_t)pf * (s.n + 1) * C * M;
    a.disc = s.d_disc;
    a.feat = s.d_features;
    a.dstat = s.d_alive_stats;
    a.psum = s.d_alive_stats + (size_t)s.n * C * M;
    a.qsum = a.psum + (size_t)s.n * (NQ - C) * nblk;
    a.nblk = nblk;
    a.lg = lg;
    a.lq = lq;
    a.chunks = (int)chunks;
    a.stride = stride;
    a.part = s.d_alive;
    a.pq = a.part + (size_t)groups * chunks * stride;
    a.coef = a.pq + (size_t)groups * NQ;
    a.coef_raw = a.coef + (size_t)groups * m;
    a.status = reinterpret_cast<int *>(a.coef_raw + (size_t)groups * m);
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    static constexpr cva_status (*by_c[8])(const AliveArgs &, bool, cudaStream_t) = {
        launch_stats<1>, launch_stats<2>, launch_stats<3>, launch_stats<4>,
        launch_stats<5>, launch_stats<6>, launch_stats<7>, launch_stats<8>};
    cva_status r = by_c[C - 1](a, capturing, st);
    if (r != CVA_OK) return r;
    GramArgs q;
    q.feat0 = s.d_features + (size_t)s.F * M;   // date 1
    q.feat_stride = (size_t)s.F * M;
    q.centre = nullptr;
    q.F = s.F;
    q.ext[0] = a.dstat + (size_t)C * M;
    q.ext_gstride[0] = (size_t)C * M;
    q.ext_cstride[0] = M;
    q.n_ext[0] = C;
    q.ext[1] = s.d_targets + ((size_t)pf * s.n + 1) * M;
    q.ext_gstride[1] = M;
    q.ext_cstride[1] = 0;
    q.n_ext[1] = 1;
    q.M = (uint32_t)M;
    q.rows_per_chunk = (uint32_t)rows_per_chunk;
    q.chunks = (int)chunks;
    q.cols = cols;
    q.rows = mY;
    q.part = a.part;
    q.stride = stride;
    r = launch_gram(q, groups, st);
    if (r != CVA_OK) return r;
    alive_pq_kernel<<<dim3((unsigned)NQ, (unsigned)groups), 256, 0, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    alive_solve_kernel<<<groups, 256, 0, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    if (pred_dev) {   // the fit at X = 0 (every counterparty alive)
        r = lsq_predict_groups(s.d_features + (size_t)s.F * M, (size_t)s.F * M, s.F, M, groups, a.coef, (size_t)m,
                               pred_dev + M, M, st);
        if (r != CVA_OK) return r;
    }
    if (coef_host || dropped_host) {
        std::vector<double> cr((size_t)groups * m);
        std::vector<int> status(groups);
        CVA_CUDA_TRY(cudaMemcpyAsync(cr.data(), a.coef_raw, sizeof(double) * cr.size(), cudaMemcpyDeviceToHost, st));
        CVA_CUDA_TRY(cudaMemcpyAsync(status.data(), a.status, sizeof(int) * groups, cudaMemcpyDeviceToHost, st));
        CVA_CUDA_TRY(cudaStreamSynchronize(st));
        if (coef_host)
            for (int g = 0; g < groups; ++g)
                for (int c = 0; c < m; ++c) coef_host[(size_t)(g + 1) * m + c] = cr[(size_t)g * m + c];
        if (dropped_host) {
            dropped_host[0] = 0;
            for (int g = 0; g < groups; ++g) dropped_host[g + 1] = status[g];
        }
    }
    return CVA_OK;
}

}  // namespace cva
