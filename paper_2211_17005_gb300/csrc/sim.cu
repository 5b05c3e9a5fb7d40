// Inner-default kernel of the hierarchical CVA simulation, and the dispatch
// of the outer-path kernel instantiations (outer_*.cu).
//
// Inner defaults (Sec. 3.2 / eq. (e:tau)): N default clocks per counterparty and
// path; tau^{k,l} falls in (t_{j-1}, t_j] when the uniform w (epsilon = -log(1 - w))
// satisfies T(j-1) < w <= T(j), T = 1 - e^{-Lambda}: the default step is the lower
// bound of w in the monotone thresholds. The averaged target of eq.
// (eq:CVA_portfolio) of every portfolio follows from the integer counts of defaults
// per (counterparty, step),
//   xi_bar_i = beta_i^{-1} (1/N) sum_{j>i} sum_c V_c(j) count_c(j),
// so the targets do not depend on the order of the draws.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "cva_internal.h"
#include "rng.cuh"

namespace cva {

namespace {

struct InnerArgs {
    uint32_t M, k0, seed_lo, seed_hi, N;
    uint32_t branch;                  // third counter word of the clocks (twin copy id, 0 otherwise)
    int n, NPF;
    int lg;                           // log2 of the paths per block
    int rows;                         // rows of the threshold area: n max(C, NPF)
    int packed;                       // 1: two 16-bit counters a word (N <= 65535)
    const float *__restrict__ thr;    // [n+1][C][M]
    const float *__restrict__ expo;   // [NPF][n+1][C][M]
    const float *__restrict__ disc;   // [n+1][M]
    float *targets;                   // [NPF][n][M]
    uint8_t *idx;                     // [M][N][C] or null
};

// First j in [1, n] with T(j) >= w for nondecreasing thresholds T, else n + 1
// (n <= 255): the lower bound by the fixed power-of-two steps 128, 64, ..., 1 (every
// lane of a warp runs the same unrolled steps, so that the searches of several
// counterparties interleave; a step past n reads nothing).
template <class Thr>
__device__ __forceinline__ int lower_bound_pow2(Thr T, int n, float w)
{
    int pos = 0;   // T(1..pos) < w
#pragma unroll
    for (int step = 128; step > 0; step >>= 1) {
        const int q = pos + step;
        if (q <= n && T(q) < w) pos = q;
    }
    return pos + 1;
}

// Draws whose defaults a thread's queue holds: two, and more where the counterparties are so few
// that the searches would run one or two at a time. One counterparty, 65536 paths, 512 draws, 50
// dates, clocks to targets: 250 us with two draws, 168 with eight (178 for the two kernels of a
// warp per path before).
__host__ __device__ constexpr int queue_draws(int C) { return C == 1 ? 8 : C == 2 ? 4 : 2; }
// A thread's draws between two stores of the staged steps: 32 bytes or so of them, so that few
// counterparties do not mean many barriers (a multiple of 4: runs of whole 16 bytes).
__host__ __device__ constexpr int idx_draws(int C) { return C >= 8 ? 4 : 32 / C / 4 * 4; }
// Shared memory of the staged steps: [2^lg] rows of idx_draws (nthr >> lg) draws, 16 bytes more
// each so that rows start in different banks; after thresholds, counters and queues.
__host__ __device__ constexpr int idx_stage_pitch(int lg, int C, int nthr) { return idx_draws(C) * (nthr >> lg) * C + 16; }
__host__ __device__ constexpr size_t idx_stage_offset(int rows, int cnt_words, int lg, int C, int nthr)
{
    return (4 * (((size_t)rows << lg) + (size_t)cnt_words + (size_t)queue_draws(C) * C * nthr) + 15) / 16 * 16;
}

// Clocks, counts and targets of a tile of PT = 2^lg outer paths in one block.
//
// A lane owns one path of the tile (lane mod PT) throughout, so shared memory is laid
// out with the path innermost: the thresholds, staged by cp.async, as [n C][PT]; the
// counts as [n C][PT], two 16-bit counters a word when every count fits (N <= 65535).
// Lanes of different paths then never share a bank, and whole rows move between shared
// and global memory without a transpose.
//
// What bounds it: instruction issue while the clocks are drawn, HBM while thresholds and
// exposures are read. Most clocks outlive the horizon (w > T(n)): a lane compares each
// with its path's T(n), as an integer bound on the draw's 23 bits, and only queues the
// ones that default (a few draws' at most, in its own column of the queue), so that the
// lower bounds run over queues a few entries long. The blocks of a multiprocessor are in
// different phases, which overlaps the two bounds.
// Paper shape, 2^17 paths, 64 draws, 100 dates: 0.40 ms; as two kernels with the counts in
// global memory between them 0.55 + 0.17 ms. Six portfolios, 2^18 paths, 256 draws: 3.0 ms
// against 2.2 + 1.45 ms.
// IDX: the default steps are kept too (cva_sim's validation output). They wait in shared memory,
// some of a thread's draws at a time (idx_draws), and leave as whole runs of a path's row.
// Stored from where they are found, a byte of another path's row per lane, they took longer
// than the clocks: four counterparties, 65536 paths, 512 draws, 50 dates, the whole simulation
// 1259 us, so 535 us (486 without the steps); the paper's shape with 256 draws and 20 dates
// 1295 and 580 us.
template <int C, bool IDX>
__global__ void __launch_bounds__(512) inner_kernel(InnerArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int n = a.n, lg = a.lg, PT = 1 << lg, NPF = a.NPF;
    const int ps = a.packed;                                                     // 1: two counters a word
    const int tid = threadIdx.x, nthr = blockDim.x;
    float *T = reinterpret_cast<float *>(smem);                                  // [rows][PT]: thresholds, then sums
    uint32_t *cnt = reinterpret_cast<uint32_t *>(T + ((size_t)a.rows << lg));    // counts
    const int cnt_words = ((n * C + ps) >> ps) << lg;
    constexpr int D = queue_draws(C);
    uint32_t *queue = cnt + cnt_words + tid;                                     // [D C][nthr], this thread's column
    uint8_t *stage = reinterpret_cast<uint8_t *>(smem + idx_stage_offset(a.rows, cnt_words, lg, C, nthr));   // IDX: [PT][pitch]
    const int pitch = idx_stage_pitch(lg, C, nthr);
    const uint32_t M = a.M, tile0 = blockIdx.x << lg;
    const int p = tid & (PT - 1);
    const bool live = tile0 + (uint32_t)p < M;

    {   // row r = (j - 1) C + c of the thresholds, PT consecutive paths
        const float *src = a.thr + (size_t)C * M + tile0;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(T);
        if (lg >= 2 && (M & 3u) == 0) {   // every piece of four paths is aligned and whole
            const int lq = lg - 2;
            for (int i = tid; i < (n * C) << lq; i += nthr) {
                const int q = i & ((1 << lq) - 1), r = i >> lq;
                if (tile0 + 4u * (uint32_t)q < M)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * (uint32_t)i),
                                 "l"(src + (size_t)r * M + 4 * q)
                                 : "memory");
            }
        } else {
            for (int i = tid; i < (n * C) << lg; i += nthr)
                if (live)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * (uint32_t)i),
                                 "l"(src + (size_t)(i >> lg) * M + p)
                                 : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int i = tid; i < cnt_words; i += nthr) cnt[i] = 0u;
    const uint32_t none = (uint32_t)(n + 1) * 0x01010101u;   // no default, four times
    if (IDX)
        for (int i = tid; i < (pitch << lg) / 16; i += nthr)
            reinterpret_cast<uint4 *>(stage)[i] = make_uint4(none, none, none, none);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // The draws of three counterparties or more whose steps are not kept, then every other case. One
    // loop for both, over spans of draws and with a counter in place of `even`, costs the first
    // 2 to 5% (eight counterparties, 2^17 paths, 1024 draws: 2.15 and 2.24 ms).
    if constexpr (!IDX && D == 2) {
        if (live) {
            const uint32_t k = a.k0 + tile0 + (uint32_t)p, stride = (uint32_t)(nthr >> lg);
            // w = (m + 1/2) 2^-23 <= T(n)  <=>  m < bound = floor(2^23 T(n) - 1/2) + 1, every
            // operation exact (T <= 1; a NaN takes every clock, as the comparison of w would)
            uint32_t bound[C];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const float t = T[(((n - 1) * C + c) << lg) + p] * 8388608.f;
                bound[c] = t >= 0.5f ? (uint32_t)floorf(fminf(t, 8388608.f) - 0.5f) + 1u : t < 0.5f ? 0u : 8388608u;
            }
            const uint32_t Tp = (uint32_t)__cvta_generic_to_shared(T + p);
            auto lds = [](uint32_t addr) {
                float v;
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
                return v;
            };
            int queued = 0;
            bool even = false;
            for (uint32_t l = (uint32_t)(tid >> lg); l < a.N; l += stride) {
#pragma unroll
                for (int cb = 0; cb < (C + 3) / 4; ++cb) {
                    const uint4 x = philox4x32_10(make_uint4(k, l, a.branch, (kStreamInner << 24) | (uint32_t)cb),
                                                  a.seed_lo, a.seed_hi);
                    const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int c = 4 * cb + i;
                        if (c < C) {
                            const bool hit = (xs[i] >> 9) < bound[c];
                            if (hit) queue[queued] = (xs[i] & ~0x1ffu) | (uint32_t)c;
                            queued += hit ? nthr : 0;
                        }
                    }
                }
                even = !even;
                if (even && l + stride < a.N) continue;   // the queue holds two draws' defaults
                even = false;
                // four entries at a time: their searches interleave
                for (int t = 0; t < queued; t += 4 * nthr) {
                    float w[4];
                    uint32_t at[4];      // shared address of the search's lower end
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t x = t + u * nthr < queued ? queue[t + u * nthr] : 0u;
                        w[u] = uniform23(x);
                        at[u] = Tp + ((x & 0x1ffu) << (lg + 2));
                    }
                    // first j with T(j) >= w among 1..n (T(n) >= w): the halving of a range of
                    // n depends on n only, so its steps are the same for every lane
                    for (int len = n; len > 1;) {
                        const int half = len >> 1;
                        const uint32_t span = (uint32_t)(half * C) << (lg + 2), probe = span - ((uint32_t)C << (lg + 2));
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (lds(at[u] + probe) < w[u]) at[u] += span;
                        len -= half;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (t + u * nthr < queued) {
                            const uint32_t ci = (at[u] - Tp) >> (lg + 2);   // step (at 0) x C + counterparty
                            atomicAdd(&cnt[((ci >> ps) << lg) + p], 1u << (16 * (ci & (uint32_t)ps)));
                        }
                }
                queued = 0;
            }
        }
    } else {
        const uint32_t k = a.k0 + tile0 + (uint32_t)p, stride = (uint32_t)(nthr >> lg);
        // w = (m + 1/2) 2^-23 <= T(n)  <=>  m < bound = floor(2^23 T(n) - 1/2) + 1, every
        // operation exact (T <= 1; a NaN takes every clock, as the comparison of w would)
        uint32_t bound[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const float t = T[(((n - 1) * C + c) << lg) + p] * 8388608.f;
            bound[c] = t >= 0.5f ? (uint32_t)floorf(fminf(t, 8388608.f) - 0.5f) + 1u : t < 0.5f ? 0u : 8388608u;
        }
        const uint32_t Tp = (uint32_t)__cvta_generic_to_shared(T + p);
        auto lds = [](uint32_t addr) {
            float v;
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
            return v;
        };
        // this thread's draws of [l0, l1)
        auto draw = [&](uint32_t l0, uint32_t l1) {
            int queued = 0;
            uint32_t held = 0;   // draws in the queue
            for (uint32_t l = l0 + (uint32_t)(tid >> lg); l < l1; l += stride) {
                // an entry: the draw's 23 bits, (IDX) which of the queue's draws, the counterparty
                const uint32_t tag = IDX ? held << 4 : 0u;
#pragma unroll
                for (int cb = 0; cb < (C + 3) / 4; ++cb) {
                    const uint4 x = philox4x32_10(make_uint4(k, l, a.branch, (kStreamInner << 24) | (uint32_t)cb),
                                                  a.seed_lo, a.seed_hi);
                    const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int c = 4 * cb + i;
                        if (c < C) {
                            const bool hit = (xs[i] >> 9) < bound[c];
                            if (hit) queue[queued] = (xs[i] & ~0x1ffu) | tag | (uint32_t)c;
                            queued += hit ? nthr : 0;
                        }
                    }
                }
                if (++held < (uint32_t)D && l + stride < l1) continue;
                // the first draw's place in the staged row
                const uint32_t row = IDX ? (uint32_t)(p * pitch) + (l - l0 - (held - 1) * stride) * C : 0u;
                held = 0;
                // four entries at a time: their searches interleave
                for (int t = 0; t < queued; t += 4 * nthr) {
                    float w[4];
                    uint32_t at[4], to[4];      // shared address of the search's lower end; place of the draw's steps
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t x = t + u * nthr < queued ? queue[t + u * nthr] : 0u;
                        w[u] = uniform23(x);
                        at[u] = Tp + ((x & (IDX ? 0xfu : 0x1ffu)) << (lg + 2));
                        if (IDX) to[u] = row + (x >> 4 & (uint32_t)(D - 1)) * stride * C;
                    }
                    // first j with T(j) >= w among 1..n (T(n) >= w): the halving of a range of
                    // n depends on n only, so its steps are the same for every lane
                    for (int len = n; len > 1;) {
                        const int half = len >> 1;
                        const uint32_t span = (uint32_t)(half * C) << (lg + 2), probe = span - ((uint32_t)C << (lg + 2));
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (lds(at[u] + probe) < w[u]) at[u] += span;
                        len -= half;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (t + u * nthr < queued) {
                            const uint32_t ci = (at[u] - Tp) >> (lg + 2);   // step (at 0) x C + counterparty
                            atomicAdd(&cnt[((ci >> ps) << lg) + p], 1u << (16 * (ci & (uint32_t)ps)));
                            if (IDX) stage[to[u] + ci % C] = (uint8_t)(ci / C + 1);
                        }
                }
                queued = 0;
            }
        };
        if constexpr (!IDX) {
            if (live) draw(0u, a.N);
        } else {
            const uint32_t span = idx_draws(C) * stride, paths = min((uint32_t)PT, M - tile0);
            // the staged rows' first `bytes` bytes to the paths' rows from draw l0, W at a time; what
            // was read is set back to "no default"
            auto store = [&](auto word, uint32_t l0, uint32_t bytes) {
                using W = decltype(word);
                constexpr uint32_t B = sizeof(W);
                const uint32_t per = bytes / B;
                for (uint32_t i = tid; i < paths * per; i += nthr) {
                    const uint32_t q = i / per, o = i % per * B;
                    W *from = reinterpret_cast<W *>(stage + q * pitch + o);
                    *reinterpret_cast<W *>(a.idx + ((size_t)(tile0 + q) * a.N + l0) * C + o) = *from;
                    if constexpr (B == 16) *from = make_uint4(none, none, none, none);
                    else *from = (W)none;
                }
            };
            for (uint32_t l0 = 0; l0 < a.N; l0 += span) {
                const uint32_t nl = min(span, a.N - l0), bytes = nl * C;
                if (live) draw(l0, l0 + nl);
                __syncthreads();
                // (span C is a multiple of 16, so only the rows' own length decides)
                if ((a.N * (uint32_t)C) % 16 == 0) store(uint4{}, l0, bytes);
                else if ((a.N * (uint32_t)C) % 4 == 0) store(uint32_t{}, l0, bytes);
                else store(uint8_t{}, l0, bytes);
                __syncthreads();
                if (span > a.N - l0) break;   // (l0 + span may not fit 32 bits)
            }
        }
    }
    __syncthreads();

    // sum_c V_c(j) count_c(j) of every (portfolio, date), over the thresholds' area
    const uint32_t kl = tile0 + (uint32_t)p;
    const uint32_t mask = ps ? 0xffffu : 0xffffffffu;
    if (live)
        for (int j = 1 + (tid >> lg); j <= n; j += nthr >> lg) {
            float cn[C];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int ci = (j - 1) * C + c;
                cn[c] = (float)((cnt[((ci >> ps) << lg) + p] >> (16 * (ci & ps))) & mask);
            }
            const float *ex = a.expo + (size_t)j * C * M + kl;
            for (int pf = 0; pf < NPF; ++pf) {
                float h = 0.f;
#pragma unroll
                for (int c = 0; c < C; ++c) h = fmaf(__ldg(ex + (size_t)c * M), cn[c], h);
                T[((pf * n + j - 1) << lg) + p] = h;
                ex += (size_t)(n + 1) * C * M;
            }
        }
    __syncthreads();
    // running sums over the dates from the last, a thread per (portfolio, path); eight
    // loads ahead of the adds
    for (int t = tid; t < NPF << lg; t += nthr) {
        float *h = T + (((t >> lg) * n) << lg) + (t & (PT - 1));
        float S = 0.f;
        int j = n - 1;
        for (; j >= 7; j -= 8) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = h[(j - i) << lg];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                S += v[i];
                h[(j - i) << lg] = S;
            }
        }
        for (; j >= 0; --j) {
            S += h[j << lg];
            h[j << lg] = S;
        }
    }
    __syncthreads();
    if (live) {
        const float invN = 1.0f / (float)a.N;
        for (int j = tid >> lg; j < n; j += nthr >> lg) {
            const float bi = expf(__ldg(a.disc + (size_t)j * M + kl)) * invN;   // beta_j^{-1} / N
            for (int pf = 0; pf < NPF; ++pf)
                a.targets[((size_t)pf * n + j) * M + kl] = T[((pf * n + j) << lg) + p] * bi;
        }
    }
}

// Sampling statistics of Prop. 1 (Sec. ss:choice1). For the pointwise loss
// g_l = (xi^{k,l}_i - phi_i(Y^k))^2 of the first two inner draws l = 0, 1 of path
// k (single-draw targets of eq. (eq:CVA_portfolio): the same clocks as the
// simulation's draws 0 and 1), block sums over paths, per date i in [1, n-1], of
// (g0 + g1)/2, (g0^2 + g1^2)/2 and g0 g1, in FP64: part[block][n][3] (date 0 zero).
struct OversimArgs {
    uint32_t M, k0, seed_lo, seed_hi;
    int n, pf;
    const float *__restrict__ thr;    // [n+1][C][M]
    const float *__restrict__ expo;   // [NPF][n+1][C][M]
    const float *__restrict__ disc;   // [n+1][M]
    const float *__restrict__ pred;   // [n][M]
    double *part;
};

template <int C>
__global__ void __launch_bounds__(256) oversim_kernel(OversimArgs a)
{
    __shared__ double red[8][3];
    const uint32_t M = a.M, kl = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = kl < M;
    const int n = a.n, np1 = n + 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int idx[2][C];
    float vs[2][C];
#pragma unroll
    for (int l = 0; l < 2; ++l)
#pragma unroll
        for (int c = 0; c < C; ++c) {
            idx[l][c] = n + 1;
            vs[l][c] = 0.f;
        }
    if (live) {
        const uint32_t k = a.k0 + kl;
#pragma unroll
        for (int l = 0; l < 2; ++l)
#pragma unroll
            for (int cb = 0; cb < (C + 3) / 4; ++cb) {
                const uint4 x = philox4x32_10(make_uint4(k, (uint32_t)l, 0u, (kStreamInner << 24) | (uint32_t)cb),
                                              a.seed_lo, a.seed_hi);
                const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = 4 * cb + t;
                    if (c < C) {
                        const float w = uniform23(xs[t]);
                        const float *Tc = a.thr + (size_t)c * M + kl;   // T(j) at Tc[j C M]
                        const int lo = lower_bound_pow2([Tc, M](int j) { return __ldg(Tc + (size_t)j * C * M); },
                                                        n, w);
                        idx[l][c] = lo;
                        if (lo <= n) vs[l][c] = __ldg(a.expo + ((size_t)(a.pf * np1 + lo) * C + c) * M + kl);
                    }
                }
            }
    }
    for (int i = 1; i < n; ++i) {
        double s[3] = {0.0, 0.0, 0.0};
        if (live) {
            float h0 = 0.f, h1 = 0.f;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (idx[0][c] > i) h0 += vs[0][c];
                if (idx[1][c] > i) h1 += vs[1][c];
            }
            const float e = expf(__ldg(a.disc + (size_t)i * M + kl));
            const double f = (double)__ldg(a.pred + (size_t)i * M + kl);
            const double g0 = ((double)(h0 * e) - f) * ((double)(h0 * e) - f),
                         g1 = ((double)(h1 * e) - f) * ((double)(h1 * e) - f);
            s[0] = 0.5 * (g0 + g1);
            s[1] = 0.5 * (g0 * g0 + g1 * g1);
            s[2] = g0 * g1;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
            if (lane == 0) red[warp][q] = s[q];
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w][threadIdx.x];
            a.part[((size_t)blockIdx.x * n + i) * 3 + threadIdx.x] = t;
        }
        __syncthreads();
    }
    if (threadIdx.x < 3) a.part[(size_t)blockIdx.x * n * 3 + threadIdx.x] = 0.0;
}

}  // namespace

cva_status launch_oversim(const Sim &s, int pf, const float *pred, uint64_t seed, double *part, unsigned blocks,
                          cudaStream_t st)
{
    OversimArgs a;
    a.M = (uint32_t)s.M;
    a.k0 = 0;
    a.seed_lo = (uint32_t)seed;
    a.seed_hi = (uint32_t)(seed >> 32);
    a.n = s.n;
    a.pf = pf;
    a.thr = s.d_thr;
    a.expo = s.d_expo;
    a.disc = s.d_disc;
    a.pred = pred;
    a.part = part;
    static constexpr void (*by_c[kMaxC])(OversimArgs) = {
        oversim_kernel<1>,  oversim_kernel<2>,  oversim_kernel<3>,  oversim_kernel<4>,
        oversim_kernel<5>,  oversim_kernel<6>,  oversim_kernel<7>,  oversim_kernel<8>,
        oversim_kernel<9>,  oversim_kernel<10>, oversim_kernel<11>, oversim_kernel<12>,
        oversim_kernel<13>, oversim_kernel<14>, oversim_kernel<15>, oversim_kernel<16>};
    if (s.C < 1 || s.C > kMaxC) return fail(CVA_ENOTSUP, "oversimulation statistics: 1 <= C <= 16");
    by_c[s.C - 1]<<<blocks, 256, 0, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    return CVA_OK;
}

// Registry of the compiled outer-kernel shapes (one translation unit each).
int outer_insts_small(const OuterInst **out);
int outer_insts_paper(const OuterInst **out);
int outer_insts_batched(const OuterInst **out);
int outer_insts_generic(const OuterInst **out);

static const OuterInst *find_outer(int E, int C, int CS, int G, int NPF)
{
    const OuterInst *best = nullptr;
    int (*tables[])(const OuterInst **) = {outer_insts_small, outer_insts_paper, outer_insts_batched};
    for (auto tab : tables) {
        const OuterInst *p = nullptr;
        const int cnt = tab(&p);
        for (int i = 0; i < cnt; ++i) {
            const OuterInst &o = p[i];
            if (o.E == E && o.C == C && o.CS == CS && o.NPF == NPF && o.G >= G && (!best || o.G < best->G))
                best = &o;
        }
    }
    return best;
}

bool outer_supported(int E, int C, int CS, int G, int NPF, int *Ginst)
{
    const OuterInst *o = find_outer(E, C, CS, G, NPF);
    if (o && Ginst) *Ginst = o->G;
    return o != nullptr;
}

void forget_const_owner(const Sim *s)
{
    int (*tables[])(const OuterInst **) = {outer_insts_small, outer_insts_paper, outer_insts_batched,
                                           outer_insts_generic};
    for (auto tab : tables) {
        const OuterInst *p = nullptr;
        const int cnt = tab(&p);
        for (int i = 0; i < cnt; ++i) p[i].forget(s);
    }
}

static const OuterInst *generic_outer()
{
    const OuterInst *p = nullptr;
    outer_insts_generic(&p);
    return p;
}

cva_status launch_adjoint(Sim &s, AdjBuffers &b, uint64_t seed, uint64_t k0, uint32_t M, cudaStream_t st)
{
    if (s.generic) return generic_outer()->adjoint(s, b, seed, k0, M, st);
    const OuterInst *o = find_outer(s.E, s.C, s.CS, s.G, s.NPF);
    if (!o || o->G != s.Ginst || !o->adjoint) return fail(CVA_ENOTSUP, "no adjoint kernel for this model shape");
    return o->adjoint(s, b, seed, k0, M, st);
}

cva_status launch_outer(Sim &s, uint64_t seed, uint64_t k0, cudaStream_t st)
{
    if (s.generic) return generic_outer()->launch(s, seed, k0, st);
    const OuterInst *o = find_outer(s.E, s.C, s.CS, s.G, s.NPF);
    if (!o || o->G != s.Ginst) return fail(CVA_ENOTSUP, "no outer kernel for this model shape");
    return o->launch(s, seed, k0, st);
}

// Shared memory of a tile: thresholds (later the portfolio sums), counters, queues and (keep)
// the staged steps.
static size_t inner_smem(int lg, int threads, int C, int n, int NPF, bool packed, bool keep)
{
    const int rows = n * std::max(C, NPF), words = (packed ? (n * C + 1) / 2 : n * C) << lg;
    return idx_stage_offset(rows, words, lg, C, threads) + (keep ? (size_t)idx_stage_pitch(lg, C, threads) << lg : 0);
}

template <int C>
static cudaError_t launch_inner_t(InnerArgs &args, int tune, int sms, int dev, cudaStream_t st)
{
    const bool packed = args.N <= 65535u, keep = args.idx != nullptr;
    const auto kern = keep ? inner_kernel<C, true> : inner_kernel<C, false>;
    static std::atomic<bool> attr[2][64];
    if (!attr[keep][dev].load(std::memory_order_acquire)) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 216 * 1024);
        if (e != cudaSuccess) return e;
        attr[keep][dev].store(true, std::memory_order_release);
    }
    // 32 paths a tile (whole 128-byte rows, no bank shared) unless two such blocks do not
    // fit a multiprocessor or the tiles do not fill the chip twice; a tile of fewer than
    // 8 paths only where 8 do not fit at all. A tile shape set by the caller (2, 4, 8:
    // tiles of 8, 16, 32 paths) replaces the first rule as far as it fits.
    auto threads_of = [&](int lg) {
        // enough for the draws of a tile, or for its thresholds and exposures where the draws are
        // few (8 counterparties, 100 dates, 2^17 paths, 8 draws: 0.63 ms with the 128 threads of
        // the draws alone, 0.33 with 512)
        const uint64_t want = std::max<uint64_t>(args.N, (uint64_t)args.n * C / 8) << lg;
        const int t = want >= 512 ? 512 : want >= 256 ? 256 : 128;
        // half the queues where that lets a second block in
        const auto two = [&](int threads) { return inner_smem(lg, threads, C, args.n, args.NPF, packed, keep) <= 108 * 1024; };
        return t == 512 && !two(512) && two(256) ? 256 : t;
    };
    auto smem_of = [&](int lg) { return inner_smem(lg, threads_of(lg), C, args.n, args.NPF, packed, keep); };
    int lg = tune == 2 ? 3 : tune == 4 ? 4 : 5;
    while (tune == 0 && lg > 3 && (smem_of(lg) > 108 * 1024 || (args.M >> lg) < 2u * (unsigned)sms)) --lg;
    while (lg > 0 && smem_of(lg) > 216 * 1024) --lg;
    args.lg = lg;
    args.packed = packed;
    args.rows = args.n * std::max(C, args.NPF);
    kern<<<(unsigned)((args.M + (1ull << lg) - 1) >> lg), threads_of(lg), smem_of(lg), st>>>(args);
    return cudaGetLastError();
}

cva_status launch_inner(Sim &s, uint64_t seed, uint64_t k0, cudaStream_t st)
{
    InnerArgs args;
    args.M = (uint32_t)s.M;
    args.k0 = (uint32_t)k0;
    args.seed_lo = (uint32_t)seed;
    args.seed_hi = (uint32_t)(seed >> 32);
    args.N = s.N;
    args.branch = s.branch;
    args.n = s.n;
    args.NPF = s.NPF;
    args.thr = s.d_thr;
    args.expo = s.d_expo;
    args.disc = s.d_disc;
    args.targets = s.d_targets;
    args.idx = s.d_idx;
    static constexpr cudaError_t (*by_c[kMaxC])(InnerArgs &, int, int, int, cudaStream_t) = {
        launch_inner_t<1>,  launch_inner_t<2>,  launch_inner_t<3>,  launch_inner_t<4>,
        launch_inner_t<5>,  launch_inner_t<6>,  launch_inner_t<7>,  launch_inner_t<8>,
        launch_inner_t<9>,  launch_inner_t<10>, launch_inner_t<11>, launch_inner_t<12>,
        launch_inner_t<13>, launch_inner_t<14>, launch_inner_t<15>, launch_inner_t<16>};
    if (s.C < 1 || s.C > kMaxC) return fail(CVA_ENOTSUP, "inner kernel: 1 <= C <= 16");
    int dev = 0, sms = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    CVA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const cudaError_t e = by_c[s.C - 1](args, s.tune_inner_P, sms, dev, st);
    if (e != cudaSuccess) return cuda_fail(e, "inner kernel launch");
    return CVA_OK;
}

}  // namespace cva
