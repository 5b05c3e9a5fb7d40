// Sums of products of data columns over rows, and the solution of the normal equations
// they form: shared by the least squares on the state (lsq.cu) and on (default
// indicators, state) (alive.cu).
#pragma once
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "cva_internal.h"
#include "sum_pair.cuh"

namespace cva {
namespace {

constexpr int kGramMaxCols = 48;   // augmented columns, six blocks of 8

// One group (pricing date) per blockIdx.y: column 0 is the constant 1, columns 1..F
// the state centred on c0 (the quadratic basis: factor 0 and its square), then the
// columns of two further arrays (not centred).
struct GramArgs {
    const float *feat0;            // [groups][F][M]
    size_t feat_stride;
    const float *centre;           // [F] centring state; null: path 0 of the group
    int F;
    const float *ext[2];           // further columns: ext[x] + group ext_gstride[x] + column ext_cstride[x]
    size_t ext_gstride[2], ext_cstride[2];
    int n_ext[2];
    uint32_t M, rows_per_chunk;    // a multiple of 64
    int chunks;
    int cols, rows;                // augmented columns; rows of the result that are wanted
    int nblk, RG;                  // 8 x 8 blocks, row groups
    double *part;                  // [groups][chunks][stride]: the upper triangle, row-major
    size_t stride;
};

// entry (i, j), i <= j, of the packed upper triangle of a matrix with `cols` columns
__host__ __device__ constexpr int tri_index(int cols, int i, int j) { return i * cols - i * (i - 1) / 2 + (j - i); }

// Tiles of TR rows arrive by cp.async in three buffers, columns contiguous; a thread
// centres the pieces it copied itself, so a tile costs one barrier. A warp owns an 8 x 8
// block of the upper triangle (and a row group where there are few blocks) and its lanes
// take two consecutive rows each: 16 eight-byte operand loads, free of bank conflicts,
// for 128 FMAs. FP32 runs of at most 256 rows a lane are reduced over the lanes by a
// butterfly (five more roundings) and added in FP64.
//
// Bound by the FMA issue (528 multiply-adds a row at 29 columns; 435 are needed) and the
// read of the data, about equal. The tiles were transposed to rows before, with eight-way
// bank conflicts in the copies and in the centring pass: 29 columns of 2^17 rows at 99
// dates took 1276 us, now 599 us (2.5 TB/s of the data, 59% of the issue slots: the warps of a
// block wait for each other's tiles).
template <int TR, int MAXT, int MINB, bool VEC>
__global__ void __launch_bounds__(MAXT, MINB) gram_kernel(GramArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float *tiles = reinterpret_cast<float *>(smem);     // [3][NC][TR]
    __shared__ const float *src[kGramMaxCols];          // copied columns: source,
    __shared__ float c0[kGramMaxCols];                  // and centre; column 1 + i of the tile
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int g = blockIdx.y, NC = (a.cols + 7) / 8 * 8;
    const uint32_t r_begin = blockIdx.x * a.rows_per_chunk, r_end = min(a.M, r_begin + a.rows_per_chunk);
    const int nstate = a.F, ncopy = nstate + a.n_ext[0] + a.n_ext[1];
    for (int i = tid; i < ncopy; i += nthr) {
        if (i < nstate) {
            const float *f = a.feat0 + (size_t)g * a.feat_stride + (size_t)i * a.M;
            src[i] = f;
            c0[i] = a.centre ? __ldg(a.centre + i) : __ldg(f);
        } else {
            const int x = i - nstate < a.n_ext[0] ? 0 : 1, c = i - nstate - (x ? a.n_ext[0] : 0);
            src[i] = a.ext[x] + (size_t)g * a.ext_gstride[x] + (size_t)c * a.ext_cstride[x];
        }
    }
    for (int i = tid; i < 3 * (NC - a.cols) * TR; i += nthr) {   // padding columns stay zero
        const int s = i / ((NC - a.cols) * TR), o = i % ((NC - a.cols) * TR);
        tiles[(s * NC + a.cols) * TR + o] = 0.f;
    }
    for (int i = tid; i < 3 * TR; i += nthr) tiles[(i / TR) * NC * TR + i % TR] = 1.f;
    __syncthreads();
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(tiles);
    const int ntiles = r_begin < r_end ? (int)((r_end - r_begin + TR - 1) / TR) : 0;
    const int nwarps = nthr >> 5;
    constexpr int PW = VEC ? 4 : 1, PL = TR / PW / 32;   // rows of a piece, pieces of a lane
    // a warp copies whole columns, its lanes the pieces lane, lane + 32, ...
    auto issue = [&](int t) {
        if (t < ntiles) {
            const uint32_t r0 = r_begin + (uint32_t)t * TR + (uint32_t)(lane * PW);
            const uint32_t to0 = sbase + (uint32_t)((t % 3) * NC * TR + lane * PW) * 4u;
            for (int cc = warp; cc < ncopy; cc += nwarps) {
                const float *from = src[cc] + r0;
                const uint32_t to = to0 + (uint32_t)((1 + cc) * TR) * 4u;
#pragma unroll
                for (int i = 0; i < PL; ++i) {
                    const bool ok = r0 + (uint32_t)(i * 32 * PW) < r_end;
                    if (VEC)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to + i * 512u),
                                     "l"(ok ? from + i * 128 : src[cc]), "r"(ok ? 16 : 0)
                                     : "memory");
                    else
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to + i * 128u),
                                     "l"(ok ? from + i * 32 : src[cc]), "r"(ok ? 4 : 0)
                                     : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // this lane's pieces of the state columns of tile t: centred, zero past the end (as the
    // constant column is in the last tile)
    auto finish = [&](int t) {
        const uint32_t r0 = r_begin + (uint32_t)t * TR + (uint32_t)(lane * PW);
        float *tile = tiles + (size_t)(t % 3) * NC * TR + lane * PW;
        for (int cc = warp; cc < nstate; cc += nwarps) {
            const float c1 = c0[cc];
            float *v = tile + (1 + cc) * TR;
#pragma unroll
            for (int i = 0; i < PL; ++i) {
                const float c = r0 + (uint32_t)(i * 32 * PW) < r_end ? c1 : 0.f;
                if (VEC) {
                    float4 x = *reinterpret_cast<float4 *>(v + i * 128);
                    x = make_float4(x.x - c, x.y - c, x.z - c, x.w - c);
                    *reinterpret_cast<float4 *>(v + i * 128) = x;
                } else {
                    v[i * 32] -= c;
                }
            }
        }
        if (t + 1 == ntiles)
            for (int r = tid; r < TR; r += nthr)
                tiles[(size_t)(t % 3) * NC * TR + r] = r_begin + (uint32_t)(t * TR + r) < r_end ? 1.f : 0.f;
    };
    // this warp's block (bi <= bj) and row group
    int bi = 0, bj = 0;
    const int rg = warp / a.nblk;
    {
        int b = warp % a.nblk;
        while (b >= NC / 8 - bi) {
            b -= NC / 8 - bi;
            ++bi;
        }
        bj = bi + b;
    }
    float acc[8][8];
    double dacc[2] = {0.0, 0.0};
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
    // the 64 sums over the lanes, lane l left with entries 2 l and 2 l + 1
    auto flush = [&]() {
        float *f = &acc[0][0];
#pragma unroll
        for (int o = 16, h = 32; o > 0; o >>= 1, h >>= 1)
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const bool up = lane & o;
                const float keep = up ? f[i + h] : f[i], send = up ? f[i] : f[i + h];
                f[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        dacc[0] += (double)f[0];
        dacc[1] += (double)f[1];
#pragma unroll
        for (int u = 0; u < 64; ++u) f[u] = 0.f;
    };
    issue(0);
    issue(1);
    int run = 0;
    for (int t = 0; t < ntiles; ++t) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        finish(t);
        __syncthreads();   // tile t is complete; every warp is done with tile t - 1
        issue(t + 2);
        const uint32_t left = r_end - (r_begin + (uint32_t)t * TR);
        const float *tile = tiles + (size_t)(t % 3) * NC * TR + 2 * lane;
        const float *px = tile + 8 * bi * TR, *py = tile + 8 * bj * TR;
#pragma unroll 1
        for (int it = rg; it < TR / 64 && (uint32_t)(it * 64) < left; it += a.RG) {
            float2 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = *reinterpret_cast<const float2 *>(px + u * TR + it * 64);
            if (bi == bj) {   // a diagonal block: its upper triangle, of its own columns
#pragma unroll
                for (int v = 0; v < 8; ++v) {
#pragma unroll
                    for (int u = 0; u <= v; ++u) acc[u][v] = fmaf(x[u].x, x[v].x, acc[u][v]);
#pragma unroll
                    for (int u = 0; u <= v; ++u) acc[u][v] = fmaf(x[u].y, x[v].y, acc[u][v]);
                }
            } else {
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    const float2 y = *reinterpret_cast<const float2 *>(py + v * TR + it * 64);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][v] = fmaf(x[u].x, y.x, acc[u][v]);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][v] = fmaf(x[u].y, y.y, acc[u][v]);
                }
            }
            if (++run == 128) {
                run = 0;
                flush();
            }
        }
    }
    flush();
    __syncthreads();
    double *red = reinterpret_cast<double *>(smem);   // [RG][nblk][64]
    red[warp * 64 + 2 * lane] = dacc[0];
    red[warp * 64 + 2 * lane + 1] = dacc[1];
    __syncthreads();
    if (rg == 0) {
        double *out = a.part + ((size_t)g * a.chunks + blockIdx.x) * a.stride;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = 2 * lane + h, i = 8 * bi + (e >> 3), j = 8 * bj + (e & 7);
            double s = red[warp * 64 + e];
            for (int q = 1; q < a.RG; ++q) s += red[(warp + q * a.nblk) * 64 + e];
            if (i <= j && j < a.cols && i < a.rows) out[tri_index(a.cols, i, j)] = s;
        }
    }
}

// The sums of the quadratic basis [1, d, d^2], d = y - y^0 of factor 0, and NT targets.
// The normal equations of d and d^2 are sensitive to rounding, so every FP32 product is
// added to a SumPair.
// Bound by latency: 49 dates of 2^14 paths take 16 us (49 us as a case of the general kernel,
// with its FP64 runs).
template <int NT>
__global__ void __launch_bounds__(256) poly_gram_kernel(GramArgs a)
{
    constexpr int NS = 4 + 4 * NT;   // d, d^2, d^3, d^4; per target xi, xi d, xi d^2, xi^2
    __shared__ double red[8][NS];
    const int g = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    const uint32_t r_begin = blockIdx.x * a.rows_per_chunk, r_end = min(a.M, r_begin + a.rows_per_chunk);
    const float *f = a.feat0 + (size_t)g * a.feat_stride, *x = a.ext[0] + (size_t)g * a.ext_gstride[0];
    const float c = a.centre ? __ldg(a.centre) : __ldg(f);
    SumPair s[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) s[i].hi = s[i].lo = 0.f;
#pragma unroll 4
    for (uint32_t r = r_begin + tid; r < r_end; r += 256) {
        const float d = __ldg(f + r) - c, d2 = __fmul_rn(d, d);
        s[0].add(d);
        s[1].add(d2);
        s[2].add(__fmul_rn(d, d2));
        s[3].add(__fmul_rn(d2, d2));
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const float v = __ldg(x + (size_t)t * a.ext_cstride[0] + r);
            s[4 + 4 * t].add(v);
            s[5 + 4 * t].add(__fmul_rn(v, d));
            s[6 + 4 * t].add(__fmul_rn(v, d2));
            s[7 + 4 * t].add(__fmul_rn(v, v));
        }
    }
#pragma unroll
    for (int i = 0; i < NS; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h = __shfl_xor_sync(0xffffffffu, s[i].hi, o), l = __shfl_xor_sync(0xffffffffu, s[i].lo, o);
            s[i].add(h, l);
        }
        if (lane == 0) red[tid >> 5][i] = (double)s[i].hi + (double)s[i].lo;
    }
    __syncthreads();
    if (tid >= NS) return;
    double v = red[0][tid];
#pragma unroll
    for (int w = 1; w < 8; ++w) v += red[w][tid];
    double *out = a.part + ((size_t)g * a.chunks + blockIdx.x) * a.stride;
    const int cols = a.cols;
    if (tid == 0) out[tri_index(cols, 0, 0)] = r_begin < r_end ? (double)(r_end - r_begin) : 0.0;
    if (tid < 4) {
        if (tid == 0) out[tri_index(cols, 0, 1)] = v;
        if (tid == 1) out[tri_index(cols, 0, 2)] = out[tri_index(cols, 1, 1)] = v;
        if (tid == 2) out[tri_index(cols, 1, 2)] = v;
        if (tid == 3) out[tri_index(cols, 2, 2)] = v;
    } else {
        const int t = (tid - 4) / 4, i = (tid - 4) % 4;
        if (i < 3) out[tri_index(cols, i, 3 + t)] = v;
        else if (a.rows > 3) out[tri_index(cols, 3, 3)] = v;   // one target: its own square too
    }
}

// Rows per chunk and chunks of a group: about `target` blocks over all groups, at least
// `min_rows` rows a block.
inline void gram_chunks(uint64_t M, int groups, int target, uint64_t min_rows, uint64_t *rows, uint64_t *chunks)
{
    uint64_t c = ((uint64_t)target + groups - 1) / groups;
    const uint64_t most = (M + min_rows - 1) / min_rows;
    if (c > most) c = most;
    if (c < 1) c = 1;
    *rows = ((M + c - 1) / c + 63) / 64 * 64;
    *chunks = (M + *rows - 1) / *rows;
}

// Lets every form take the shared memory of its widest call, once per device: a limit that
// followed the call's own width would be lowered under another thread's launch, or under a
// captured call of a wider system. (Inside a capture it is left as it is.)
inline cva_status gram_allow_smem(cudaStream_t st)
{
    static std::atomic<uint64_t> ready{0};
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
    if (ready.load(std::memory_order_acquire) & bit) return CVA_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CVA_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
    if (cap != cudaStreamCaptureStatusNone) return CVA_OK;
    auto allow = [](auto kern, size_t bytes) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    constexpr size_t f = sizeof(float);
    CVA_CUDA_TRY(allow(gram_kernel<512, 320, 2, true>, 3 * 16 * 512 * f));
    CVA_CUDA_TRY(allow(gram_kernel<512, 320, 2, false>, 3 * 16 * 512 * f));
    CVA_CUDA_TRY(allow(gram_kernel<256, 320, 2, true>, 3 * 32 * 256 * f));
    CVA_CUDA_TRY(allow(gram_kernel<256, 320, 2, false>, 3 * 32 * 256 * f));
    CVA_CUDA_TRY(allow(gram_kernel<256, 640, 1, true>, 3 * kGramMaxCols * 256 * f));
    CVA_CUDA_TRY(allow(gram_kernel<256, 640, 1, false>, 3 * kGramMaxCols * 256 * f));
    ready.fetch_or(bit, std::memory_order_release);
    return CVA_OK;
}

// Launch: the widest form whose registers and tiles fit, two blocks per multiprocessor
// up to 32 columns (10 warps), one beyond; 512-row tiles where three column blocks or
// fewer leave shared memory for them. 16-byte copies where every column allows them.
inline cva_status launch_gram(GramArgs &a, int groups, cudaStream_t st)
{
    const int nb = (a.cols + 7) / 8, nr = (a.rows + 7) / 8;
    a.nblk = 0;
    for (int i = 0; i < nr; ++i) a.nblk += nb - i;
    if (a.cols > kGramMaxCols || a.nblk > 20) return fail(CVA_ENOTSUP, "regress: too many columns");
    a.RG = a.nblk == 1 ? 8 : a.nblk <= 3 ? 3 : 1;
    bool vec = a.M % 4 == 0 && a.feat_stride % 4 == 0 && (reinterpret_cast<uintptr_t>(a.feat0) & 15u) == 0;
    for (int x = 0; x < 2; ++x)
        if (a.n_ext[x] > 0)
            vec = vec && a.ext_gstride[x] % 4 == 0 && (a.ext_cstride[x] % 4 == 0 || a.n_ext[x] == 1) &&
                  (reinterpret_cast<uintptr_t>(a.ext[x]) & 15u) == 0;
    const dim3 grid((unsigned)a.chunks, (unsigned)groups);
    const int threads = 32 * a.nblk * a.RG;
    const int TR = nb <= 2 ? 512 : 256;
    const size_t smem = std::max((size_t)3 * nb * 8 * TR * sizeof(float), (size_t)a.nblk * a.RG * 64 * sizeof(double));
    const cva_status allowed = gram_allow_smem(st);
    if (allowed != CVA_OK) return allowed;
    auto go = [&](auto kern) -> cva_status {
        kern<<<grid, threads, smem, st>>>(a);
        CVA_CUDA_TRY(cudaGetLastError());
        return CVA_OK;
    };
    if (nb <= 2) return vec ? go(gram_kernel<512, 320, 2, true>) : go(gram_kernel<512, 320, 2, false>);
    if (threads <= 320) return vec ? go(gram_kernel<256, 320, 2, true>) : go(gram_kernel<256, 320, 2, false>);
    return vec ? go(gram_kernel<256, 640, 1, true>) : go(gram_kernel<256, 640, 1, false>);
}

// sums over the chunks of a group, 8 chunk lanes per entry, in a fixed order: used where
// few groups would leave one multiprocessor each to add hundreds of chunks
__global__ void __launch_bounds__(256) gram_reduce_kernel(const double *part, int chunks, size_t stride, double *out)
{
    __shared__ double sh[8][32];
    const int e = blockIdx.x * 32 + (threadIdx.x & 31), cl = threadIdx.x >> 5;
    double s = 0.0;
    if ((size_t)e < stride)
        for (int c = cl; c < chunks; c += 8) s += part[((size_t)blockIdx.y * chunks + c) * stride + e];
    sh[cl][threadIdx.x & 31] = s;
    __syncthreads();
    if (cl == 0 && (size_t)e < stride) {
#pragma unroll
        for (int q = 1; q < 8; ++q) s += sh[q][threadIdx.x & 31];
        out[(size_t)blockIdx.y * stride + e] = s;
    }
}

// Normal equations A w = b of m unknowns and nt right-hand sides by the whole block
// (256 threads): A [m + nt][LD] in shared memory, lower triangle, the right-hand sides as
// rows m.. ; Jacobi scaling, then the right-looking factorisation L D L^T with the right-hand
// sides carried along as further rows, then one warp per right-hand side for the back
// substitution. A column whose pivot vanishes is dropped: its part of L is zero and its
// coefficient 0. w [nt][m] receives the solutions in the unscaled basis; returns the number
// of dropped columns.
//
// Bound by the FP64 pipe (two lanes a clock and multiprocessor) and by the chain of pivots,
// so one warp alone computes a pivot's reciprocal, by Newton steps on an FP32 estimate
// (scaled pivots lie in (1e-12, 1]), and nothing is divided or rooted in FP64. 28 unknowns:
// 118 us with FP64 square roots and divisions and one thread's triangular solves, now 39 us
// (99 systems in one launch).
template <int LD>
__device__ int solve_normal(double *A, int m, int nt, double *w, double *sc, int *drop)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ double s_inv[2];
    for (int r = tid; r < m; r += blockDim.x) {
        const double d = A[r * LD + r];
        drop[r] = !(d > 0.0);
        sc[r] = drop[r] ? 0.0 : rsqrt(d);
    }
    __syncthreads();
    for (int r = tid >> 4; r < m + nt; r += blockDim.x >> 4)
        for (int c = tid & 15; c < m && c <= r; c += 16) A[r * LD + c] *= sc[c] * (r < m ? sc[r] : 1.0);
    __syncthreads();
    for (int j = 0; j < m; ++j) {
        if (warp == 0) {
            const double s = A[j * LD + j];
            const bool out = drop[j] || !(s > 1e-12);
            double y = out ? 0.0 : (double)__frcp_rn((float)s);
            y = fma(y, fma(-s, y, 1.0), y);
            y = fma(y, fma(-s, y, 1.0), y);
            __syncwarp();
            if (lane == 0) {
                s_inv[j & 1] = y;
                drop[j] = out;
                A[j * LD + j] = y;   // the reciprocal of the pivot
            }
        }
        __syncthreads();
        const double inv = s_inv[j & 1];
        for (int r = j + 1 + (tid >> 4); r < m + nt; r += blockDim.x >> 4) {
            const double lr = -A[r * LD + j] * inv;
            for (int c = j + 1 + (tid & 15); c < m && c <= r; c += 16) A[r * LD + c] = fma(lr, A[c * LD + j], A[r * LD + c]);
        }
        __syncthreads();
    }
    // L^T x = D^{-1} c, w = S x: lanes over the unknowns, two each
    for (int t = warp; t < nt; t += blockDim.x >> 5) {
        double y0 = lane < m ? A[(m + t) * LD + lane] : 0.0, y1 = lane + 32 < m ? A[(m + t) * LD + lane + 32] : 0.0;
        for (int i = m - 1; i >= 0; --i) {
            const double z = __shfl_sync(0xffffffffu, i >= 32 ? y1 : y0, i & 31) * A[i * LD + i];   // 0 if dropped
            if (lane < i) y0 = fma(-A[i * LD + lane], z, y0);
            if (i > 32 && lane + 32 < i) y1 = fma(-A[i * LD + lane + 32], z, y1);
            if (lane == (i & 31)) w[t * m + i] = z * sc[i];
        }
    }
    int dropped = 0;
    __syncthreads();
    for (int r = 0; r < m; ++r) dropped += drop[r];
    return dropped;
}

}  // namespace
}  // namespace cva
