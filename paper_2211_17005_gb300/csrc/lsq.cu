// Grouped least-squares regression of eq. (e:forw), one group per pricing date:
//   w = argmin_w sum_k (xi_k - w^T phi(Y_k))^2.
// The augmented Gram matrix [phi, xi]^T [phi, xi] of the basis centred on path 0's
// state is accumulated by gram.cuh (FP32 products in short FP32 runs, then FP64 in a
// fixed order; every byte of the features and targets is read once) and solved by a
// Jacobi-scaled factorisation L D L^T in FP64. A second pass over the features makes
// the predictions, from the last group back, whose features are still in L2.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <math.h>

#include <mutex>
#include <vector>

#include "cva_internal.h"
#include "gram.cuh"

namespace cva {

namespace {

struct LsqArgs {
    const float *feat0;
    size_t feat_stride;   // floats between groups' feature blocks ([F][M] each)
    const float *targ0;
    size_t targ_stride;   // floats between groups' targets
    float *pred0;
    size_t pred_stride;
    int F, m, basis, chunks;
    uint32_t M, rows_per_chunk;
    double *part;         // [groups][chunks][stride] (gram.cuh)
    size_t stride;
    double *coef;         // [groups][nt][m] centred basis
    double *coef_raw;     // [groups][nt][m] raw basis
    int *status;          // [groups] dropped columns
    int nt = 1;                 // target columns sharing one normal matrix
    size_t targ_tstride = 0;    // floats between a group's targets
    size_t pred_tstride = 0;    // floats between a group's predictions
    size_t coef_stride = 0;     // doubles between groups' coefficients (0: nt m)
    const float *centre = nullptr;   // [F] (poly2: [1]) centring state; null: path 0 of the group
};

// the centring state of the basis: the given one, else path 0 of the group's features
__device__ __forceinline__ float centre_of(const LsqArgs &a, const float *feat, int f)
{
    return a.centre ? __ldg(a.centre + f) : __ldg(feat + (size_t)f * a.M);
}

// The normal equations of a group: the chunks added in order, solved for every target
// column, the coefficients in the centred and in the raw basis.
__global__ void __launch_bounds__(256) lsq_solve(LsqArgs a)
{
    constexpr int LD = 41;
    __shared__ double A[40 * LD], w[400], sc[40];   // m + nt <= 40
    __shared__ int drop[40];
    const int g = blockIdx.x, tid = threadIdx.x, m = a.m, mA = m + a.nt;
    for (int i = tid >> 4; i < m; i += 16)
        for (int j = i + (tid & 15); j < mA; j += 16) {
            const double *p = a.part + (size_t)g * a.chunks * a.stride + tri_index(mA, i, j);
            double s = 0.0;
#pragma unroll 8
            for (int c = 0; c < a.chunks; ++c) s += p[(size_t)c * a.stride];
            A[j * LD + i] = s;
        }
    __syncthreads();
    const int dropped = solve_normal<LD>(A, m, a.nt, w, sc, drop);
    if (tid == 0) a.status[g] = dropped;
    const float *feat = a.feat0 + (size_t)g * a.feat_stride;
    for (int t = tid >> 5; t < a.nt; t += 8) {   // a warp per target column
        const int lane = tid & 31;
        double *co = a.coef + ((size_t)g * a.nt + t) * m, *cr = a.coef_raw + ((size_t)g * a.nt + t) * m;
        const double *wt = w + t * m;
        for (int i = lane; i < m; i += 32) co[i] = wt[i];
        if (a.basis == CVA_BASIS_POLY2) {
            if (lane == 0) {
                const double c = (double)centre_of(a, feat, 0);
                cr[0] = wt[0] - wt[1] * c + wt[2] * c * c;
                cr[1] = wt[1] - 2.0 * wt[2] * c;
                cr[2] = wt[2];
            }
        } else {
            double s = 0.0;   // sum of the shifts, lanes over the factors
            for (int f = lane; f < a.F; f += 32) {
                cr[1 + f] = wt[1 + f];
                s = fma(wt[1 + f], (double)centre_of(a, feat, f), s);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) cr[0] = wt[0] - s;
        }
    }
}

// Predictions of every target column of group g (blockIdx.y) at one path per
// thread: the features are read once per path for all nt columns, and the block
// converts the group's FP64 coefficients to FP32 once (FP64 conversions run on
// the slow FP64 pipe). The FMA order per column is the basis order. Groups run from the last
// back: the Gram has just read that one, so part of it is still in the L2 cache.
__global__ void __launch_bounds__(256) lsq_predict(LsqArgs a)
{
    __shared__ float cs[40 * 40];   // [nt][m], m + nt <= 40
    __shared__ float f0[40];        // path 0's state: the centring of the basis
    const int g = (int)(gridDim.y - 1 - blockIdx.y), nt = a.nt, m = a.m;   // from the last group back
    const double *co = a.coef + (size_t)g * (a.coef_stride ? a.coef_stride : (size_t)nt * m);
    const float *feat = a.feat0 + (size_t)g * a.feat_stride;
    for (int i = threadIdx.x; i < nt * m; i += blockDim.x) cs[i] = (float)co[i];
    const int nf = a.basis == CVA_BASIS_POLY2 ? 1 : a.F;
    for (int f = threadIdx.x; f < nf; f += blockDim.x) f0[f] = centre_of(a, feat, f);
    __syncthreads();
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.M) return;
    float *out = a.pred0 + (size_t)g * a.pred_stride + k;
    if (a.basis == CVA_BASIS_POLY2) {
        const float d = __ldg(feat + k) - f0[0];
        for (int t = 0; t < nt; ++t)
            out[(size_t)t * a.pred_tstride] = fmaf(cs[t * m + 2], d * d, fmaf(cs[t * m + 1], d, cs[t * m]));
        return;
    }
    for (int t0 = 0; t0 < nt; t0 += 8) {
        const int tn = nt - t0 < 8 ? nt - t0 : 8;
        float acc[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] = u < tn ? cs[(t0 + u) * m] : 0.f;
#pragma unroll 4
        for (int f = 0; f < a.F; ++f) {
            const float x = __ldg(feat + (size_t)f * a.M + k) - f0[f];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (u < tn) acc[u] = fmaf(cs[(t0 + u) * m + 1 + f], x, acc[u]);
        }
        for (int u = 0; u < tn; ++u) out[(size_t)(t0 + u) * a.pred_tstride] = acc[u];
    }
}

// The linear-basis predictions of lsq_predict for 4 consecutive paths per thread:
// 16-byte feature loads and prediction stores, the same FMA order per path (so the
// same bits). Needs M, the strides and the base addresses to be multiples of 4
// floats (checked by lsq_predict_launch). TM: targets a thread carries at a time, 1 or 8
// (one target leaves the registers to loads in flight). Bound by HBM: one target, 27 factors,
// 2^17 paths and 99 dates 294 -> 216 us, 6.8 TB/s.
template <int TM>
__global__ void __launch_bounds__(256) lsq_predict4(LsqArgs a)
{
    __shared__ float cs[40 * 40];   // [nt][m], m + nt <= 40
    __shared__ float f0[40];
    const int g = (int)(gridDim.y - 1 - blockIdx.y), nt = a.nt, m = a.m;   // from the last group back
    const double *co = a.coef + (size_t)g * (a.coef_stride ? a.coef_stride : (size_t)nt * m);
    const float *feat = a.feat0 + (size_t)g * a.feat_stride;
    for (int i = threadIdx.x; i < nt * m; i += blockDim.x) cs[i] = (float)co[i];
    for (int f = threadIdx.x; f < a.F; f += blockDim.x) f0[f] = centre_of(a, feat, f);
    __syncthreads();
    const uint32_t k = 4u * (blockIdx.x * blockDim.x + threadIdx.x);
    if (k >= a.M) return;
    float *out = a.pred0 + (size_t)g * a.pred_stride + k;
    for (int t0 = 0; t0 < nt; t0 += TM) {
        const int tn = nt - t0 < TM ? nt - t0 : TM;
        float4 acc[TM];
#pragma unroll
        for (int u = 0; u < TM; ++u) {
            const float c = u < tn ? cs[(t0 + u) * m] : 0.f;
            acc[u] = make_float4(c, c, c, c);
        }
#pragma unroll (TM == 1 ? 9 : 4)
        for (int f = 0; f < a.F; ++f) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(feat + (size_t)f * a.M + k));
            const float c0 = f0[f];
            const float x0 = v.x - c0, x1 = v.y - c0, x2 = v.z - c0, x3 = v.w - c0;
#pragma unroll
            for (int u = 0; u < TM; ++u)
                if (u < tn) {
                    const float c = cs[(t0 + u) * m + 1 + f];
                    acc[u].x = fmaf(c, x0, acc[u].x);
                    acc[u].y = fmaf(c, x1, acc[u].y);
                    acc[u].z = fmaf(c, x2, acc[u].z);
                    acc[u].w = fmaf(c, x3, acc[u].w);
                }
        }
        for (int u = 0; u < tn; ++u) *reinterpret_cast<float4 *>(out + (size_t)(t0 + u) * a.pred_tstride) = acc[u];
    }
}

// Predictions of every group: 4 paths per thread where the shapes allow 16-byte
// accesses, else one path per thread.
cva_status lsq_predict_launch(const LsqArgs &a, int groups, cudaStream_t st)
{
    const bool wide = a.basis == CVA_BASIS_LINEAR && a.M % 4 == 0 && a.feat_stride % 4 == 0 && a.pred_stride % 4 == 0 &&
                      a.pred_tstride % 4 == 0 && (reinterpret_cast<uintptr_t>(a.feat0) & 15u) == 0 &&
                      (reinterpret_cast<uintptr_t>(a.pred0) & 15u) == 0;
    if (wide)
        (a.nt == 1 ? lsq_predict4<1> : lsq_predict4<8>)<<<dim3((unsigned)((a.M / 4 + 255) / 256), (unsigned)groups), 256, 0, st>>>(a);
    else
        lsq_predict<<<dim3((unsigned)((a.M + 255) / 256), (unsigned)groups), 256, 0, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    return CVA_OK;
}

// Library-owned scratch for the Gram partials and coefficients, per device.
// Reuse is ordered by an event: a call waits for the previous call's kernels.
struct LsqScratch {
    double *buf = nullptr;
    size_t cap = 0;   // doubles
    cudaEvent_t done = nullptr;
};
std::mutex g_lsq_mu;
LsqScratch g_lsq[64];

}  // namespace

// Scratch of the grouped regression: [groups][chunks][stride] Gram partials, their sums
// where the chunks are many ([groups][stride]), 2 [groups][nt][m] coefficients, groups ints.
struct LsqPlan {
    int m, rows;                // unknowns; rows of the Gram matrix (with the target's own for one target)
    size_t stride;              // doubles of a partial
    uint64_t rows_per_chunk, chunks;
    bool reduce;                // add the chunks in a launch of their own
    size_t doubles;
};

static LsqPlan lsq_plan(int F, int basis, int nt, uint64_t M, int groups, int target)
{
    LsqPlan p;
    p.m = basis == CVA_BASIS_POLY2 ? 3 : F + 1;
    p.rows = p.m + (nt == 1);
    p.stride = (size_t)tri_index(p.m + nt, p.rows - 1, p.m + nt - 1) + 1;
    // 1024 rows a block at least, 512 where that would leave multiprocessors without work; the
    // quadratic basis takes a quarter of the blocks, whose reduction otherwise outweighs the
    // few products of their rows (49 dates of 2^14 paths: 17 us with 784 blocks), and fewer the
    // more targets a block reduces (six targets, 119 dates, the whole regression, with the
    // blocks of one target / so: 2^11 paths 59 / 39 us, 2^13 79 / 54, 30001 paths 132 / 106)
    target = target > 0 ? target : 2432;
    uint64_t min_rows = (uint64_t)groups * ((M + 1023) / 1024) < 304 ? 512 : 1024;
    if (basis == CVA_BASIS_POLY2) {
        target = std::max(target / 4 / (1 + nt / 3), 1);
        if (nt >= 3) min_rows = 2048;
    }
    gram_chunks(M, groups, target, min_rows, &p.rows_per_chunk, &p.chunks);
    p.reduce = p.chunks > 48;
    p.doubles = (size_t)groups * (p.chunks + p.reduce) * p.stride + 2 * (size_t)groups * nt * p.m + (size_t)groups;
    return p;
}

// the Gram partials of every group (columns of the basis, then the targets)
static cva_status lsq_gram(const LsqArgs &a, int rows, int groups, cudaStream_t st)
{
    GramArgs q;
    q.feat0 = a.feat0;
    q.feat_stride = a.feat_stride;
    q.centre = a.centre;
    q.F = a.F;
    q.ext[0] = a.targ0;
    q.ext_gstride[0] = a.targ_stride;
    q.ext_cstride[0] = a.targ_tstride;
    q.n_ext[0] = a.nt;
    q.ext[1] = nullptr;
    q.ext_gstride[1] = q.ext_cstride[1] = 0;
    q.n_ext[1] = 0;
    q.M = a.M;
    q.rows_per_chunk = a.rows_per_chunk;
    q.chunks = a.chunks;
    q.cols = a.m + a.nt;
    q.rows = rows;
    q.part = a.part;
    q.stride = a.stride;
    if (a.basis == CVA_BASIS_LINEAR) return launch_gram(q, groups, st);
    const dim3 grid((unsigned)a.chunks, (unsigned)groups);
    switch (a.nt) {
    case 1: poly_gram_kernel<1><<<grid, 256, 0, st>>>(q); break;
    case 2: poly_gram_kernel<2><<<grid, 256, 0, st>>>(q); break;
    case 3: poly_gram_kernel<3><<<grid, 256, 0, st>>>(q); break;
    case 4: poly_gram_kernel<4><<<grid, 256, 0, st>>>(q); break;
    case 5: poly_gram_kernel<5><<<grid, 256, 0, st>>>(q); break;
    case 6: poly_gram_kernel<6><<<grid, 256, 0, st>>>(q); break;
    default: return fail(CVA_ENOTSUP, "regress: at most 6 targets on the quadratic basis");
    }
    CVA_CUDA_TRY(cudaGetLastError());
    return CVA_OK;
}

cva_status lsq_launch(const LsqJob &j, double *scratch, size_t scratch_cap, double *coef_host, cudaStream_t st)
{
    if (!j.feat0 || !j.targ0 || j.M == 0 || j.groups <= 0 || j.nt < 1)
        return fail(CVA_EINVAL, "regress: bad arguments");
    if (j.M > 0x7fffffffull) return fail(CVA_EINVAL, "regress: M too large");
    if (j.basis != CVA_BASIS_LINEAR && j.basis != CVA_BASIS_POLY2) return fail(CVA_EINVAL, "regress: unknown basis");
    const int m = (j.basis == CVA_BASIS_POLY2) ? 3 : j.F + 1;
    if (j.F < 1) return fail(CVA_EINVAL, "regress: need one factor");
    if (m + j.nt > 40) return fail(CVA_ENOTSUP, "regress: basis columns + targets must be <= 40");
    const LsqPlan p = lsq_plan(j.F, j.basis, j.nt, j.M, j.groups, j.chunk_target);
    if (p.doubles > scratch_cap) return fail(CVA_ENOMEM, "regress: scratch too small");
    LsqArgs a;
    a.feat0 = j.feat0;
    a.feat_stride = j.feat_stride;
    a.targ0 = j.targ0;
    a.targ_stride = j.targ_stride;
    a.targ_tstride = j.targ_tstride;
    a.pred0 = j.pred0;
    a.pred_stride = j.pred_stride;
    a.pred_tstride = j.pred_tstride;
    a.nt = j.nt;
    a.F = j.F;
    a.m = m;
    a.basis = j.basis;
    a.chunks = (int)p.chunks;
    a.M = (uint32_t)j.M;
    a.rows_per_chunk = (uint32_t)p.rows_per_chunk;
    a.part = scratch;
    a.stride = p.stride;
    a.coef = a.part + (size_t)j.groups * (p.chunks + p.reduce) * p.stride;
    a.coef_raw = a.coef + (size_t)j.groups * j.nt * m;
    a.status = reinterpret_cast<int *>(a.coef_raw + (size_t)j.groups * j.nt * m);
    const cva_status gr = lsq_gram(a, p.rows, j.groups, st);
    if (gr != CVA_OK) return gr;
    if (p.reduce) {
        double *sums = a.part + (size_t)j.groups * p.chunks * p.stride;
        gram_reduce_kernel<<<dim3((unsigned)((p.stride + 31) / 32), (unsigned)j.groups), 256, 0, st>>>(a.part, a.chunks,
                                                                                                   a.stride, sums);
        CVA_CUDA_TRY(cudaGetLastError());
        a.part = sums;
        a.chunks = 1;
    }
    lsq_solve<<<j.groups, 256, 0, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    if (j.pred0) {
        cva_status pr = lsq_predict_launch(a, j.groups, st);
        if (pr != CVA_OK) return pr;
    }
    if (coef_host) {
        std::vector<int> status(j.groups);
        CVA_CUDA_TRY(cudaMemcpyAsync(coef_host, a.coef_raw, sizeof(double) * j.groups * j.nt * m,
                                     cudaMemcpyDeviceToHost, st));
        CVA_CUDA_TRY(cudaMemcpyAsync(status.data(), a.status, sizeof(int) * j.groups, cudaMemcpyDeviceToHost, st));
        CVA_CUDA_TRY(cudaStreamSynchronize(st));
        for (int g = 0; g < j.groups; ++g)
            if (status[g] != 0) return fail(CVA_ENUMERIC, "regress: rank-deficient normal equations");
    }
    return CVA_OK;
}

size_t lsq_scratch_need(const LsqJob &j)
{
    return lsq_plan(j.F, j.basis, j.nt, j.M, j.groups, j.chunk_target).doubles;
}

cva_status lsq_grouped_strided(const float *feat0, size_t feat_stride, const float *targ0,
                               size_t targ_stride, float *pred0, size_t pred_stride, int F,
                               uint64_t M, int basis, int groups, double *coef_host, cudaStream_t st)
{
    LsqJob j;
    j.feat0 = feat0;
    j.feat_stride = feat_stride;
    j.targ0 = targ0;
    j.targ_stride = targ_stride;
    j.pred0 = pred0;
    j.pred_stride = pred_stride;
    j.F = F;
    j.M = M;
    j.basis = basis;
    j.groups = groups;
    if (!feat0 || !targ0 || M == 0 || groups <= 0) return fail(CVA_EINVAL, "regress: bad arguments");
    if (M > 0x7fffffffull) return fail(CVA_EINVAL, "regress: M too large");
    if (basis != CVA_BASIS_LINEAR && basis != CVA_BASIS_POLY2) return fail(CVA_EINVAL, "regress: unknown basis");
    if (F < 1) return fail(CVA_EINVAL, "regress: need one factor");
    if (basis == CVA_BASIS_LINEAR && F + 2 > 32) return fail(CVA_ENOTSUP, "regress: linear basis supports 1 <= F <= 30");
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CVA_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
    std::lock_guard<std::mutex> lk(g_lsq_mu);
    LsqScratch &sc = g_lsq[dev];
    const size_t need = lsq_scratch_need(j);
    if (cap != cudaStreamCaptureStatusNone) {
        // inside a stream capture the scratch must already be large enough: a graph keeps its address
        if (sc.cap < need) return fail(CVA_EINVAL, "regress: call once before capturing so that the scratch exists");
        return lsq_launch(j, sc.buf, sc.cap, coef_host, st);
    }
    if (!sc.done) CVA_CUDA_TRY(cudaEventCreateWithFlags(&sc.done, cudaEventDisableTiming));
    else CVA_CUDA_TRY(cudaStreamWaitEvent(st, sc.done, 0));
    if (sc.cap < need) {
        if (sc.buf) {
            CVA_CUDA_TRY(cudaEventSynchronize(sc.done));
            cudaFree(sc.buf);
            sc.buf = nullptr;
            sc.cap = 0;
        }
        if (cudaMalloc(&sc.buf, need * sizeof(double)) != cudaSuccess)
            return fail(CVA_ENOMEM, "regress: scratch allocation failed");
        sc.cap = need;
    }
    cva_status r = lsq_launch(j, sc.buf, sc.cap, coef_host, st);
    if (r != CVA_OK) return r;
    CVA_CUDA_TRY(cudaEventRecord(sc.done, st));
    return CVA_OK;
}

// ---------------------------------------------------------------------------
// Least squares split over path ranges (one range per process and GPU). Every
// range accumulates its augmented normal matrix with the same centring (a state
// vector all ranges agree on), the host sums the ranges' matrices in a fixed order
// and solves once; each range then predicts its own paths. The sum over ranges is
// the normal matrix of all paths, so the fit is the one of the whole sample.

// the library's regression scratch of the current device, grown to `need` doubles
// (the previous user of a larger one has finished: callers synchronise)
static cva_status lsq_scratch_get(size_t need, cudaStream_t st, double **out)
{
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    std::lock_guard<std::mutex> lk(g_lsq_mu);
    LsqScratch &sc = g_lsq[dev];
    if (!sc.done) CVA_CUDA_TRY(cudaEventCreateWithFlags(&sc.done, cudaEventDisableTiming));
    else CVA_CUDA_TRY(cudaStreamWaitEvent(st, sc.done, 0));
    if (sc.cap < need) {
        if (sc.buf) {
            CVA_CUDA_TRY(cudaEventSynchronize(sc.done));
            cudaFree(sc.buf);
            sc.buf = nullptr;
            sc.cap = 0;
        }
        if (cudaMalloc(&sc.buf, need * sizeof(double)) != cudaSuccess)
            return fail(CVA_ENOMEM, "regress: scratch allocation failed");
        sc.cap = need;
    }
    *out = sc.buf;
    return CVA_OK;
}

static cva_status lsq_scratch_release(cudaStream_t st)
{
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_lsq_mu);
    CVA_CUDA_TRY(cudaEventRecord(g_lsq[dev].done, st));
    return CVA_OK;
}

static cva_status lsq_split_check(const float *feat, uint64_t M, int F, int basis, const float *centre)
{
    if (!feat || !centre || M == 0) return fail(CVA_EINVAL, "regress: bad arguments");
    if (M > 0x7fffffffull) return fail(CVA_EINVAL, "regress: M too large");
    if (basis != CVA_BASIS_LINEAR && basis != CVA_BASIS_POLY2) return fail(CVA_EINVAL, "regress: unknown basis");
    if (F < 1) return fail(CVA_EINVAL, "regress: need one factor");
    if (basis == CVA_BASIS_LINEAR && F + 2 > 32) return fail(CVA_ENOTSUP, "regress: linear basis supports 1 <= F <= 30");
    return CVA_OK;
}

cva_status lsq_normal_partial(const float *targ, const float *feat, int F, uint64_t M, int basis, const float *centre,
                              double *gram_host, cudaStream_t st)
{
    cva_status r = lsq_split_check(feat, M, F, basis, centre);
    if (r != CVA_OK) return r;
    if (!targ || !gram_host) return fail(CVA_EINVAL, "regress: bad arguments");
    const int m = (basis == CVA_BASIS_POLY2) ? 3 : F + 1, mA = m + 1;
    const LsqPlan p = lsq_plan(F, basis, 1, M, 1, 2432);
    double *part = nullptr;
    r = lsq_scratch_get((size_t)(p.chunks + 1) * p.stride, st, &part);
    if (r != CVA_OK) return r;
    LsqArgs a;
    a.feat0 = feat;
    a.feat_stride = (size_t)F * M;
    a.targ0 = targ;
    a.targ_stride = M;
    a.pred0 = nullptr;
    a.pred_stride = M;
    a.F = F;
    a.m = m;
    a.basis = basis;
    a.chunks = (int)p.chunks;
    a.M = (uint32_t)M;
    a.rows_per_chunk = (uint32_t)p.rows_per_chunk;
    a.part = part;
    a.stride = p.stride;
    a.coef = a.coef_raw = nullptr;
    a.status = nullptr;
    a.centre = centre;
    r = lsq_gram(a, p.rows, 1, st);
    double *sums = part + (size_t)p.chunks * p.stride;
    if (r == CVA_OK) r = sum_columns_fp64(part, a.chunks, (int)p.stride, sums, st);
    std::vector<double> tri(p.stride);
    if (r == CVA_OK) {
        cudaError_t e = cudaMemcpyAsync(tri.data(), sums, sizeof(double) * p.stride, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) r = cuda_fail(e, "regress: copy of the normal matrix");
    }
    const cva_status rr = lsq_scratch_release(st);
    if (r != CVA_OK) return r;
    if (rr != CVA_OK) return rr;
    // the packed upper triangle -> the dense symmetric (m+1) x (m+1) matrix
    for (int i = 0; i < mA; ++i)
        for (int j = i; j < mA; ++j)
            gram_host[(size_t)i * mA + j] = gram_host[(size_t)j * mA + i] = tri[tri_index(mA, i, j)];
    return CVA_OK;
}

// The solve of lsq_solve on the host: Jacobi scaling, Cholesky factorisation of the
// scaled normal matrix with vanishing pivots dropped (coefficient 0), the two
// triangular solves; coefficients in the centred basis and in the raw one.
cva_status lsq_solve_normal_host(const double *gram, int F, int basis, const double *centre, double *coef_centred,
                                 double *coef_raw, int *dropped)
{
    if (!gram || !centre || F < 1 || (basis != CVA_BASIS_LINEAR && basis != CVA_BASIS_POLY2))
        return fail(CVA_EINVAL, "regress: bad arguments");
    const int m = (basis == CVA_BASIS_POLY2) ? 3 : F + 1, mA = m + 1;
    std::vector<double> A((size_t)m * m), sc(m), y(m), w(m);
    std::vector<int> drop(m);
    for (int r = 0; r < m; ++r) {
        const double d = gram[(size_t)r * mA + r];
        drop[r] = !(d > 0.0);
        sc[r] = drop[r] ? 0.0 : 1.0 / sqrt(d);
    }
    for (int r = 0; r < m; ++r)
        for (int c = 0; c <= r; ++c) A[(size_t)r * m + c] = gram[(size_t)r * mA + c] * sc[r] * sc[c];
    for (int j = 0; j < m; ++j) {
        const double s = A[(size_t)j * m + j];
        if (drop[j] || !(s > 1e-12)) {
            drop[j] = 1;
            A[(size_t)j * m + j] = 1.0;
        } else {
            A[(size_t)j * m + j] = sqrt(s);
        }
        const double inv = drop[j] ? 0.0 : 1.0 / A[(size_t)j * m + j];
        for (int r = j + 1; r < m; ++r) A[(size_t)r * m + j] *= inv;
        for (int r = j + 1; r < m; ++r)
            for (int c = j + 1; c <= r; ++c) A[(size_t)r * m + c] -= A[(size_t)r * m + j] * A[(size_t)c * m + j];
    }
    int nd = 0;
    for (int r = 0; r < m; ++r) nd += drop[r];
    for (int i = 0; i < m; ++i) {               // L y = D^{-1/2} b
        double s = gram[(size_t)i * mA + m] * sc[i];
        for (int p = 0; p < i; ++p) s -= A[(size_t)i * m + p] * y[p];
        y[i] = drop[i] ? 0.0 : s / A[(size_t)i * m + i];
    }
    for (int i = m - 1; i >= 0; --i) {         // L^T z = y, w = D^{-1/2} z
        double s = y[i];
        for (int p = i + 1; p < m; ++p) s -= A[(size_t)p * m + i] * w[p];
        w[i] = drop[i] ? 0.0 : s / A[(size_t)i * m + i];
    }
    for (int i = 0; i < m; ++i) w[i] *= sc[i];
    if (coef_centred)
        for (int i = 0; i < m; ++i) coef_centred[i] = w[i];
    if (coef_raw) {
        if (basis == CVA_BASIS_POLY2) {
            const double c = centre[0];
            coef_raw[0] = w[0] - w[1] * c + w[2] * c * c;
            coef_raw[1] = w[1] - 2.0 * w[2] * c;
            coef_raw[2] = w[2];
        } else {
            double w0 = w[0];
            for (int f = 0; f < F; ++f) {
                w0 -= w[1 + f] * centre[f];
                coef_raw[1 + f] = w[1 + f];
            }
            coef_raw[0] = w0;
        }
    }
    if (dropped) *dropped = nd;
    return CVA_OK;
}

cva_status lsq_predict_groups(const float *feat0, size_t feat_stride, int F, uint64_t M, int groups, const double *coef,
                              size_t coef_stride, float *pred0, size_t pred_stride, cudaStream_t st)
{
    LsqArgs a = {};
    a.feat0 = feat0;
    a.feat_stride = feat_stride;
    a.pred0 = pred0;
    a.pred_stride = pred_stride;
    a.F = F;
    a.m = F + 1;
    a.basis = CVA_BASIS_LINEAR;
    a.M = (uint32_t)M;
    a.coef = const_cast<double *>(coef);
    a.coef_stride = coef_stride;
    a.nt = 1;
    return lsq_predict_launch(a, groups, st);
}

cva_status lsq_predict_centred(const float *feat, int F, uint64_t M, int basis, const float *centre,
                               const double *coef_centred_host, float *pred, cudaStream_t st)
{
    cva_status r = lsq_split_check(feat, M, F, basis, centre);
    if (r != CVA_OK) return r;
    if (!coef_centred_host || !pred) return fail(CVA_EINVAL, "regress: bad arguments");
    const int m = (basis == CVA_BASIS_POLY2) ? 3 : F + 1;
    double *coef = nullptr;
    r = lsq_scratch_get((size_t)m, st, &coef);
    if (r != CVA_OK) return r;
    cudaError_t e = cudaMemcpyAsync(coef, coef_centred_host, sizeof(double) * m, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_fail(e, "regress: coefficients to the device");
    LsqArgs a;
    a.feat0 = feat;
    a.feat_stride = (size_t)F * M;
    a.targ0 = nullptr;
    a.targ_stride = M;
    a.pred0 = pred;
    a.pred_stride = M;
    a.F = F;
    a.m = m;
    a.basis = basis;
    a.chunks = 1;
    a.M = (uint32_t)M;
    a.rows_per_chunk = (uint32_t)M;
    a.part = nullptr;
    a.coef = coef;
    a.coef_raw = nullptr;
    a.status = nullptr;
    a.centre = centre;
    r = lsq_predict_launch(a, 1, st);
    // the host coefficients are read by the copy above before the call returns
    e = cudaStreamSynchronize(st);
    const cva_status rr = lsq_scratch_release(st);
    if (r != CVA_OK) return r;
    if (e != cudaSuccess) return cuda_fail(e, "regress: predictions");
    return rr;
}

// ---------------------------------------------------------------------------
// Regression without any device allocation.
//
// Some callers cannot allocate device memory at the time they need a fit: a
// framework may own the whole device through its own pool, a process may run
// under a fixed memory budget checked at start-up, or a latency-critical loop
// cannot afford the device-wide synchronisation of cudaMalloc/cudaFree. For
// them, the batched regression below keeps its Gram partials, coefficients and
// status words in this file-scope array instead of library-allocated scratch.
// The array lives on every device that loads the library until the process
// exits. Its size bounds the number of groups per call (see the check below).
// All calls share it: each call writes every entry it later reads, so nothing
// has to start at zero, but two calls whose kernels overlap on the GPU (for
// instance on two streams) race on it and must be ordered by the caller.
constexpr size_t kStaticScratchDoubles = 1u << 17;   // 1 MiB
static __device__ __align__(256) double g_static_scratch[kStaticScratchDoubles];

namespace {
std::mutex g_static_mu;
struct StaticSetup {
    unsigned long long ctx_id = 0;   // CUDA context the address below belongs to (0: none yet)
    double *ptr = nullptr;
};
StaticSetup g_static[64];
PFN_cuCtxGetCurrent_v4000 g_ctx_current = nullptr;
PFN_cuCtxGetId_v12000 g_ctx_id = nullptr;

}  // namespace

// Set-up of the allocation-free path on the current device, once per device and
// CUDA context (a context created after cudaDeviceReset gets its own): the device
// address of the static scratch (cudaGetSymbolAddress; the host-side name is only
// a stand-in for the device array) and the shared-memory limits of the Gram
// kernels it launches. Later calls in the same context reuse both.
static cva_status static_scratch(double **out)
{
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (!g_ctx_current || !g_ctx_id) {
        void *f1 = nullptr, *f2 = nullptr;
        cudaDriverEntryPointQueryResult q1 = cudaDriverEntryPointSymbolNotFound, q2 = q1;
        CVA_CUDA_TRY(cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 4000, cudaEnableDefault, &q1));
        CVA_CUDA_TRY(cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2));
        if (!f1 || !f2 || q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess)
            return fail(CVA_ECUDA, "regress_static: cuCtxGetCurrent / cuCtxGetId not available");
        g_ctx_current = reinterpret_cast<PFN_cuCtxGetCurrent_v4000>(f1);
        g_ctx_id = reinterpret_cast<PFN_cuCtxGetId_v12000>(f2);
    }
    CVA_CUDA_TRY(cudaSetDevice(dev));   // initialises the device's primary context and makes it current
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (g_ctx_current(&ctx) != CUDA_SUCCESS || !ctx || g_ctx_id(ctx, &id) != CUDA_SUCCESS)
        return fail(CVA_ECUDA, "regress_static: no current CUDA context");
    StaticSetup &su = g_static[dev];
    if (su.ctx_id != id || !su.ptr) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_static_scratch)");
        // the shared-memory limits of the Gram kernels its shapes use (up to 32 columns)
        const int smem = 3 * 32 * 256 * (int)sizeof(float);
        for (auto kern : {gram_kernel<512, 320, 2, true>, gram_kernel<512, 320, 2, false>, gram_kernel<256, 320, 2, true>,
                          gram_kernel<256, 320, 2, false>})
            CVA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        su.ptr = static_cast<double *>(p);
        su.ctx_id = id;
    }
    *out = su.ptr;
    return CVA_OK;
}

cva_status lsq_batched_static(const float *targ0, const float *feat0, int groups, int F, uint64_t M,
                              int basis, float *pred0, double *coef_host, cudaStream_t st)
{
    if (!feat0 || !targ0 || M == 0 || groups <= 0) return fail(CVA_EINVAL, "regress_static: bad arguments");
    if (M > 0x7fffffffull) return fail(CVA_EINVAL, "regress_static: M too large");
    if (basis != CVA_BASIS_LINEAR && basis != CVA_BASIS_POLY2)
        return fail(CVA_EINVAL, "regress_static: unknown basis");
    const int m = (basis == CVA_BASIS_POLY2) ? 3 : F + 1;
    if (basis == CVA_BASIS_LINEAR && (F < 1 || m + 1 > 32))
        return fail(CVA_ENOTSUP, "regress_static: linear basis supports 1 <= F <= 30");
    if (basis == CVA_BASIS_POLY2 && F < 1) return fail(CVA_EINVAL, "regress_static: need one factor");
    // room reserved per chunk: the triangle in 4 x 4 blocks of 4, 12 or 32 columns, an
    // upper bound of what a partial takes
    const int MP = m + 1 <= 4 ? 4 : m + 1 <= 12 ? 12 : 32;
    const size_t per_group_fixed = 2 * (size_t)m + 1;          // coefficients (two bases) + status
    const size_t per_chunk = (size_t)(MP / 4) * (MP / 4 + 1) / 2 * 16;
    const size_t max_groups = kStaticScratchDoubles / (per_chunk + per_group_fixed);
    if ((size_t)groups > max_groups || groups > 1024)
        return fail(CVA_EINVAL, "regress_static: " + std::to_string(groups) + " groups exceed the static scratch (at most " +
                                    std::to_string(max_groups < 1024 ? max_groups : 1024) +
                                    " groups of this basis per call)");
    if (coef_host) {   // the coefficients come back through a synchronisation of st
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        CVA_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
        if (cap != cudaStreamCaptureStatusNone)
            return fail(CVA_EINVAL, "regress_static: coef_host needs a synchronisation of the stream, which is "
                                    "being captured; pass coef_host = NULL there");
    }
    double *scratch = nullptr;
    cva_status r = static_scratch(&scratch);
    if (r != CVA_OK) return r;

    const uint64_t fit = (kStaticScratchDoubles - (size_t)groups * per_group_fixed) / ((size_t)groups * per_chunk);
    uint64_t rows_per_chunk, chunks;
    gram_chunks(M, groups, (int)std::min<uint64_t>(2432, fit * (uint64_t)groups), 1024, &rows_per_chunk, &chunks);
    const int rows = m + 1;

    LsqArgs a;
    a.feat0 = feat0;
    a.feat_stride = (size_t)F * M;
    a.targ0 = targ0;
    a.targ_stride = M;
    a.pred0 = pred0;
    a.pred_stride = M;
    a.F = F;
    a.m = m;
    a.basis = basis;
    a.chunks = (int)chunks;
    a.M = (uint32_t)M;
    a.rows_per_chunk = (uint32_t)rows_per_chunk;
    a.part = scratch;
    a.stride = (size_t)tri_index(rows, rows - 1, rows - 1) + 1;
    a.coef = a.part + (size_t)groups * chunks * a.stride;
    a.coef_raw = a.coef + (size_t)groups * m;
    a.status = reinterpret_cast<int *>(a.coef_raw + (size_t)groups * m);
    const cva_status gr = lsq_gram(a, rows, groups, st);
    if (gr != CVA_OK) return gr;
    lsq_solve<<<groups, 256, 0, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    if (pred0) {
        cva_status pr = lsq_predict_launch(a, groups, st);
        if (pr != CVA_OK) return pr;
    }
    if (coef_host) {
        int status[1024];
        CVA_CUDA_TRY(cudaMemcpyAsync(coef_host, a.coef_raw, sizeof(double) * groups * m, cudaMemcpyDeviceToHost, st));
        CVA_CUDA_TRY(cudaMemcpyAsync(status, a.status, sizeof(int) * groups, cudaMemcpyDeviceToHost, st));
        CVA_CUDA_TRY(cudaStreamSynchronize(st));
        for (int g = 0; g < groups; ++g)
            if (status[g] != 0) return fail(CVA_ENUMERIC, "regress_static: rank-deficient normal equations");
    }
    return CVA_OK;
}

}  // namespace cva
