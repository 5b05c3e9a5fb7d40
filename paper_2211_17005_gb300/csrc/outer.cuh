// Outer-path kernels of the hierarchical CVA simulation, templated on the model
// shape. Each translation unit that includes this header gets its own copy of
// the constant-memory tables and of their ownership state, so instantiations
// compile in parallel.
//
// sim_kernel (32 outer paths per block, Sec. 3.2): the time loop. Per
// Euler-Maruyama sub-step (Remark rem:finecoarse): Philox normals, correlation
// by the Cholesky factor, Hull-White rates with the quanto drift, lognormal FX,
// CIR intensities with full truncation (App. B), and the left-point integrals
// int r^0 (FP64) and Lambda^c (compensated FP32). At each pricing date it
// stores the state Y_j, int r^0 and the threshold 1 - exp(-Lambda_c(t_j)).
//
// price_kernel (two outer paths per thread, a period's pricing dates per block): the
// portfolio MtM per counterparty from the App. B swap formula, regrouped exactly by
// (counterparty, currency, reset date), and the exposure (1-R_c) beta_j MtM^+.
// It reads the state of date j and the short rates of the last reset date
// (Remark rem:pathdep) from the stored states; every (path, date) is
// independent, so the pricing runs at full occupancy.
//
// Outputs are structure-of-arrays with the path index fastest.
#pragma once
#include <algorithm>
#include <climits>
#include <mutex>
#include <type_traits>

#include "cva_internal.h"
#include "rng.cuh"
#include "sum_pair.cuh"
#include "umma.cuh"

namespace cva {
namespace {

static __constant__ SimConsts c_sim;
#ifdef CVA_CONST_WEIGHTS   // the run-time-shape adjoint's; every other kernel reads them from global memory
static __constant__ SimWeights c_w;
#endif

// two FP32 values in one register pair, operated on together
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// expm1(x) by its Taylor series to degree 8 for |x| <= 1/4 (relative error below
// 2e-10 there, so the rounding of the FMAs dominates), library expm1f elsewhere.
__device__ __forceinline__ float expm1_small(float x)
{
    if (fabsf(x) > 0.25f) return expm1f(x);
    float p = 1.f / 40320.f;
    p = fmaf(p, x, 1.f / 5040.f);
    p = fmaf(p, x, 1.f / 720.f);
    p = fmaf(p, x, 1.f / 120.f);
    p = fmaf(p, x, 1.f / 24.f);
    p = fmaf(p, x, 1.f / 6.f);
    p = fmaf(p, x, 0.5f);
    p = fmaf(p, x, 1.f);
    return p * x;
}

enum class SimMode { plain, adjoint, forward, restart };

struct OuterArgs {
    uint32_t M, k0, seed_lo, seed_hi;
    int branch_step;                   // fine steps q >= branch_step draw with counter word `branch`
    uint32_t branch;
    const float4 *__restrict__ zc;     // [n+1][E][G] (lnA, B, dlnA, dB)
    const float2 *__restrict__ fix;    // [periods+1][E] (lnA, B)
    const float *__restrict__ drift;   // [n*S][E]
    float *features, *disc, *thr, *expo, *mtm;
    const float *w_glob;               // device copy of the date-bucketed weights: wA [kMaxW], then wK [kMaxW]
    // a run that starts at pricing date `start` > 0 takes the state there from features and
    // ckpt, which a run with save_date = start has left: [2C][M] Lambda and its compensation,
    // ckpt_I0 [M] int r^0
    int start, save_date;
    float *ckpt;
    double *ckpt_I0;
    float *inc, *gpre;                 // the adjoint's only: [n*S][F][M] increments, [n*S][C][M] intensities before a fine step
};

// Block: 32 outer paths (lane = path), NW warps. The normals of a fine step depend on no
// state, so the block takes 8 steps at a time: its warps draw and correlate a step's
// increments W = L z of the 32 paths each into shared memory, then the recursions run over
// the 8 steps with the factors split over the warps (economies and counterparties w, w + NW,
// ...; every warp that holds an FX rate carries its own copy of r^0). The noise is 97% of
// the instructions and is spread evenly; 2^15 paths give 8192 warps instead of 1024.
//
// The correlation multiplies by packed pairs of rows of L (fma.rn.f32x2, each half rounded
// as a single FMA): 352 instructions a step at 27 factors against 728 with one constant
// load and one FMA per entry.
//
// Modes: forward, for the smooth CVA_0, which keeps e^{-Lambda} in the place of the thresholds;
// adjoint, which also keeps the increments and intensities of every fine step; restart, a
// run that starts at a pricing date or saves what such a run needs. Separate instances, as
// their pointers would cost the plain one's four-warp form its registers; the eight-warp
// forms, which small path counts take, hold 80 for three blocks a multiprocessor and spill
// some of them.
//
// Bound by instruction issue (Philox, logarithm, square root and sine-cosine of 14
// Box-Muller pairs, the correlation): 2650 instructions a (path, step) at 27 factors and
// 85% of the issue slots. Paper shape, 2^17 paths and 100 steps: 1.28 -> 1.09 ms against a
// thread per path over all steps (96 registers, 7 to 14 warps a multiprocessor); 2^15
// paths and 2500 steps 9.09 -> 6.3 ms; 2^14 paths and 100 steps 0.43 -> 0.18 ms.
template <int E, int C, int CS, int NW, SimMode MODE>
__global__ void __launch_bounds__(32 * NW, NW == 8 ? 3 : 5) sim_kernel(OuterArgs a)
{
    constexpr int F = 2 * E - 1 + CS;
    constexpr int NB = (F + 3) / 4, FP = (F + 1) / 2 * 2;
    constexpr int ME = (E + NW - 1) / NW, MC = (C + NW - 1) / NW;   // factors of a warp
    constexpr bool ADJ = MODE == SimMode::adjoint, SURV = ADJ || MODE == SimMode::forward, CKPT = MODE == SimMode::restart;
    constexpr int NS = F <= 8 ? 32 : 8;                             // fine steps at a time
    __shared__ float Ws[NS][F][32], R0[NS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t kl = blockIdx.x * 32u + (uint32_t)lane;
    const bool live = kl < a.M;
    const uint32_t k = a.k0 + kl;
    const size_t M = a.M;
    const int n = c_sim.n, S = c_sim.S;
    const float ds = c_sim.ds;
    const double ds_d = c_sim.ds_d;

    // this warp's factors and their coefficients
    float r0 = c_sim.r0[0], r[ME], lchi[ME], gam[MC], lam[MC], lamc[MC];
    double I0 = 0.0;
    auto has_e = [&](int i) { return NW * (i + 1) <= E || warp + NW * i < E; };
    auto has_c = [&](int i) { return NW * (i + 1) <= C || warp + NW * i < C; };
    auto is_cir = [&](int i) { return NW * (i + 1) <= CS || warp + NW * i < CS; };
#pragma unroll
    for (int i = 0; i < ME; ++i) {
        const int e = has_e(i) ? warp + NW * i : 0;
        r[i] = c_sim.r0[e];
        lchi[i] = c_sim.lchi0[e];
    }
#pragma unroll
    for (int i = 0; i < MC; ++i) {
        const int c = has_c(i) ? warp + NW * i : 0;
        gam[i] = c_sim.gamma0[c];
        lam[i] = lamc[i] = 0.f;
    }
    const int start = CKPT ? a.start : 0;
    if (start > 0) {
        const float *fe = a.features + (size_t)start * F * M + (live ? kl : 0u);
        const uint32_t kr = live ? kl : 0u;
        r0 = __ldg(fe);
#pragma unroll
        for (int i = 0; i < ME; ++i)
            if (has_e(i)) {
                const int e = warp + NW * i;
                r[i] = __ldg(fe + (size_t)e * M);
                if (e > 0) lchi[i] = __ldg(fe + (size_t)(E - 1 + e) * M);
            }
#pragma unroll
        for (int i = 0; i < MC; ++i)
            if (has_c(i)) {
                const int c = warp + NW * i;
                if (is_cir(i)) gam[i] = __ldg(fe + (size_t)(2 * E - 1 + c) * M);
                lam[i] = a.ckpt[(size_t)c * M + kr];
                lamc[i] = a.ckpt[(size_t)(C + c) * M + kr];
            }
        I0 = a.ckpt_I0[kr];
    }
    // rows of a date this warp writes: the rate and the log FX rate of its first economy,
    // its first counterparty's intensity and threshold; the next ones follow NW rows apart
    float *pr = a.features + (size_t)warp * M + kl, *px = pr + (size_t)(E - 1) * M, *pg = pr + (size_t)(2 * E - 1) * M;
    float *pt = a.thr + (size_t)warp * M + kl, *pd = a.disc + kl;
    int date = 0;
    auto write_date = [&]() {
        if (live) {
            if (CKPT && date == a.save_date)
#pragma unroll
                for (int i = 0; i < MC; ++i)
                    if (has_c(i)) {
                        a.ckpt[(size_t)(warp + NW * i) * M + kl] = lam[i];
                        a.ckpt[(size_t)(C + warp + NW * i) * M + kl] = lamc[i];
                    }
#pragma unroll
            for (int i = 0; i < ME; ++i)
                if (has_e(i)) {
                    pr[(size_t)(NW * i) * M] = r[i];
                    if (i > 0 || warp > 0) px[(size_t)(NW * i) * M] = lchi[i];
                }
#pragma unroll
            for (int i = 0; i < MC; ++i)
                if (has_c(i)) {
                    if (is_cir(i)) pg[(size_t)(NW * i) * M] = gam[i];
                    // threshold (0 at date 0) or survival factor
                    pt[(size_t)(NW * i) * M] = SURV ? expf(-lam[i]) : -expm1f(-lam[i]);
                }
        }
        pr += (size_t)F * M;
        px += (size_t)F * M;
        pg += (size_t)F * M;
        pt += (size_t)C * M;
        ++date;
    };
    const int steps = n * S, first = start * S;
    const float *drow = a.drift + (size_t)first * E;
    if (start > 0) {   // the dates up to the start are in place
        pr += (size_t)(start + 1) * F * M;
        px += (size_t)(start + 1) * F * M;
        pg += (size_t)(start + 1) * F * M;
        pt += (size_t)(start + 1) * C * M;
        pd += (size_t)start * M;
        date = start + 1;
    } else {
        write_date();
        if (warp == NW - 1 && live) *pd = 0.f;
    }
    int jd = start;   // dates of int r^0 written so far
    int s = 0, sd = 0;   // sub-step of the next fine step (of the factors, of int r^0)
    for (int q0 = first; q0 < steps; q0 += NS) {
#pragma unroll 1
        for (int v = warp; v < NS && q0 + v < steps; v += NW) {
            const int q = q0 + v;
            // correlated increments W = L z, accumulated one Philox block (four
            // normals) at a time
            f32x2 W[FP / 2];
#pragma unroll
            for (int i = 0; i < FP / 2; ++i) W[i] = pack2(0.f, 0.f);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const uint4 x = philox4x32_10(make_uint4(k, (uint32_t)q, q >= a.branch_step ? a.branch : 0u,
                                                         (kStreamOuter << 24) | (uint32_t)b),
                                              a.seed_lo, a.seed_hi);
                float z[4];
                box_muller(x.x, x.y, z[0], z[1]);
                box_muller(x.z, x.w, z[2], z[3]);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int col = 4 * b + t;
                    if (col < F) {
                        const f32x2 zz = pack2(z[t], z[t]);
#pragma unroll
                        for (int i = col / 2; i < FP / 2; ++i) {
                            const float2 l = *reinterpret_cast<const float2 *>(&c_sim.Lc[col * FP + 2 * i]);
                            W[i] = fma2(pack2(l.x, l.y), zz, W[i]);
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < F; ++i) {
                const float2 w = unpack2(W[i / 2]);
                Ws[v][i][lane] = i & 1 ? w.y : w.x;
                if (ADJ && live) a.inc[((size_t)q * F + i) * M + kl] = i & 1 ? w.y : w.x;
            }
        }
        __syncthreads();
        const int chunk = min(NS, steps - q0);
        const float *W = &Ws[0][0][lane];
        // the coefficients, in registers over the chunk only
        float ha[ME], hs[ME], fd[ME], fs[ME], ckt[MC], ck[MC], cn[MC], ha0 = c_sim.hw_a_ds[0], hs0 = c_sim.hw_sig_sqds[0];
#pragma unroll
        for (int i = 0; i < ME; ++i) {
            const int e = has_e(i) ? warp + NW * i : 0;
            ha[i] = c_sim.hw_a_ds[e];
            hs[i] = c_sim.hw_sig_sqds[e];
            fd[i] = c_sim.fx_drift_ds[e];
            fs[i] = c_sim.fx_sig_sqds[e];
            asm volatile("" : "+f"(ha[i]), "+f"(hs[i]), "+f"(fd[i]), "+f"(fs[i]));
        }
#pragma unroll
        for (int i = 0; i < MC; ++i) {
            const int c = has_c(i) ? warp + NW * i : 0;
            ckt[i] = c_sim.cir_ktds[c];
            ck[i] = c_sim.cir_kds[c];
            cn[i] = c_sim.cir_nu_sqds[c];
            asm volatile("" : "+f"(ckt[i]), "+f"(ck[i]), "+f"(cn[i]));
        }
        asm volatile("" : "+f"(ha0), "+f"(hs0));
#pragma unroll 1
        for (int u = 0; u < chunk; ++u, W += F * 32, drow += E) {
            if (warp == 0) R0[u][lane] = r0;
            // Lambda^c: left-point integral, compensated FP32, kept non-decreasing
#pragma unroll
            for (int i = 0; i < MC; ++i)
                if (has_c(i)) {
                    if (ADJ && live) a.gpre[((size_t)(q0 + u) * C + warp + NW * i) * M + kl] = gam[i];
                    const float gp = fmaxf(gam[i], 0.f);
                    const float y = fmaf(gp, ds, -lamc[i]);
                    const float t = lam[i] + y;
                    lamc[i] = (t - lam[i]) - y;
                    lam[i] = fmaxf(t, lam[i]);
                    if (is_cir(i))
                        gam[i] += ckt[i] - ck[i] * gp + cn[i] * sqrtf(gp) * W[(2 * E - 1 + warp + NW * i) * 32];
                }
#pragma unroll
            for (int i = 0; i < ME; ++i)
                if (has_e(i)) {
                    const int e = warp + NW * i;
                    if (i > 0 || warp > 0) lchi[i] += fmaf(r0 - r[i], ds, fd[i]) + fs[i] * W[(E - 1 + e) * 32];
                    r[i] += (__ldg(drow + e) - ha[i] * r[i]) + hs[i] * W[e * 32];
                }
            r0 += (__ldg(drow) - ha0 * r0) + hs0 * W[0];
            if (++s == S) {   // pricing date
                s = 0;
                write_date();
            }
        }
        __syncthreads();   // the increments are read before the next steps overwrite them
        // int r^0 in FP64, left points; one warp and one loop for it (the FP64 pipe is
        // narrow, and instructions predicated off in the other warps would still occupy it)
        if (warp == NW - 1)
            for (int u = 0; u < chunk; ++u) {
                I0 = fma((double)R0[u][lane], ds_d, I0);
                if (++sd == S) {
                    sd = 0;
                    pd += M;
                    ++jd;
                    if (live) {
                        *pd = (float)I0;
                        if (CKPT && jd == a.save_date) a.ckpt_I0[kl] = I0;
                    }
                }
            }
    }
}

// sim_kernel for one economy: a thread per path, with the noise of a step (one Philox block) in its
// registers. There are no factors to split over warps, and where the paths fill the chip the
// barriers and idle warps of sim_kernel only cost. Same operations in the same order, so
// the same bits. Two counterparties of constant intensity, 50 dates, four warps per 32 paths / a
// thread per path: 2^14 paths 27 / 28 us, 2^15 36 / 31, 2^17 97 / 63, 2^20 669 / 382 us.
template <int C, int CS, SimMode MODE>
__global__ void __launch_bounds__(128, 8) sim_thread_kernel(OuterArgs a)
{
    constexpr int F = 1 + CS, NB = (F + 3) / 4;
    constexpr bool ADJ = MODE == SimMode::adjoint, SURV = ADJ || MODE == SimMode::forward, CKPT = MODE == SimMode::restart;
    const uint32_t kl = blockIdx.x * 128u + threadIdx.x;
    if (kl >= a.M) return;
    const uint32_t k = a.k0 + kl;
    const size_t M = a.M;
    const int n = c_sim.n, S = c_sim.S;
    const float ds = c_sim.ds;
    const double ds_d = c_sim.ds_d;
    float r = c_sim.r0[0], gam[C], lam[C], lamc[C];
    double I0 = 0.0;
#pragma unroll
    for (int c = 0; c < C; ++c) {
        gam[c] = c_sim.gamma0[c];
        lam[c] = lamc[c] = 0.f;
    }
    const int start = CKPT ? a.start : 0;
    float *fe = a.features + kl, *th = a.thr + kl, *di = a.disc + kl;
    auto write_date = [&](int j) {
        fe[0] = r;
        *di = (float)I0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (c < CS) fe[(size_t)(1 + c) * M] = gam[c];
            th[(size_t)c * M] = SURV ? expf(-lam[c]) : -expm1f(-lam[c]);   // survival factor or threshold
            if (CKPT && j == a.save_date) {
                a.ckpt[(size_t)c * M + kl] = lam[c];
                a.ckpt[(size_t)(C + c) * M + kl] = lamc[c];
            }
        }
        if (CKPT && j == a.save_date) a.ckpt_I0[kl] = I0;
        fe += (size_t)F * M;
        th += (size_t)C * M;
        di += M;
    };
    if (start > 0) {   // the dates up to the start are in place
        fe += (size_t)start * F * M;
        r = fe[0];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (c < CS) gam[c] = fe[(size_t)(1 + c) * M];
            lam[c] = a.ckpt[(size_t)c * M + kl];
            lamc[c] = a.ckpt[(size_t)(C + c) * M + kl];
        }
        I0 = a.ckpt_I0[kl];
        fe += (size_t)F * M;
        th += (size_t)(start + 1) * C * M;
        di += (size_t)(start + 1) * M;
    } else {
        write_date(0);
    }
    for (int j = start + 1; j <= n; ++j) {
        for (int q = (j - 1) * S; q < j * S; ++q) {
            float W[F];
#pragma unroll
            for (int i = 0; i < F; ++i) W[i] = 0.f;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const uint4 x = philox4x32_10(make_uint4(k, (uint32_t)q, q >= a.branch_step ? a.branch : 0u,
                                                         (kStreamOuter << 24) | (uint32_t)b),
                                              a.seed_lo, a.seed_hi);
                float z[4];
                box_muller(x.x, x.y, z[0], z[1]);
                box_muller(x.z, x.w, z[2], z[3]);
#pragma unroll
                for (int t = 0; t < 4; ++t)
#pragma unroll
                    for (int i = 4 * b + t; i < F; ++i) W[i] = fmaf(c_sim.L[i * (i + 1) / 2 + 4 * b + t], z[t], W[i]);
            }
            I0 = fma((double)r, ds_d, I0);
#pragma unroll
            for (int i = 0; i < F; ++i)
                if (ADJ) a.inc[((size_t)q * F + i) * M + kl] = W[i];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (ADJ) a.gpre[((size_t)q * C + c) * M + kl] = gam[c];
                const float gp = fmaxf(gam[c], 0.f);
                const float y = fmaf(gp, ds, -lamc[c]);
                const float t = lam[c] + y;
                lamc[c] = (t - lam[c]) - y;
                lam[c] = fmaxf(t, lam[c]);
                if (c < CS)
                    gam[c] += c_sim.cir_ktds[c] - c_sim.cir_kds[c] * gp + c_sim.cir_nu_sqds[c] * sqrtf(gp) * W[c < CS ? 1 + c : 0];
            }
            r += (__ldg(a.drift + q) - c_sim.hw_a_ds[0] * r) + c_sim.hw_sig_sqds[0] * W[0];
        }
        write_date(j);
    }
}

// The path simulation in the form for its shape and path count (four: four warps per 32 paths
// whatever the count).
//  - 4 warps have the fewest instructions (more factors a warp) unless such blocks leave the
//    chip short of warps: at the paper shape 8 warps take 91 us against 115 us for 2^10 paths,
//    215 against 184 for 2^14 and 1265 against 1111 for 2^17;
//  - one economy takes a thread per path from six blocks of 32 paths a multiprocessor on
//    (sim_thread_kernel).
template <int E, int C, int CS, SimMode MODE>
void launch_sim(const OuterArgs &a, bool four, int sms, cudaStream_t st)
{
    const unsigned blocks = (a.M + 31u) / 32u;
    if constexpr (E == 1) {
        if (!four && blocks >= 6u * (unsigned)sms) {
            sim_thread_kernel<C, CS, MODE><<<(a.M + 127u) / 128u, 128, 0, st>>>(a);
            return;
        }
    }
    if (!four && blocks < 2u * (unsigned)sms) sim_kernel<E, C, CS, 8, MODE><<<blocks, 256, 0, st>>>(a);
    else sim_kernel<E, C, CS, 4, MODE><<<blocks, 128, 0, st>>>(a);
}

// Pricing on the FMA pipe: two paths per thread in packed FP32 pairs, the dates of one
// period (p delta, (p+1) delta] per block, NPB portfolios per block (blockIdx.z picks the
// group).
//
// A period's dates share the number LV = G - p of live reset dates, so the block runs the
// instantiation for it: bond prices and weight products of dead reset dates (45% of them
// on average) are not computed, and the loops over reset dates are unrolled without a
// test. All packed operations round each half as the scalar one (fma.rn.f32x2), and the
// terms left out are products with 0, so every split, period and portfolio grouping gives
// the same bits. The economies are a real loop: the code of one instantiation stays
// within the instruction cache (fully unrolled over economies and reset dates, a third of
// the warps waited for instructions).
//
// The group's weights wait in shared memory, negated and doubled (w, w) as the packed
// multiply wants them, two reset dates in a 16-byte broadcast load; so do the date's bond
// tables (read through L1 they were the longest wait) and, where they fit beside the
// weights, the running coupons at the fixing, which the period's dates share. The MtM enters as
//   acc = sum_h (-wA)(-D_h) + sum_g (-wK) Z_g,
// with -D_h = Z_{h-1} expm1(x_h), which is what the chain of bond prices produces.
//
// Bound by instruction issue and, within it, by shared-memory reads of the weights. Paper
// shape, 2^17 paths, 101 dates: 2.19 ms with a thread per (path, date), every reset date and
// the weights in constant memory, 1.19 ms with live dates and packed pairs, 1.00 ms with the
// tables and coupons in shared memory, 0.98 ms with a date's states in the L2 cache ahead.
struct PriceShape {
    int dates_per_block, splits;   // a period's dates in `splits` blocks of dates_per_block
    int start = 0;                 // dates up to this one are priced already
};

// Rates, log FX rates and discount integral of the warp's 32 paths from k at a date (state
// rows from fe, discount row dj) into the L2 cache, a lane per row; nothing past `end`.
template <int E>
__device__ __forceinline__ void prefetch_state(const float *fe, const float *dj, size_t M, uint32_t k, uint32_t end)
{
    static_assert(2 * E <= 32, "a lane per row");
    const uint32_t q = threadIdx.x & 31u;
    if (q < 2 * E && k < end)
        asm volatile("prefetch.global.L2 [%0];" ::"l"((q < 2 * E - 1 ? fe + q * M : dj) + k));
}

// fn(LV) for the run-time LV in 1..G (0: nothing is live)
template <int G, int LV = G, class Fn>
__device__ __forceinline__ void with_live(int lv, Fn &&fn)
{
    if constexpr (LV >= 0) {
        if (lv == LV) fn(std::integral_constant<int, LV>{});
        else with_live<G, LV - 1>(lv, fn);
    }
}

// expm1_small of both halves: the series for both, the library function for a half
// outside its range
__device__ __forceinline__ f32x2 expm1_small2(f32x2 x)
{
    f32x2 p = pack2(1.f / 40320.f, 1.f / 40320.f);
    p = fma2(p, x, pack2(1.f / 5040.f, 1.f / 5040.f));
    p = fma2(p, x, pack2(1.f / 720.f, 1.f / 720.f));
    p = fma2(p, x, pack2(1.f / 120.f, 1.f / 120.f));
    p = fma2(p, x, pack2(1.f / 24.f, 1.f / 24.f));
    p = fma2(p, x, pack2(1.f / 6.f, 1.f / 6.f));
    p = fma2(p, x, pack2(0.5f, 0.5f));
    p = fma2(p, x, pack2(1.f, 1.f));
    f32x2 r = mul2(p, x);
    const float2 xs = unpack2(x);
    if (fmaxf(fabsf(xs.x), fabsf(xs.y)) > 0.25f) {
        float2 v = unpack2(r);
        if (fabsf(xs.x) > 0.25f) v.x = expm1f(xs.x);
        if (fabsf(xs.y) > 0.25f) v.y = expm1f(xs.y);
        r = pack2(v.x, v.y);
    }
    return r;
}

// shared memory of price_kernel: weights, the date's tables, the coupons where they fit
template <int E, int C, int G, int NPB>
struct PriceSmem {
    static constexpr int weights = E * NPB * C * 2 * G * 8, tables = E * G * 16, coupons = E * 256 * 8;
    static constexpr bool keep = weights + tables + coupons <= 48 * 1024;   // the default limit
    static constexpr int bytes = weights + tables + (keep ? coupons : 0);
    static_assert(bytes <= 48 * 1024, "portfolio weights exceed the default shared-memory limit");
};

template <int E, int C, int CS, int G, int NPB>
__global__ void __launch_bounds__(256, NPB == 1 ? 3 : 2) price_kernel(OuterArgs a, PriceShape ps)
{
    using SM = PriceSmem<E, C, G, NPB>;
    constexpr int F = 2 * E - 1 + CS, R = NPB * C;   // rows of weights per economy
    extern __shared__ __align__(16) unsigned char price_smem[];
    f32x2 *w_s = reinterpret_cast<f32x2 *>(price_smem);      // [E][R][2 LV] (-wA, then -wK), doubled
    float4 *tab_s = reinterpret_cast<float4 *>(price_smem + SM::weights);                          // [E][LV]
    f32x2 *fix_s = reinterpret_cast<f32x2 *>(price_smem + SM::weights + SM::tables) + threadIdx.x;  // [E], stride 256
    const int tid = threadIdx.x, nthr = blockDim.x, pf0 = (int)blockIdx.z * NPB;
    const size_t M = a.M;
    const int n = c_sim.n, ppp = c_sim.ppp;
    const int p = (int)blockIdx.y / ps.splits, part = (int)blockIdx.y % ps.splits;
    const int jp = p * ppp + 1 + part * ps.dates_per_block, j0 = max(jp, ps.start + 1);
    const int j1 = min(min(jp + ps.dates_per_block, (p + 1) * ppp + 1), n + 1);   // dates [j0, j1)
    if (j0 >= j1 && blockIdx.y > 0) return;
    const uint32_t k0 = blockIdx.x * 2u * (uint32_t)nthr + (uint32_t)tid, k1 = k0 + (uint32_t)nthr;
    const bool live0 = k0 < a.M, live1 = k1 < a.M;
    const uint32_t r0 = live0 ? k0 : 0u, r1 = live1 ? k1 : r0;   // paths read
    auto store = [&](int j, int row, float2 mt, float2 ex) {     // row = pb C + c
        const size_t o = ((size_t)((pf0 + row / C) * (n + 1) + j) * C + row % C) * M;
        if (live0) a.expo[o + k0] = ex.x;
        if (live1) a.expo[o + k1] = ex.y;
        if (a.mtm) {
            if (live0) a.mtm[o + k0] = mt.x;
            if (live1) a.mtm[o + k1] = mt.y;
        }
    };
    if (blockIdx.y == 0)   // no default at t_0: exposures of date 0 are never used
        for (int row = 0; row < R; ++row) store(0, row, make_float2(0.f, 0.f), make_float2(0.f, 0.f));

    with_live<G>(p < G ? G - p : 0, [&](auto lv_) {
        constexpr int LV = decltype(lv_)::value;
        if constexpr (LV == 0) {   // every swap has matured
            for (int j = j0; j < j1; ++j)
                for (int row = 0; row < R; ++row) store(j, row, make_float2(0.f, 0.f), make_float2(0.f, 0.f));
            return;
        } else {
            constexpr int P0 = G - LV;   // = p
            for (int i = tid; i < E * R * 2 * LV; i += nthr) {
                const int q = i % (2 * LV), row = i / (2 * LV) % R, e = i / (2 * LV * R);
                const int wrow = ((pf0 * C + row) * E + e) * G + P0;
                const float w = q < LV ? __ldg(a.w_glob + wrow + q) : __ldg(a.w_glob + kMaxW + wrow + q - LV);
                w_s[i] = pack2(-w, -w);
            }
            const float *ffix = a.features + (size_t)(p * ppp) * F * M;   // state at the last reset
            const float2 *fx = a.fix + (size_t)p * E;
            // 1/ZC_{t_-}(t_+) - 1 of economy e
            auto coupon = [&](int e) {
                const float2 f2 = __ldg(fx + e);
                const float *f = ffix + (size_t)e * M;
                return pack2(expm1f(fmaf(f2.y, __ldg(f + r0), -f2.x)), expm1f(fmaf(f2.y, __ldg(f + r1), -f2.x)));
            };
            if (SM::keep) {
#pragma unroll 2
                for (int e = 0; e < E; ++e) fix_s[e * 256] = coupon(e);
            }
            for (int j = j0; j < j1; ++j) {
                __syncthreads();   // the weights, and every warp is done with the last date's tables
                for (int i = tid; i < E * LV; i += nthr) tab_s[i] = __ldg(a.zc + ((size_t)j * E + i / LV) * G + P0 + i % LV);
                const float *fe = a.features + (size_t)j * F * M;
                const float4 *tab = tab_s;
                f32x2 mt[R];
#pragma unroll
                for (int i = 0; i < R; ++i) mt[i] = pack2(0.f, 0.f);
                const float *dj = a.disc + (size_t)j * M;
                const float beta0 = expf(-__ldg(dj + r0)), beta1 = expf(-__ldg(dj + r1));
                float re0 = __ldg(fe + r0), re1 = __ldg(fe + r1);
                float lc0 = 0.f, lc1 = 0.f;
                const f32x2 *w = w_s;
                if (j + 1 < j1) {   // the next date's states, so that its loads find them in the L2 cache
                    prefetch_state<E>(fe + (size_t)F * M, dj + M, M, k0 & ~31u, a.M);
                    prefetch_state<E>(fe + (size_t)F * M, dj + M, M, k1 & ~31u, a.M);
                }
                __syncthreads();
#pragma unroll 1
                for (int e = 0; e < E; ++e, tab += LV, w += R * 2 * LV) {
                    // bond prices Z[g] = ZC_t((p + g + 1) delta) of the live reset dates, chained
                    // from the first: Z[g] = Z[g-1] (1 + expm1(x_g)), x_g = ln ZC_t of this date
                    // - ln ZC_t of the one before. D[g] = ZC_t of the date before - Z[g] = -Z[g-1]
                    // expm1(x_g) keeps full relative accuracy; D[0] carries the running floating
                    // coupon ZC_t(t_+) (1/ZC_{t_-}(t_+) - 1). X holds -D, then Z.
                    f32x2 X[2 * LV];
                    const float2 fm = unpack2(SM::keep ? fix_s[e * 256] : coupon(e));
                    const float4 tp = tab[0];
                    const float z0 = expf(fmaf(-tp.y, re0, tp.x)), z1 = expf(fmaf(-tp.y, re1, tp.x));
                    X[0] = pack2(-(z0 * fm.x), -(z1 * fm.y));
                    X[LV] = pack2(z0, z1);
                    const f32x2 re = pack2(re0, re1);
                    const f32x2 chi = e == 0 ? pack2(1.f, 1.f) : pack2(expf(lc0), expf(lc1));
                    if (e + 1 < E) {   // the next economy's state, ahead of this one's products
                        fe += M;
                        re0 = __ldg(fe + r0);
                        re1 = __ldg(fe + r1);
                        lc0 = __ldg(fe + (size_t)(E - 1) * M + r0);
                        lc1 = __ldg(fe + (size_t)(E - 1) * M + r1);
                    }
#pragma unroll
                    for (int g = 1; g < LV; ++g) {
                        const float4 t4 = tab[g];
                        const f32x2 em = expm1_small2(fma2(pack2(-t4.w, -t4.w), re, pack2(t4.z, t4.z)));
                        X[g] = mul2(X[LV + g - 1], em);
                        X[LV + g] = fma2(X[LV + g - 1], em, X[LV + g - 1]);
                    }
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        f32x2 acc = pack2(0.f, 0.f);
#pragma unroll
                        for (int q = 0; q < 2 * LV; q += 2) {
                            const ulonglong2 w2 = *reinterpret_cast<const ulonglong2 *>(w + i * 2 * LV + q);
                            acc = fma2(w2.x, X[q], acc);
                            acc = fma2(w2.y, X[q + 1], acc);
                        }
                        mt[i] = fma2(chi, acc, mt[i]);
                    }
                }
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const float2 m = unpack2(mt[i]);
                    const float l = c_sim.lgd[i % C];
                    store(j, i, m, make_float2(l * beta0 * fmaxf(m.x, 0.f), l * beta1 * fmaxf(m.y, 0.f)));
                }
            }
        }
    });
}

#include "price_tc.cuh"

}  // namespace
}  // namespace cva

#include "adjoint.cuh"

namespace cva {
namespace {

// Constant-memory ownership of this translation unit: a launch for another
// simulation re-uploads the tables, and every launch first waits for the
// previous one (on whichever stream) before constant memory can change.
static std::mutex t_const_mu;
static const Sim *t_owner[64] = {};
static cudaEvent_t t_last[64] = {};

static cudaError_t upload_consts(const Sim &s, cudaStream_t st)
{
    cudaError_t e = cudaMemcpyToSymbolAsync(c_sim, s.d_const_img, sizeof(SimConsts), 0, cudaMemcpyDeviceToDevice, st);
#ifdef CVA_CONST_WEIGHTS
    if (e == cudaSuccess)
        e = cudaMemcpyToSymbolAsync(c_w, s.d_const_img + sizeof(SimConsts), sizeof(SimWeights), 0,
                                    cudaMemcpyDeviceToDevice, st);
#endif
    return e;
}

static void outer_forget(const Sim *s)
{
    std::lock_guard<std::mutex> lk(t_const_mu);
    for (auto &o : t_owner)
        if (o == s) o = nullptr;
}

// a period's dates share one block's weights; they are split while `blocks` blocks do not
// fill the chip four times
static PriceShape price_shape(uint64_t blocks, int ppp, int sms)
{
    PriceShape ps = {ppp, 1, 0};
    while (blocks * ps.splits < 4u * (unsigned)sms && ps.dates_per_block > 1) {
        ps.dates_per_block = (ps.dates_per_block + 1) / 2;
        ps.splits = (ppp + ps.dates_per_block - 1) / ps.dates_per_block;
    }
    return ps;
}

template <int E, int C, int CS, int G, int NPF>
cva_status outer_launch(Sim &s, uint64_t seed, uint64_t k0, cudaStream_t st)
{
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    OuterArgs args = {};
    args.M = (uint32_t)s.M;
    args.k0 = (uint32_t)k0;
    args.seed_lo = (uint32_t)seed;
    args.start = s.start_date;
    args.save_date = s.save_date;
    args.ckpt = s.d_ckpt;
    args.ckpt_I0 = reinterpret_cast<double *>(s.d_ckpt + 2 * (size_t)C * s.M);
    args.branch_step = s.branch_date <= s.n ? s.branch_date * s.S : INT_MAX;
    args.branch = s.branch;
    args.seed_hi = (uint32_t)(seed >> 32);
    args.zc = s.d_zc;
    args.fix = s.d_fix;
    args.drift = s.d_drift;
    args.features = s.d_features;
    args.disc = s.d_disc;
    args.thr = s.d_thr;
    args.expo = s.d_expo;
    args.mtm = s.d_mtm;
    args.w_glob = reinterpret_cast<const float *>(s.d_const_img + sizeof(SimConsts));
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CVA_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    std::lock_guard<std::mutex> lk(t_const_mu);
    if (capturing) {
        // a captured graph uploads its own tables every time it runs
        CVA_CUDA_TRY(upload_consts(s, st));
        t_owner[dev] = nullptr;
    } else {
        if (!t_last[dev]) CVA_CUDA_TRY(cudaEventCreateWithFlags(&t_last[dev], cudaEventDisableTiming));
        else CVA_CUDA_TRY(cudaStreamWaitEvent(st, t_last[dev], 0));
        if (t_owner[dev] != &s) {
            CVA_CUDA_TRY(upload_consts(s, st));
            t_owner[dev] = &s;
        }
    }
    const unsigned pb = (unsigned)(s.tune_price_block > 0 && s.tune_price_block <= 256 ? s.tune_price_block : 256);
    int sms = 0;
    CVA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const bool four = s.tune_sim_block == 64;
    if (s.start_date > 0 || s.save_date >= 0) launch_sim<E, C, CS, SimMode::restart>(args, four, sms, st);
    else launch_sim<E, C, CS, SimMode::plain>(args, four, sms, st);
    CVA_CUDA_TRY(cudaGetLastError());
    if (s.ev[1]) CVA_CUDA_TRY(cudaEventRecord(s.ev[1], st));
    if (s.tune_price_pf == 4) {   // every portfolio per 128-path tile on the tensor cores
        constexpr int bytes = price_tc_bytes<E, NPF, C, G>();
        static bool attr[64] = {};
        if (!attr[dev]) {
            if (capturing) return fail(CVA_EINVAL, "price: run once before capturing (kernel attribute)");
            CVA_CUDA_TRY(cudaFuncSetAttribute(price_tc_kernel<E, C, CS, G, NPF>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
            attr[dev] = true;
        }
        // at least six path tiles per slot and part of a period, so that the last round of
        // tiles is a small part of them; at most kPriceTcDates dates, whose tables a block keeps
        const uint32_t tiles = (args.M + 127u) / 128u, slots = (uint32_t)sms * kPriceSlots;
        const unsigned periods = (unsigned)((s.n + s.ppp - 1) / s.ppp);
        PriceShape ps = {s.ppp, 1, s.start_date};
        while (ps.dates_per_block > kPriceTcDates ||
               ((uint64_t)tiles * ps.splits < 6ull * slots && ps.dates_per_block > 1)) {
            ps.dates_per_block = (ps.dates_per_block + 1) / 2;
            ps.splits = (s.ppp + ps.dates_per_block - 1) / ps.dates_per_block;
        }
        const dim3 tgrid(std::min((tiles + kPriceSlots - 1) / kPriceSlots, (uint32_t)sms), periods * (unsigned)ps.splits);
        price_tc_kernel<E, C, CS, G, NPF><<<tgrid, 128 * kPriceSlots, bytes, st>>>(args, tiles, ps);
        CVA_CUDA_TRY(cudaGetLastError());
        if (!capturing) CVA_CUDA_TRY(cudaEventRecord(t_last[dev], st));
        return CVA_OK;
    }
    // portfolios per block: as set, or (0) the largest of 3, 2, 1 that divides their number
    // (bond prices are computed once per block)
    const int ppb = s.tune_price_pf ? (NPF % s.tune_price_pf == 0 ? s.tune_price_pf : 1)
                                    : (NPF % 3 == 0 ? 3 : NPF % 2 == 0 ? 2 : 1);
    const unsigned tiles = (args.M + 2 * pb - 1) / (2 * pb), periods = (unsigned)((s.n + s.ppp - 1) / s.ppp);
    PriceShape ps = price_shape((uint64_t)tiles * periods * (NPF / ppb), s.ppp, sms);
    ps.start = s.start_date;
    const dim3 pgrid(tiles, periods * (unsigned)ps.splits, (unsigned)(NPF / ppb));
    if constexpr (NPF % 3 == 0) {
        if (ppb == 3) price_kernel<E, C, CS, G, 3><<<pgrid, pb, PriceSmem<E, C, G, 3>::bytes, st>>>(args, ps);
    }
    if constexpr (NPF % 2 == 0) {
        if (ppb == 2) price_kernel<E, C, CS, G, 2><<<pgrid, pb, PriceSmem<E, C, G, 2>::bytes, st>>>(args, ps);
    }
    if (ppb == 1) price_kernel<E, C, CS, G, 1><<<pgrid, pb, PriceSmem<E, C, G, 1>::bytes, st>>>(args, ps);
    CVA_CUDA_TRY(cudaGetLastError());
    if (!capturing) CVA_CUDA_TRY(cudaEventRecord(t_last[dev], st));
    return CVA_OK;
}

// The adjoint of one range of paths; `b` holds the tables, the scratch and the sums that
// this range adds. Without scratch only its size is computed, nothing launched.
template <int E, int C, int CS, int G>
cva_status adjoint_launch(Sim &s, AdjBuffers &b, uint64_t seed, uint64_t k0, uint32_t M, cudaStream_t st)
{
    // (the run-time shapes' limits, kept here so that what a call takes does not depend on the shape)
    constexpr int KMAX = 16, SMAX = 4, F = 2 * E - 1 + CS, NPAR = 3 * E - 1 + 3 * C;
    if (b.K < 1 || b.K > KMAX || s.S > SMAX) return fail(CVA_ENOTSUP, "adjoint: checkpoint interval <= 16, sub-steps <= 4");
    int dev = 0, sms = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    CVA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t n = s.n, q = n * s.S, Mz = M;
    const unsigned tiles = (M + 255u) / 256u, periods = (unsigned)((s.n + s.ppp - 1) / s.ppp), rblocks = (M + 31u) / 32u;
    const PriceShape ps = price_shape((uint64_t)tiles * periods, s.ppp, sms);
    const size_t pblocks = (size_t)tiles * periods * ps.splits;
    // scratch: the block sums (FP64), then the arrays of the range
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) / 256 * 256;
        return b.scratch ? b.scratch + at : nullptr;
    };
    AdjSplitArgs a = {};
    a.part_p = reinterpret_cast<double *>(take(pblocks * (2 * E + 1) * 8));
    auto take_rev = [&](size_t bytes) { return b.forward_only ? nullptr : take(bytes); };   // the reverse sweep's
    a.part_r = reinterpret_cast<double *>(take_rev((size_t)rblocks * NPAR * 8));
    float *features = reinterpret_cast<float *>(take((n + 1) * F * Mz * 4));
    float *disc = reinterpret_cast<float *>(take((n + 1) * Mz * 4));
    float *surv = reinterpret_cast<float *>(take((n + 1) * C * Mz * 4));
    float *inc = reinterpret_cast<float *>(take_rev(q * F * Mz * 4));
    float *gpre = reinterpret_cast<float *>(take_rev(q * C * Mz * 4));
    a.V = reinterpret_cast<float *>(take_rev((n + 1) * C * Mz * 4));
    a.rbin = reinterpret_cast<float *>(take_rev(n * E * Mz * 4));
    a.lbin = reinterpret_cast<float *>(take_rev(n * E * Mz * 4));
    a.ibin = reinterpret_cast<float *>(take_rev(n * Mz * 4));
    a.fixin = reinterpret_cast<float *>(take_rev((size_t)periods * ps.splits * E * Mz * 4));
    if (!b.scratch) {
        b.scratch_bytes = off;
        return CVA_OK;
    }
    if (off > b.scratch_bytes) return fail(CVA_ENOMEM, "adjoint: scratch too small");
    a.M = M;
    a.zc = s.d_zc;
    a.fix = s.d_fix;
    a.dzc = b.dzc;
    a.dfix = b.dfix;
    a.ddrift = b.ddrift;
    a.rho = b.rho;
    a.sig = b.sig;
    a.w_glob = reinterpret_cast<const float *>(s.d_const_img + sizeof(SimConsts));
    a.features = features;
    a.disc = disc;
    a.surv = surv;
    a.inc = inc;
    a.gpre = gpre;
    OuterArgs o = {};
    o.M = M;
    o.k0 = (uint32_t)k0;
    o.seed_lo = (uint32_t)seed;
    o.seed_hi = (uint32_t)(seed >> 32);
    o.branch_step = INT_MAX;
    o.drift = s.d_drift;
    o.features = features;
    o.disc = disc;
    o.thr = surv;
    o.inc = inc;
    o.gpre = gpre;
    std::lock_guard<std::mutex> lk(t_const_mu);
    if (!t_last[dev]) CVA_CUDA_TRY(cudaEventCreateWithFlags(&t_last[dev], cudaEventDisableTiming));
    else CVA_CUDA_TRY(cudaStreamWaitEvent(st, t_last[dev], 0));
    if (t_owner[dev] != &s) {
        CVA_CUDA_TRY(upload_consts(s, st));
        t_owner[dev] = &s;
    }
    if (b.forward_only) launch_sim<E, C, CS, SimMode::forward>(o, false, sms, st);
    else launch_sim<E, C, CS, SimMode::adjoint>(o, false, sms, st);
    CVA_CUDA_TRY(cudaGetLastError());
    const dim3 pgrid(tiles, periods * (unsigned)ps.splits);
    // weights, fixing adjoints, coupons, tables, parameter adjoints
    constexpr size_t psmem = (size_t)E * C * 2 * G * 8 + (size_t)E * 128 * (8 + 8 + 16) + 2 * (size_t)E * G * 16;
    static_assert(3 * (psmem + 2048) <= 227 * 1024, "adjoint pricing: three blocks a multiprocessor");
    for (auto kern : {adj_price_kernel<E, C, CS, G, false>, adj_price_kernel<E, C, CS, G, true>})
        CVA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem));
    if (b.forward_only) {
        adj_price_kernel<E, C, CS, G, false><<<pgrid, 128, psmem, st>>>(a, ps);
        CVA_CUDA_TRY(cudaGetLastError());
    } else {
        adj_price_kernel<E, C, CS, G, true><<<pgrid, 128, psmem, st>>>(a, ps);
        CVA_CUDA_TRY(cudaGetLastError());
        adj_reverse_kernel<E, C, CS, 8><<<rblocks, 256, 0, st>>>(a, ps.splits);
        CVA_CUDA_TRY(cudaGetLastError());
    }
    CVA_CUDA_TRY(cudaEventRecord(t_last[dev], st));
    // the range's sums: [2E + 1] of the pricing, then [NPAR] of the recursions
    cva_status r = sum_columns_fp64(a.part_p, (int)pblocks, 2 * E + 1, b.sum, st);
    if (r == CVA_OK && !b.forward_only) r = sum_columns_fp64(a.part_r, (int)rblocks, NPAR, b.sum + 2 * E + 1, st);
    return r;
}

}  // namespace
}  // namespace cva
