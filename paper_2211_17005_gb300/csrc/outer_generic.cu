// Outer-path kernels for any model shape within the library's limits (E <= 16
// economies, C <= 16 counterparties with CIR and constant intensities in any order,
// up to 6 portfolios), the model's sizes run-time values. The block layout is the compiled
// kernels': 32 paths and eight warps with the factors split over them for the simulation, a
// period's dates and two paths per thread for the pricing. The arithmetic, and its order, is
// that of sim_kernel and price_kernel (outer.cuh), so a shape that also has a
// compiled instantiation gives the same bits on either; the compiled ones stay the
// fast paths. The stochastic intensity of counterparty c is state factor
// c_sim.gpos[c] (the factors are r^0..r^{E-1}, log chi^1..log chi^{E-1}, then the
// CIR intensities in counterparty order), or -1 for a constant intensity.
// Three economies, five counterparties, four portfolios, 20011 paths, 40 dates: simulation
// 177 us and pricing 273 us with a thread per path and per (path, date, portfolio), now 68 and
// 80 us.
#include <atomic>

#define CVA_CONST_WEIGHTS
#include "outer.cuh"

namespace cva {
namespace {

constexpr int kGenSteps = 8;            // fine steps at a time of the simulation
constexpr int kGenPriceThreads = 128;
static_assert(kMaxE <= 16 && kMaxC <= 16, "eight warps hold two factors each");

// NW warps per 32 paths, at most two economies and two counterparties a warp.
template <int NW>
__global__ void __launch_bounds__(32 * NW) sim_generic_kernel(OuterArgs a)
{
    constexpr int NS = kGenSteps, ME = 2, MC = 2;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t kl = blockIdx.x * 32u + (uint32_t)lane;
    const bool live = kl < a.M;
    const uint32_t k = a.k0 + kl;
    const size_t M = a.M;
    const int E = c_sim.E, C = c_sim.C, F = c_sim.F, n = c_sim.n, S = c_sim.S, NB = (F + 3) / 4, FR = 4 * NB;
    const float ds = c_sim.ds;
    const double ds_d = c_sim.ds_d;
    float *Ws = reinterpret_cast<float *>(smem);        // [NS][4 NB][32] normals, then increments
    float *R0 = Ws + NS * FR * 32;                      // [NS][32]

    float r0 = c_sim.r0[0], r[ME], lchi[ME], gam[MC], lam[MC], lamc[MC];
    int gp_[MC];
    double I0 = 0.0;
#pragma unroll
    for (int i = 0; i < ME; ++i) {
        const int e = min(warp + NW * i, E - 1);
        r[i] = c_sim.r0[e];
        lchi[i] = c_sim.lchi0[e];
    }
#pragma unroll
    for (int i = 0; i < MC; ++i) {
        const int c = min(warp + NW * i, C - 1);
        gam[i] = c_sim.gamma0[c];
        gp_[i] = c_sim.gpos[c];
        lam[i] = lamc[i] = 0.f;
    }
    auto write_date = [&](int j) {
        if (!live) return;
        float *fe = a.features + (size_t)j * F * M + kl;
#pragma unroll
        for (int i = 0; i < ME; ++i) {
            const int e = warp + NW * i;
            if (e >= E) break;
            fe[(size_t)e * M] = r[i];
            if (e > 0) fe[(size_t)(E - 1 + e) * M] = lchi[i];
        }
#pragma unroll
        for (int i = 0; i < MC; ++i) {
            const int c = warp + NW * i;
            if (c >= C) break;
            if (gp_[i] >= 0) fe[(size_t)gp_[i] * M] = gam[i];
            a.thr[((size_t)j * C + c) * M + kl] = -expm1f(-lam[i]);   // 0 at date 0
        }
    };
    write_date(0);
    if (warp == NW - 1 && live) a.disc[kl] = 0.f;

    const int steps = n * S;
    int j = 0, s = 0, jd = 0, sd = 0;
    for (int q0 = 0; q0 < steps; q0 += NS) {
        for (int v = warp; v < NS && q0 + v < steps; v += NW) {   // the increments W = L z of a step, in place of the normals
            const int q = q0 + v;
            float *w = Ws + v * FR * 32 + lane;
            for (int b = 0; b < NB; ++b) {
                const uint4 x = philox4x32_10(make_uint4(k, (uint32_t)q, q >= a.branch_step ? a.branch : 0u,
                                                         (kStreamOuter << 24) | (uint32_t)b),
                                              a.seed_lo, a.seed_hi);
                float z[4];
                box_muller(x.x, x.y, z[0], z[1]);
                box_muller(x.z, x.w, z[2], z[3]);
#pragma unroll
                for (int t = 0; t < 4; ++t) w[(4 * b + t) * 32] = z[t];
            }
            for (int i = F - 1; i >= 0; --i) {   // row i needs the normals 0..i only
                const float *L = c_sim.L + i * (i + 1) / 2;
                float acc = 0.f;
#pragma unroll 4
                for (int col = 0; col <= i; ++col) acc = fmaf(L[col], w[col * 32], acc);
                w[i * 32] = acc;
            }
        }
        __syncthreads();
        const int chunk = min(NS, steps - q0);
        for (int u = 0; u < chunk; ++u) {
            const float *W = Ws + u * FR * 32 + lane;
            const float *drow = a.drift + (size_t)(q0 + u) * E;
            if (warp == 0) R0[u * 32 + lane] = r0;
            // Lambda^c: left-point integral, compensated FP32, non-decreasing
#pragma unroll
            for (int i = 0; i < MC; ++i) {
                const int c = warp + NW * i;
                if (c >= C) break;
                const float gp = fmaxf(gam[i], 0.f);
                const float y = fmaf(gp, ds, -lamc[i]);
                const float t = lam[i] + y;
                lamc[i] = (t - lam[i]) - y;
                lam[i] = fmaxf(t, lam[i]);
                if (gp_[i] >= 0)
                    gam[i] += c_sim.cir_ktds[c] - c_sim.cir_kds[c] * gp + c_sim.cir_nu_sqds[c] * sqrtf(gp) * W[gp_[i] * 32];
            }
#pragma unroll
            for (int i = 0; i < ME; ++i) {
                const int e = warp + NW * i;
                if (e >= E) break;
                if (e > 0)
                    lchi[i] += fmaf(r0 - r[i], ds, c_sim.fx_drift_ds[e]) + c_sim.fx_sig_sqds[e] * W[(E - 1 + e) * 32];
                r[i] += (__ldg(drow + e) - c_sim.hw_a_ds[e] * r[i]) + c_sim.hw_sig_sqds[e] * W[e * 32];
            }
            r0 += (__ldg(drow) - c_sim.hw_a_ds[0] * r0) + c_sim.hw_sig_sqds[0] * W[0];
            if (++s == S) {
                s = 0;
                write_date(++j);
            }
        }
        __syncthreads();   // the increments are read before the next steps overwrite them
        if (warp == NW - 1)   // int r^0 in FP64, left points: one warp for the narrow FP64 pipe
            for (int u = 0; u < chunk; ++u) {
                I0 = fma((double)R0[u * 32 + lane], ds_d, I0);
                if (++sd == S) {
                    sd = 0;
                    ++jd;
                    if (live) a.disc[(size_t)jd * M + kl] = (float)I0;
                }
            }
    }
}

// price_kernel with run-time sizes: two paths per thread in packed pairs, a period's dates
// per block and the instantiation for its live reset dates, NPB portfolios from pf0 =
// blockIdx.z NPB. The MtM sums live in shared memory, [row][thread] (their number is not
// known at compile time), the weights as in price_kernel. Same order of operations, so a
// shape with a compiled kernel gives its bits.
__global__ void __launch_bounds__(kGenPriceThreads, 4) price_generic_kernel(OuterArgs a, PriceShape ps, int NPB)
{
    constexpr int NT = kGenPriceThreads;
    extern __shared__ __align__(16) unsigned char smem[];
    const int E = c_sim.E, C = c_sim.C, F = c_sim.F, G = c_sim.G, n = c_sim.n, ppp = c_sim.ppp;
    const int tid = threadIdx.x, pf0 = (int)blockIdx.z * NPB, R = min(NPB, c_sim.NPF - pf0) * C;
    f32x2 *mt_s = reinterpret_cast<f32x2 *>(smem) + tid;         // [NPB C], stride NT
    f32x2 *w_s = reinterpret_cast<f32x2 *>(smem) + NPB * C * NT;  // [E][R][2 LV] (-wA, -wK), doubled
    const size_t M = a.M;
    const int p = (int)blockIdx.y / ps.splits, part = (int)blockIdx.y % ps.splits;
    const int j0 = p * ppp + 1 + part * ps.dates_per_block;
    const int j1 = min(min(j0 + ps.dates_per_block, (p + 1) * ppp + 1), n + 1);   // dates [j0, j1)
    const uint32_t k0 = blockIdx.x * 2u * NT + (uint32_t)tid, k1 = k0 + NT;
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
    const float2 zero = make_float2(0.f, 0.f);
    if (blockIdx.y == 0)   // no default at t_0: exposures of date 0 are never used
        for (int row = 0; row < R; ++row) store(0, row, zero, zero);
    with_live<kMaxG>(p < G ? G - p : 0, [&](auto lv_) {
        constexpr int LV = decltype(lv_)::value;
        if constexpr (LV == 0) {   // every swap has matured
            for (int j = j0; j < j1; ++j)
                for (int row = 0; row < R; ++row) store(j, row, zero, zero);
        } else {
            for (int i = tid; i < E * R * 2 * LV; i += NT) {
                const int q = i % (2 * LV), row = i / (2 * LV) % R, e = i / (2 * LV * R);
                const int wrow = ((pf0 * C + row) * E + e) * G + p;
                const float w = q < LV ? __ldg(a.w_glob + wrow + q) : __ldg(a.w_glob + kMaxW + wrow + q - LV);
                w_s[i] = pack2(-w, -w);
            }
            __syncthreads();
            const float *ffix = a.features + (size_t)(p * ppp) * F * M;   // state at the last reset
            const float2 *fx = a.fix + (size_t)p * E;
            for (int j = j0; j < j1; ++j) {
                const float *fe = a.features + (size_t)j * F * M;
                const float4 *tab = a.zc + (size_t)j * E * G + p;
                const float *dj = a.disc + (size_t)j * M;
                const float beta0 = expf(-__ldg(dj + r0)), beta1 = expf(-__ldg(dj + r1));
                for (int e = 0; e < E; ++e, tab += G) {
                    // bond prices of the live reset dates (price_kernel): X holds -D, then Z
                    f32x2 X[2 * LV];
                    const float re0 = __ldg(fe + (size_t)e * M + r0), re1 = __ldg(fe + (size_t)e * M + r1);
                    const float rf0 = __ldg(ffix + (size_t)e * M + r0), rf1 = __ldg(ffix + (size_t)e * M + r1);
                    const float *lc = fe + (size_t)(E - 1 + (e > 0 ? e : 1)) * M;
                    const f32x2 chi = e == 0 ? pack2(1.f, 1.f) : pack2(expf(__ldg(lc + r0)), expf(__ldg(lc + r1)));
                    const float2 f2 = __ldg(fx + e);
                    const float4 tp = __ldg(tab);
                    const float z0 = expf(fmaf(-tp.y, re0, tp.x)), z1 = expf(fmaf(-tp.y, re1, tp.x));
                    X[0] = pack2(-(z0 * expm1f(fmaf(f2.y, rf0, -f2.x))), -(z1 * expm1f(fmaf(f2.y, rf1, -f2.x))));
                    X[LV] = pack2(z0, z1);
                    const f32x2 re = pack2(re0, re1);
#pragma unroll
                    for (int g = 1; g < LV; ++g) {
                        const float4 t4 = __ldg(tab + g);
                        const f32x2 em = expm1_small2(fma2(pack2(-t4.w, -t4.w), re, pack2(t4.z, t4.z)));
                        X[g] = mul2(X[LV + g - 1], em);
                        X[LV + g] = fma2(X[LV + g - 1], em, X[LV + g - 1]);
                    }
                    const f32x2 *w = w_s + e * R * 2 * LV;
#pragma unroll 2
                    for (int i = 0; i < R; ++i) {
                        f32x2 acc = pack2(0.f, 0.f);
#pragma unroll
                        for (int q = 0; q < 2 * LV; q += 2) {
                            const ulonglong2 w2 = *reinterpret_cast<const ulonglong2 *>(w + i * 2 * LV + q);
                            acc = fma2(w2.x, X[q], acc);
                            acc = fma2(w2.y, X[q + 1], acc);
                        }
                        mt_s[i * NT] = fma2(chi, acc, e == 0 ? pack2(0.f, 0.f) : mt_s[i * NT]);
                    }
                }
                for (int i = 0; i < R; ++i) {
                    const float2 m = unpack2(mt_s[i * NT]);
                    const float l = c_sim.lgd[i % C];
                    store(j, i, m, make_float2(l * beta0 * fmaxf(m.x, 0.f), l * beta1 * fmaxf(m.y, 0.f)));
                }
            }
        }
    });
}

// ---- adjoint of the smooth CVA_0 for run-time shapes ----
// One thread per path: a forward sweep with checkpoints every K dates, then segment by segment
// from the last a recompute and the reverse of the pricing and of the Euler sub-steps. The
// functional and its derivatives are those of adjoint.cuh, whose kernels add in another
// order. The stochastic intensity of counterparty c
// is state factor c_sim.gpos[c] (-1: constant, whose kappa, theta, nu receive
// nothing). Per-thread arrays are sized at the library's limits (local memory); the
// parameter adjoints live in dynamic shared memory, NPAR x 128 floats.
constexpr int kAdjKMax = 16, kAdjSMax = 4;

struct AdjArgs {
    uint32_t M, k0, seed_lo, seed_hi;
    int K, nseg;
    int forward_only;                   // 1: the smooth CVA_0 of the forward sweep only
    const float4 *__restrict__ zc;      // [n+1][E][G] (lnA, B, dlnA, dB)
    const float2 *__restrict__ fix;     // [periods+1][E] (lnA, B)
    const int *__restrict__ date_p;     // [n+1]
    const float *__restrict__ drift;    // [n*S][E]
    const float4 *__restrict__ dzc;     // [n+1][E][G] d/df, d/dsigma of (lnA, dlnA)
    const float2 *__restrict__ dfix;    // [periods+1][E] d/df, d/dsigma of lnA at the fixing
    const float2 *__restrict__ ddrift;  // [n*S][E] d drift/df, d drift/dsigma^r (quanto included)
    const float *__restrict__ rho;      // [E] correlation of r^e and log chi^e (entry 0 unused)
    const float *__restrict__ sig;      // [E] sigma^r, [E] sigma^chi, [C] kappa, [C] theta, [C] nu
    float *ckpt;                        // [nseg][2E+3C][M]
    double *ckpt_I0;                    // [nseg][M]
    float *fixr;                        // [periods+1][E][M]
    double *part;                       // [blocks][npar + 1]
};

// bond prices Z and their differences D (and the expm1 factors EM) of economy e at
// date j for one path: the chained form of price_kernel
__device__ __forceinline__ void bonds_generic(const AdjArgs &a, int j, int e, int p, float re, float fixm1,
                                              float (&Z)[kMaxG], float (&D)[kMaxG], float (&EM)[kMaxG])
{
    const int E = c_sim.E, G = c_sim.G;
    const float4 *tab = a.zc + ((size_t)j * E + e) * G;
    const float4 tp = __ldg(tab + (p < G ? p : G - 1));
    const float z_first = expf(fmaf(-tp.y, re, tp.x));
    for (int g = 0; g < G; ++g) {
        EM[g] = 0.f;
        if (g < p) {
            Z[g] = 0.f;
            D[g] = 0.f;
        } else if (g == p) {
            Z[g] = z_first;
            D[g] = z_first * fixm1;
        } else {
            const float4 t4 = __ldg(tab + g);
            const float zp = Z[g > 0 ? g - 1 : 0];
            const float em = expm1_small(fmaf(-t4.w, re, t4.z));
            EM[g] = em;
            D[g] = -zp * em;
            Z[g] = fmaf(zp, em, zp);
        }
    }
}

// correlated increments W = L z of fine step q for path k
__device__ __forceinline__ void increments_generic(const AdjArgs &a, uint32_t k, uint32_t q, float (&W)[kMaxF])
{
    const int F = c_sim.F, NB = (F + 3) / 4;
    for (int i = 0; i < F; ++i) W[i] = 0.f;
    for (int b = 0; b < NB; ++b) {
        const uint4 x = philox4x32_10(make_uint4(k, q, 0u, (kStreamOuter << 24) | (uint32_t)b), a.seed_lo, a.seed_hi);
        float z[4];
        box_muller(x.x, x.y, z[0], z[1]);
        box_muller(x.z, x.w, z[2], z[3]);
        for (int t = 0; t < 4; ++t) {
            const int col = 4 * b + t;
            if (col < F)
                for (int i = col; i < F; ++i) W[i] = fmaf(c_sim.L[i * (i + 1) / 2 + col], z[t], W[i]);
        }
    }
}

__global__ void __launch_bounds__(128) adjoint_generic_kernel(AdjArgs a)
{
    const int E = c_sim.E, C = c_sim.C, G = c_sim.G;
    const int NV = 2 * E + 3 * C, NPAR = 3 * E - 1 + 3 * C;
    const int PF = 0, PSR = E, PSX = 2 * E - 1, PK = 3 * E - 1, PT = PK + C, PN = PT + C;
    extern __shared__ float pb_s[];                    // [NPAR][128]
    __shared__ double red_s[128];
    const int tid = threadIdx.x;
    const uint32_t kl = blockIdx.x * blockDim.x + tid;
    const bool active = kl < a.M;
    const uint32_t k = a.k0 + kl;
    const size_t M = a.M;
    const int n = c_sim.n, S = c_sim.S, ppp = c_sim.ppp, K = a.K;
    const float ds = c_sim.ds, sqds = c_sim.sqds;
    const double ds_d = c_sim.ds_d;
    float *pb = pb_s + tid;
    for (int i = 0; i < NPAR; ++i) pb[i * 128] = 0.f;
    double J = 0.0;

    if (active) {
        float r[kMaxE], lchi[kMaxE], gam[kMaxC], lam[kMaxC], lamc[kMaxC], lam_prev[kMaxC];
        float W[kMaxF], Z[kMaxG], D[kMaxG], EM[kMaxG], mt[kMaxC];
        for (int e = 0; e < E; ++e) {
            r[e] = c_sim.r0[e];
            lchi[e] = c_sim.lchi0[e];
        }
        for (int c = 0; c < C; ++c) {
            gam[c] = c_sim.gamma0[c];
            lam[c] = lamc[c] = lam_prev[c] = 0.f;
        }
        double I0 = 0.0;
        // one Euler sub-step of the state (sim_kernel's order)
        auto step = [&](uint32_t q) {
            increments_generic(a, k, q, W);
            const float r0 = r[0];
            I0 = fma((double)r0, ds_d, I0);
            for (int c = 0; c < C; ++c) {
                const float gp = fmaxf(gam[c], 0.f);
                const float y = fmaf(gp, ds, -lamc[c]);
                const float t = lam[c] + y;
                lamc[c] = (t - lam[c]) - y;
                lam[c] = fmaxf(t, lam[c]);
                const int w = c_sim.gpos[c];
                if (w >= 0) gam[c] += c_sim.cir_ktds[c] - c_sim.cir_kds[c] * gp + c_sim.cir_nu_sqds[c] * sqrtf(gp) * W[w];
            }
            const float *drow = a.drift + (size_t)q * E;
            for (int e = 1; e < E; ++e)
                lchi[e] += fmaf(r0 - r[e], ds, c_sim.fx_drift_ds[e]) + c_sim.fx_sig_sqds[e] * W[E - 1 + e];
            for (int e = 0; e < E; ++e) r[e] += (__ldg(drow + e) - c_sim.hw_a_ds[e] * r[e]) + c_sim.hw_sig_sqds[e] * W[e];
        };
        // the MtM of every counterparty at date j from the rates and FX levels given
        auto mtm = [&](int j, int p, const float *rr, const float *ll) {
            for (int c = 0; c < C; ++c) mt[c] = 0.f;
            for (int e = 0; e < E; ++e) {
                const float2 f2 = __ldg(a.fix + (size_t)p * E + e);
                const float fixm1 = expm1f(fmaf(f2.y, a.fixr[((size_t)p * E + e) * M + kl], -f2.x));
                bonds_generic(a, j, e, p, rr[e], fixm1, Z, D, EM);
                const float chi = (e == 0) ? 1.f : expf(ll[e]);
                for (int c = 0; c < C; ++c) {
                    const int base = (c * E + e) * G;
                    float acc = 0.f;
                    for (int h = 0; h < G; ++h) acc = fmaf(c_w.wA[base + h], D[h], acc);
                    for (int g = 0; g < G; ++g) acc = fmaf(-c_w.wK[base + g], Z[g], acc);
                    mt[c] = fmaf(chi, acc, mt[c]);
                }
            }
        };

        // ---------------- forward sweep: checkpoints and fixings ----------------
        for (int j = 0; j <= n; ++j) {
            if (j > 0)
                for (int s = 0; s < S; ++s) step((uint32_t)((j - 1) * S + s));
            if (j % ppp == 0)
                for (int e = 0; e < E; ++e) a.fixr[((size_t)(j / ppp) * E + e) * M + kl] = r[e];
            if (a.forward_only && j > 0) {
                const int p = __ldg(a.date_p + j);
                const float beta = expf(-(float)I0);
                mtm(j, p, r, lchi);
                for (int c = 0; c < C; ++c) {
                    const float V = c_sim.lgd[c] * beta * fmaxf(mt[c], 0.f);
                    J += (double)V * (double)(expf(-lam_prev[c]) - expf(-lam[c]));
                }
            }
            for (int c = 0; c < C; ++c) lam_prev[c] = lam[c];
            if (j % K == 0 && j / K < a.nseg) {
                float *cp = a.ckpt + (size_t)(j / K) * NV * M + kl;
                int v = 0;
                for (int e = 0; e < E; ++e) cp[(size_t)(v++) * M] = r[e];
                for (int e = 0; e < E; ++e) cp[(size_t)(v++) * M] = lchi[e];
                for (int c = 0; c < C; ++c) cp[(size_t)(v++) * M] = gam[c];
                for (int c = 0; c < C; ++c) cp[(size_t)(v++) * M] = lam[c];
                for (int c = 0; c < C; ++c) cp[(size_t)(v++) * M] = lamc[c];
                a.ckpt_I0[(size_t)(j / K) * M + kl] = I0;
            }
        }

        if (!a.forward_only) {
            // ---------------- reverse sweep ----------------
            float rb[kMaxE], lb[kMaxE], rfb[kMaxE], gb[kMaxC], Lb[kMaxC], Vnext[kMaxC], mtb[kMaxC];
            for (int e = 0; e < E; ++e) rb[e] = lb[e] = rfb[e] = 0.f;
            for (int c = 0; c < C; ++c) gb[c] = Lb[c] = Vnext[c] = 0.f;
            float Ib = 0.f;
            float st_g[kAdjKMax * kAdjSMax][kMaxC];
            float dt_r[kAdjKMax + 1][kMaxE], dt_l[kAdjKMax + 1][kMaxE], dt_lam[kAdjKMax + 1][kMaxC];
            double dt_I0[kAdjKMax + 1];
            for (int seg = a.nseg - 1; seg >= 0; --seg) {
                const int d0 = seg * K, d1 = min(d0 + K, n);
                {
                    const float *cp = a.ckpt + (size_t)seg * NV * M + kl;
                    int v = 0;
                    for (int e = 0; e < E; ++e) r[e] = cp[(size_t)(v++) * M];
                    for (int e = 0; e < E; ++e) lchi[e] = cp[(size_t)(v++) * M];
                    for (int c = 0; c < C; ++c) gam[c] = cp[(size_t)(v++) * M];
                    for (int c = 0; c < C; ++c) lam[c] = cp[(size_t)(v++) * M];
                    for (int c = 0; c < C; ++c) lamc[c] = cp[(size_t)(v++) * M];
                    I0 = a.ckpt_I0[(size_t)seg * M + kl];
                }
                for (int e = 0; e < E; ++e) {
                    dt_r[0][e] = r[e];
                    dt_l[0][e] = lchi[e];
                }
                for (int c = 0; c < C; ++c) dt_lam[0][c] = lam[c];
                dt_I0[0] = I0;
                for (int j = d0 + 1; j <= d1; ++j) {
                    for (int s = 0; s < S; ++s) {
                        const int qs = (j - d0 - 1) * S + s;
                        for (int c = 0; c < C; ++c) st_g[qs][c] = gam[c];
                        step((uint32_t)((j - 1) * S + s));
                    }
                    for (int e = 0; e < E; ++e) {
                        dt_r[j - d0][e] = r[e];
                        dt_l[j - d0][e] = lchi[e];
                    }
                    for (int c = 0; c < C; ++c) dt_lam[j - d0][c] = lam[c];
                    dt_I0[j - d0] = I0;
                }

                for (int j = d1; j > d0; --j) {
                    const int jj = j - d0;
                    const int p = __ldg(a.date_p + j);
                    const float beta = expf(-(float)dt_I0[jj]);
                    mtm(j, p, dt_r[jj], dt_l[jj]);
                    // ---- survival terms and exposure adjoints ----
                    for (int c = 0; c < C; ++c) {
                        const float V = c_sim.lgd[c] * beta * fmaxf(mt[c], 0.f);
                        const float Sp = expf(-dt_lam[jj - 1][c]), Sc = expf(-dt_lam[jj][c]);
                        J += (double)V * (double)(Sp - Sc);
                        const float Vb = Sp - Sc;
                        Lb[c] += Sc * (V - Vnext[c]);
                        Vnext[c] = V;
                        mtb[c] = mt[c] > 0.f ? Vb * c_sim.lgd[c] * beta : 0.f;
                        Ib -= Vb * V;
                    }
                    // ---- pricing at t_j: reverse, economy by economy ----
                    for (int e = 0; e < E; ++e) {
                        const float re = dt_r[jj][e];
                        const float2 f2 = __ldg(a.fix + (size_t)p * E + e);
                        const float rfix = a.fixr[((size_t)p * E + e) * M + kl];
                        const float fixm1 = expm1f(fmaf(f2.y, rfix, -f2.x));
                        const float4 *tab = a.zc + ((size_t)j * E + e) * G;
                        const float4 *dtab = a.dzc + ((size_t)j * E + e) * G;
                        bonds_generic(a, j, e, p, re, fixm1, Z, D, EM);
                        const float4 tp = __ldg(tab + (p < G ? p : G - 1));
                        const float chi = (e == 0) ? 1.f : expf(dt_l[jj][e]);
                        float Db[kMaxG], Zb[kMaxG];
                        for (int g = 0; g < G; ++g) Db[g] = Zb[g] = 0.f;
                        float chib = 0.f;
                        for (int c = 0; c < C; ++c) {
                            const int base = (c * E + e) * G;
                            float acc = 0.f;
                            for (int h = 0; h < G; ++h) acc = fmaf(c_w.wA[base + h], D[h], acc);
                            for (int g = 0; g < G; ++g) acc = fmaf(-c_w.wK[base + g], Z[g], acc);
                            chib = fmaf(mtb[c], acc, chib);
                            const float accb = mtb[c] * chi;
                            for (int h = 0; h < G; ++h) Db[h] = fmaf(accb, c_w.wA[base + h], Db[h]);
                            for (int g = 0; g < G; ++g) Zb[g] = fmaf(-accb, c_w.wK[base + g], Zb[g]);
                        }
                        if (e > 0) lb[e] += chib * chi;
                        float rbe = 0.f, pf = 0.f, ps = 0.f;
                        for (int g = G - 1; g >= 0; --g) {
                            if (g > p) {
                                const int gm = g - 1 >= 0 ? g - 1 : 0;
                                const float zp = Z[gm];
                                const float em = EM[g];
                                Zb[gm] += Zb[g] * (1.f + em) - Db[g] * em;
                                const float xb = (Zb[g] - Db[g]) * zp * (1.f + em);
                                const float4 t4 = __ldg(tab + g);
                                const float4 d4 = __ldg(dtab + g);
                                rbe -= xb * t4.w;
                                pf += xb * d4.z;
                                ps += xb * d4.w;
                            } else if (g == p) {
                                Zb[g] += Db[g] * fixm1;
                                const float fixb = Db[g] * Z[g];
                                const float yb = Zb[g] * Z[g];
                                const float4 d4 = __ldg(dtab + g);
                                rbe -= yb * tp.y;
                                pf += yb * d4.x;
                                ps += yb * d4.y;
                                const float ub = fixb * (1.f + fixm1);
                                const float2 df2 = __ldg(a.dfix + (size_t)p * E + e);
                                rfb[e] += ub * f2.y;
                                pf -= ub * df2.x;
                                ps -= ub * df2.y;
                            }
                        }
                        rb[e] += rbe;
                        pb[(PF + e) * 128] += pf;
                        pb[(PSR + e) * 128] += ps;
                    }
                    // ---- Euler sub-steps of (t_{j-1}, t_j], in reverse ----
                    for (int s = S - 1; s >= 0; --s) {
                        const int qs = (jj - 1) * S + s;
                        const uint32_t q = (uint32_t)((j - 1) * S + s);
                        increments_generic(a, k, q, W);
                        const float2 *dd = a.ddrift + (size_t)q * E;
                        for (int e = 0; e < E; ++e) {
                            const float2 d2 = __ldg(dd + e);
                            pb[(PF + e) * 128] += rb[e] * d2.x;
                            pb[(PSR + e) * 128] += rb[e] * fmaf(sqds, W[e], d2.y);
                        }
                        for (int e = 1; e < E; ++e) {
                            const float sx = __ldg(a.sig + E + e), sr = __ldg(a.sig + e);
                            pb[(PSX + e) * 128] += lb[e] * fmaf(sqds, W[E - 1 + e], -sx * ds)
                                                   - rb[e] * __ldg(a.rho + e) * sr * ds;
                        }
                        float rb0_extra = Ib * ds;
                        for (int e = 1; e < E; ++e) rb0_extra = fmaf(lb[e], ds, rb0_extra);
                        for (int e = 0; e < E; ++e) {
                            float v = rb[e] - rb[e] * c_sim.hw_a_ds[e];
                            if (e > 0) v -= lb[e] * ds;
                            else v += rb0_extra;
                            rb[e] = v;
                        }
                        for (int c = 0; c < C; ++c) {
                            const float g = st_g[qs][c];
                            const float gp = fmaxf(g, 0.f);
                            float gbn = gb[c];
                            const int w = c_sim.gpos[c];
                            if (w >= 0) {
                                const float Wc = W[w];
                                const float kap = __ldg(a.sig + 2 * E + c), th = __ldg(a.sig + 2 * E + C + c);
                                pb[(PK + c) * 128] += gb[c] * (th - gp) * ds;
                                pb[(PT + c) * 128] += gb[c] * kap * ds;
                                pb[(PN + c) * 128] += gb[c] * sqrtf(gp) * sqds * Wc;
                                if (g > 0.f)
                                    gbn = gb[c] * (1.f - c_sim.cir_kds[c] + c_sim.cir_nu_sqds[c] * Wc * 0.5f * rsqrtf(g));
                            }
                            if (g > 0.f) gbn += Lb[c] * ds;
                            gb[c] = gbn;
                        }
                    }
                    // the state at t_{j-1}: a reset date receives the adjoint of its fixing
                    if ((j - 1) % ppp == 0)
                        for (int e = 0; e < E; ++e) {
                            rb[e] += rfb[e];
                            rfb[e] = 0.f;
                        }
                }
            }
            // r_0 = f
            for (int e = 0; e < E; ++e) pb[(PF + e) * 128] += rb[e];
        }
    }

    // ---- block reduction of the parameter adjoints and of J (FP64, fixed order) ----
    __syncthreads();
    double *out = a.part + (size_t)blockIdx.x * (NPAR + 1);
    for (int i = 0; i <= NPAR; ++i) {
        red_s[tid] = (i < NPAR) ? (double)pb_s[i * 128 + tid] : J;
        __syncthreads();
        for (int s = 64; s > 0; s >>= 1) {
            if (tid < s) red_s[tid] += red_s[tid + s];
            __syncthreads();
        }
        if (tid == 0) out[i] = red_s[0];
        __syncthreads();
    }
}

cva_status adjoint_generic_launch(Sim &s, AdjBuffers &b, uint64_t seed, uint64_t k0, uint32_t M, cudaStream_t st)
{
    if (b.K < 1 || b.K > kAdjKMax || s.S > kAdjSMax)
        return fail(CVA_ENOTSUP, "adjoint: checkpoint interval <= 16, sub-steps <= 4");
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    AdjArgs a;
    a.M = M;
    a.k0 = (uint32_t)k0;
    a.seed_lo = (uint32_t)seed;
    a.seed_hi = (uint32_t)(seed >> 32);
    a.K = b.K;
    a.nseg = b.nseg;
    a.forward_only = b.forward_only;
    a.zc = s.d_zc;
    a.fix = s.d_fix;
    a.date_p = s.d_date_p;
    a.drift = s.d_drift;
    a.dzc = b.dzc;
    a.dfix = b.dfix;
    a.ddrift = b.ddrift;
    a.rho = b.rho;
    a.sig = b.sig;
    a.ckpt = b.ckpt;
    a.ckpt_I0 = b.ckpt_I0;
    a.fixr = b.fixr;
    a.part = b.part;
    const int npar = 3 * s.E - 1 + 3 * s.C;
    const size_t smem = (size_t)npar * 128 * sizeof(float);
    static bool attr = false;
    if (!attr) {
        CVA_CUDA_TRY(cudaFuncSetAttribute(adjoint_generic_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)((3 * kMaxE - 1 + 3 * kMaxC) * 128 * sizeof(float))));
        attr = true;
    }
    std::lock_guard<std::mutex> lk(t_const_mu);
    if (!t_last[dev]) CVA_CUDA_TRY(cudaEventCreateWithFlags(&t_last[dev], cudaEventDisableTiming));
    else CVA_CUDA_TRY(cudaStreamWaitEvent(st, t_last[dev], 0));
    if (t_owner[dev] != &s) {
        CVA_CUDA_TRY(upload_consts(s, st));
        t_owner[dev] = &s;
    }
    adjoint_generic_kernel<<<(M + 127u) / 128u, 128, smem, st>>>(a);
    CVA_CUDA_TRY(cudaGetLastError());
    CVA_CUDA_TRY(cudaEventRecord(t_last[dev], st));
    return CVA_OK;
}

cva_status outer_generic_launch(Sim &s, uint64_t seed, uint64_t k0, cudaStream_t st)
{
    int dev = 0;
    CVA_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CVA_EINVAL, "device index out of range");
    OuterArgs args = {};
    args.M = (uint32_t)s.M;
    args.k0 = (uint32_t)k0;
    args.seed_lo = (uint32_t)seed;
    args.seed_hi = (uint32_t)(seed >> 32);
    args.branch_step = s.branch_date <= s.n ? s.branch_date * s.S : INT_MAX;
    args.branch = s.branch;
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
    static std::atomic<bool> attr[64];
    if (!attr[dev].load(std::memory_order_acquire)) {
        for (auto kern : {sim_generic_kernel<1>, sim_generic_kernel<4>, sim_generic_kernel<8>})
            CVA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
        CVA_CUDA_TRY(cudaFuncSetAttribute(price_generic_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        attr[dev].store(true, std::memory_order_release);
    }
    int sms = 0;
    CVA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // eight warps per 32 paths while such blocks do not fill the chip twice (and for shapes that
    // need them), then four, and one where it can hold the factors and the blocks fill the chip
    // six times. Two economies and counterparties, 50 dates, eight / four / one warp: 2^11 paths
    // 42 / 48 / 89 us, 2^14 64 / 58 / 91, 2^16 181 / 149 / 130, 2^18 642 / 503 / 386 us
    const size_t ssmem = (size_t)kGenSteps * (((size_t)s.F + 3) / 4 * 4 + 1) * 32 * sizeof(float);
    const unsigned sblocks = (args.M + 31u) / 32u;
    const int most = std::max(s.E, s.C);
    if (sblocks < 2u * (unsigned)sms || most > 8) sim_generic_kernel<8><<<sblocks, 256, ssmem, st>>>(args);
    else if (sblocks < 6u * (unsigned)sms || most > 2) sim_generic_kernel<4><<<sblocks, 128, ssmem, st>>>(args);
    else sim_generic_kernel<1><<<sblocks, 32, ssmem, st>>>(args);
    CVA_CUDA_TRY(cudaGetLastError());
    if (s.ev[1]) CVA_CUDA_TRY(cudaEventRecord(s.ev[1], st));
    // portfolios per block: bond prices are computed once for them; up to 32 sums a thread
    const int NPB = std::max(1, std::min(s.NPF, 32 / s.C)), G = s.Ginst;
    const unsigned tiles = (args.M + 2u * kGenPriceThreads - 1) / (2u * kGenPriceThreads);
    const unsigned periods = (unsigned)((s.n + s.ppp - 1) / s.ppp), zb = (unsigned)((s.NPF + NPB - 1) / NPB);
    const PriceShape ps = price_shape((uint64_t)tiles * periods * zb, s.ppp, sms);
    const size_t psmem = ((size_t)NPB * s.C * kGenPriceThreads + (size_t)s.E * NPB * s.C * 2 * G) * sizeof(f32x2);
    price_generic_kernel<<<dim3(tiles, periods * (unsigned)ps.splits, zb), kGenPriceThreads, psmem, st>>>(args, ps, NPB);
    CVA_CUDA_TRY(cudaGetLastError());
    if (!capturing) CVA_CUDA_TRY(cudaEventRecord(t_last[dev], st));
    return CVA_OK;
}

}  // namespace

int outer_insts_generic(const OuterInst **out)
{
    // E, C, CS, NPF of -1: any shape within the limits; G: the schedules' longest
    static const OuterInst insts[] = {
        {-1, -1, -1, kMaxG, -1, outer_generic_launch, outer_forget, adjoint_generic_launch},
    };
    *out = insts;
    return (int)(sizeof(insts) / sizeof(insts[0]));
}

}  // namespace cva
