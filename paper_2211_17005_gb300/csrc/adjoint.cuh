// Adjoint (reverse-mode) sensitivities of the smooth CVA_0, included by outer.cuh so that
// it reads the same constant-memory tables.
//
// The sampled default indicators have zero pathwise derivative, so the function
// differentiated is the smooth functional the oversimulated average estimates: the
// exact discrete conditional default probabilities e^{-Lambda(t_{j-1})} -
// e^{-Lambda(t_j)} (the intensity form of eq. (eq:CVAint)):
//   J_k = sum_c sum_{j=1..n} V_c(j) (e^{-Lambda_c(j-1)} - e^{-Lambda_c(j)}),
//   V_c(j) = (1 - R_c) beta_j MtM_c(j)^+,  CVA_0 = mean_k J_k.
// Parameters: flat curve levels f_e, rate volatilities sigma^r_e, FX volatilities
// sigma^chi_e (e >= 1), CIR kappa_c, theta_c, nu_c (gamma_0 held fixed; fixed
// rates of the swaps held at their base-curve par values).
//
// Three kernels over a range of outer paths:
//   sim_kernel (adjoint) the states, discount integrals and survival factors e^{-Lambda} of
//                        every date, and of every fine step the increments W and the
//                        intensities before it;
//   adj_price_kernel     the pricing at every date, which depends on that date's state only:
//                        V_c and, in reverse, what the date adds to the adjoints of its
//                        rates, log FX rates, discount integral and fixings, and to the
//                        parameters of the bond tables;
//   adj_reverse_kernel   the adjoint recursions over the fine steps from the last, in which
//                        the factors are independent but for r^0.
// Keeping the states and increments (40 KB a path at 100 dates and 27 factors) instead of
// recomputing them from checkpoints lets the pricing, the bulk of the work, run over all
// (path, date) pairs at once, and draws the normals once instead of three times. One
// thread per path with checkpoints held 255 registers and local arrays and took 23.0 ms at
// 2^17 paths, the three kernels 6.2 ms; the calling code bounds the memory by taking the
// paths in ranges.
#pragma once

namespace cva {
namespace {

struct AdjSplitArgs {
    uint32_t M;
    const float4 *__restrict__ zc;      // [n+1][E][G] (lnA, B, dlnA, dB)
    const float2 *__restrict__ fix;     // [periods+1][E] (lnA, B)
    const float4 *__restrict__ dzc;     // [n+1][E][G] d/df, d/dsigma of (lnA, dlnA)
    const float2 *__restrict__ dfix;    // [periods+1][E] d/df, d/dsigma of lnA at the fixing
    const float2 *__restrict__ ddrift;  // [n*S][E] d drift/df, d drift/dsigma^r (quanto included)
    const float *__restrict__ rho;      // [E] correlation of r^e and log chi^e (entry 0 unused)
    const float *__restrict__ sig;      // [E] sigma^r, [E] sigma^chi, [C] kappa, [C] theta, [C] nu
    const float *w_glob;                // the weights
    const float *features, *disc;       // [n+1][F][M], [n+1][M]
    const float *surv;                  // [n+1][C][M] e^{-Lambda}
    const float *inc, *gpre;            // [n*S][F][M] increments, [n*S][C][M] intensities before a fine step
    float *V;                           // [n+1][C][M]
    float *rbin, *lbin, *ibin;          // [n][E][M] (lbin row 0: the sum of the others), [n][M]: row j-1 = date j
    float *fixin;                       // [periods * splits][E][M]
    double *part_p;                     // [blocks][2E + 1]: f_e, sigma^r_e of the bond tables, J
    double *part_r;                     // [blocks][NPAR]
};

// Block: 256 paths (two a thread, in packed pairs as price_kernel) and the dates of one part of
// a period. The adjoint needs the chain of bond prices from the last reset date back, so a
// thread keeps an economy's in registers. J runs as an FP32 value and its rounding errors
// without the FP64 pipe (its results and those of FP64 sums differ by 2e-16 at most over the
// shapes and path counts of the benchmark; FP64 sums take 1.3% of the call longer, 8% of the
// forward's). The parameters' adjoints of a path run in FP32 over the block's dates and go to
// FP64 path by path. Bound by the latency of its chains at three blocks a multiprocessor (no
// more fit its registers, of which 200 bytes still spill). The states are requested an
// economy ahead, from the L2 cache, into which they come a date ahead. 2^15 paths, 100 dates:
// 1051 us with loads where they are used and four blocks, 787 us.
template <int E, int C, int CS, int G, bool REV>
__global__ void __launch_bounds__(128, 3) adj_price_kernel(AdjSplitArgs a, PriceShape ps)
{
    constexpr int F = 2 * E - 1 + CS, NT = 128;
    extern __shared__ __align__(16) unsigned char adj_smem[];
    f32x2 *w_s = reinterpret_cast<f32x2 *>(adj_smem);            // [E][C][2 LV] (-wA, -wK), doubled
    f32x2 *rf_s = w_s + E * C * 2 * G;                           // [E][NT] adjoints of the fixings
    f32x2 *fix_s = rf_s + E * NT;                                // [E][NT] running coupons at the fixing
    float4 *tab_s = reinterpret_cast<float4 *>(fix_s + E * NT);  // [2][E][LV] the date's bond tables, their derivatives
    f32x2 *par_s = reinterpret_cast<f32x2 *>(tab_s + 2 * E * G); // [2E][NT] parameter adjoints
    __shared__ double j_s[NT];
    const int tid = threadIdx.x;
    const size_t M = a.M;
    const int n = c_sim.n, ppp = c_sim.ppp;
    const int p = (int)blockIdx.y / ps.splits, part = (int)blockIdx.y % ps.splits;
    const int j0 = p * ppp + 1 + part * ps.dates_per_block;
    const int j1 = min(min(j0 + ps.dates_per_block, (p + 1) * ppp + 1), n + 1);   // dates [j0, j1)
    const uint32_t k0 = blockIdx.x * 2u * NT + (uint32_t)tid, k1 = k0 + NT;
    const bool live0 = k0 < a.M, live1 = k1 < a.M;
    const uint32_t r0 = live0 ? k0 : 0u, r1 = live1 ? k1 : r0;   // paths read
    auto put = [&](float *row, float x, float y) {
        if (live0) row[k0] = x;
        if (live1) row[k1] = y;
    };
    SumPair J = {0.f, 0.f};
    if (REV)
        for (int e = 0; e < E; ++e) {
            rf_s[e * NT + tid] = pack2(0.f, 0.f);
            par_s[2 * e * NT + tid] = par_s[(2 * e + 1) * NT + tid] = pack2(0.f, 0.f);
        }
    with_live<G>(p < G ? G - p : 0, [&](auto lv_) {
        constexpr int LV = decltype(lv_)::value;
        if constexpr (LV == 0) {   // every swap has matured: no exposure, no adjoints
            if (REV)
                for (int j = j0; j < j1; ++j) {
                    for (int c = 0; c < C; ++c) put(a.V + ((size_t)j * C + c) * M, 0.f, 0.f);
                    for (int e = 0; e < E; ++e) {
                        put(a.rbin + ((size_t)(j - 1) * E + e) * M, 0.f, 0.f);
                        put(a.lbin + ((size_t)(j - 1) * E + e) * M, 0.f, 0.f);
                    }
                    put(a.ibin + (size_t)(j - 1) * M, 0.f, 0.f);
                }
        } else {
            constexpr int P0 = G - LV;   // = p
            for (int i = tid; i < E * C * 2 * LV; i += NT) {
                const int q = i % (2 * LV), row = i / (2 * LV) % C, e = i / (2 * LV * C), wrow = (row * E + e) * G + P0;
                const float w = q < LV ? __ldg(a.w_glob + wrow + q) : __ldg(a.w_glob + kMaxW + wrow + q - LV);
                w_s[i] = pack2(-w, -w);
            }
            const float2 *fx = a.fix + (size_t)p * E;
            {   // 1/ZC_{t_-}(t_+) - 1, which the period's dates share
                const float *ffix = a.features + (size_t)(p * ppp) * F * M;   // state at the last reset
#pragma unroll 2
                for (int e = 0; e < E; ++e) {
                    const float2 f2 = __ldg(fx + e);
                    fix_s[e * NT + tid] = pack2(expm1f(fmaf(f2.y, __ldg(ffix + (size_t)e * M + r0), -f2.x)),
                                                expm1f(fmaf(f2.y, __ldg(ffix + (size_t)e * M + r1), -f2.x)));
                }
            }
            // bond prices of economy e (price_kernel's): X holds -D, then Z; em[g] = expm1(x_g)
            auto bonds = [&](const float4 *tab, f32x2 re, f32x2 fixm1, f32x2 (&X)[2 * LV], f32x2 (&em)[LV]) {
                const float2 r = unpack2(re), fm = unpack2(fixm1);
                const float4 tp = tab[0];
                const float z0 = expf(fmaf(-tp.y, r.x, tp.x)), z1 = expf(fmaf(-tp.y, r.y, tp.x));
                X[0] = pack2(-(z0 * fm.x), -(z1 * fm.y));
                X[LV] = pack2(z0, z1);
                em[0] = pack2(0.f, 0.f);
#pragma unroll
                for (int g = 1; g < LV; ++g) {
                    const float4 t4 = tab[g];
                    em[g] = expm1_small2(fma2(pack2(-t4.w, -t4.w), re, pack2(t4.z, t4.z)));
                    X[g] = mul2(X[LV + g - 1], em[g]);
                    X[LV + g] = fma2(X[LV + g - 1], em[g], X[LV + g - 1]);
                }
            };
            for (int j = j0; j < j1; ++j) {
                __syncthreads();   // the weights, and every warp is done with the last date's tables
                for (int i = tid; i < E * LV; i += NT) {
                    const size_t o = ((size_t)j * E + i / LV) * G + P0 + i % LV;
                    tab_s[i] = __ldg(a.zc + o);
                    if (REV) tab_s[E * LV + i] = __ldg(a.dzc + o);
                }
                __syncthreads();
                const float *fe = a.features + (size_t)j * F * M;
                if (j + 1 < j1) {   // the next date's states, so that its loads find them in the L2 cache
                    const float *dn = a.disc + (size_t)(j + 1) * M;
                    prefetch_state<E>(fe + (size_t)F * M, dn, M, k0 & ~31u, a.M);
                    prefetch_state<E>(fe + (size_t)F * M, dn, M, k1 & ~31u, a.M);
                }
                // economy e's rate and log FX rate, requested one economy ahead
                float xr0, xr1, xl0 = 0.f, xl1 = 0.f;
                auto request = [&](int e) {
                    if (e >= E) return;
                    const float *rp = fe + (size_t)e * M, *lp = rp + (size_t)(E - 1) * M;
                    xr0 = __ldg(rp + r0);
                    xr1 = __ldg(rp + r1);
                    if (e > 0) {
                        xl0 = __ldg(lp + r0);
                        xl1 = __ldg(lp + r1);
                    }
                };
                f32x2 mt[C];
#pragma unroll
                for (int c = 0; c < C; ++c) mt[c] = pack2(0.f, 0.f);
                request(0);
#pragma unroll 1
                for (int e = 0; e < E; ++e) {
                    f32x2 X[2 * LV], em[LV];
                    const f32x2 re = pack2(xr0, xr1);
                    const f32x2 chi = e == 0 ? pack2(1.f, 1.f) : pack2(expf(xl0), expf(xl1));
                    request(e + 1);
                    bonds(tab_s + e * LV, re, fix_s[e * NT + tid], X, em);
                    const f32x2 *w = w_s + e * C * 2 * LV;
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        f32x2 acc = pack2(0.f, 0.f);
#pragma unroll
                        for (int q = 0; q < 2 * LV; q += 2) {
                            const ulonglong2 w2 = *reinterpret_cast<const ulonglong2 *>(w + c * 2 * LV + q);
                            acc = fma2(w2.x, X[q], acc);
                            acc = fma2(w2.y, X[q + 1], acc);
                        }
                        mt[c] = fma2(chi, acc, mt[c]);
                    }
                }
                // exposures, survival terms and the adjoints of the MtM and of int r^0
                const float b0 = expf(-__ldg(a.disc + (size_t)j * M + r0)), b1 = expf(-__ldg(a.disc + (size_t)j * M + r1));
                f32x2 mtb[C];
                float ib0 = 0.f, ib1 = 0.f;
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const float2 m = unpack2(mt[c]);
                    const float l = c_sim.lgd[c];
                    const float V0 = l * b0 * fmaxf(m.x, 0.f), V1 = l * b1 * fmaxf(m.y, 0.f);
                    const float *s1 = a.surv + ((size_t)j * C + c) * M, *s0 = s1 - (size_t)C * M;
                    const float d0 = __ldg(s0 + r0) - __ldg(s1 + r0), d1 = __ldg(s0 + r1) - __ldg(s1 + r1);
                    // V d with its rounding error: as exact as FP64 without its narrow pipe
                    const float t0 = live0 ? d0 : 0.f, t1 = live1 ? d1 : 0.f;
                    const float q0 = __fmul_rn(V0, t0), q1 = __fmul_rn(V1, t1);
                    J.add(q0, fmaf(V0, t0, -q0));
                    J.add(q1, fmaf(V1, t1, -q1));
                    if (REV) {
                        put(a.V + ((size_t)j * C + c) * M, V0, V1);
                        mtb[c] = pack2(m.x > 0.f ? d0 * l * b0 : 0.f, m.y > 0.f ? d1 * l * b1 : 0.f);
                        ib0 -= d0 * V0;
                        ib1 -= d1 * V1;
                    }
                }
                if (!REV) continue;
                put(a.ibin + (size_t)(j - 1) * M, ib0, ib1);
                float lb0 = 0.f, lb1 = 0.f;
                request(0);
#pragma unroll 1
                for (int e = 0; e < E; ++e) {
                    f32x2 X[2 * LV], em[LV], u[2 * LV];
                    const f32x2 fixm1 = fix_s[e * NT + tid];
                    const float4 *tab = tab_s + e * LV, *dtab = tab + E * LV;
                    const f32x2 re = pack2(xr0, xr1);
                    const f32x2 chi = e == 0 ? pack2(1.f, 1.f) : pack2(expf(xl0), expf(xl1));
                    request(e + 1);
                    bonds(tab, re, fixm1, X, em);
                    // u = sum_c (adjoint of MtM_c) w_c: times chi the adjoint of X
                    const f32x2 *w = w_s + e * C * 2 * LV;
#pragma unroll
                    for (int q = 0; q < 2 * LV; ++q) u[q] = pack2(0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < C; ++c)
#pragma unroll
                        for (int q = 0; q < 2 * LV; q += 2) {
                            const ulonglong2 w2 = *reinterpret_cast<const ulonglong2 *>(w + c * 2 * LV + q);
                            u[q] = fma2(w2.x, mtb[c], u[q]);
                            u[q + 1] = fma2(w2.y, mtb[c], u[q + 1]);
                        }
                    f32x2 chib = pack2(0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < 2 * LV; ++q) {
                        chib = fma2(u[q], X[q], chib);
                        u[q] = mul2(u[q], chi);
                    }
                    // -D_g = Z_{g-1} em_g, Z_g = Z_{g-1} (1 + em_g), em_g = expm1(x_g), x_g = dlnA - dB r
                    const f32x2 one = pack2(1.f, 1.f);
                    f32x2 rb = pack2(0.f, 0.f), pf = rb, psg = rb;
#pragma unroll
                    for (int g = LV - 1; g >= 1; --g) {
                        const f32x2 em1 = fma2(em[g], one, one);
                        const f32x2 xb = mul2(mul2(fma2(u[LV + g], one, u[g]), X[LV + g - 1]), em1);
                        u[LV + g - 1] = fma2(u[LV + g], em1, fma2(u[g], em[g], u[LV + g - 1]));
                        const float4 t4 = tab[g], d4 = dtab[g];
                        rb = fma2(xb, pack2(-t4.w, -t4.w), rb);
                        pf = fma2(xb, pack2(d4.z, d4.z), pf);
                        psg = fma2(xb, pack2(d4.w, d4.w), psg);
                    }
                    // the first live date: -D_0 = -Z_0 fixm1, Z_0 = exp(lnA - B r)
                    {
                        const f32x2 ndb = u[0];   // adjoint of -D_0
                        const float2 nd = unpack2(ndb);
                        const f32x2 db = pack2(-nd.x, -nd.y);
                        const f32x2 yb = mul2(fma2(db, fixm1, u[LV]), X[LV]);
                        const f32x2 ub = mul2(mul2(db, X[LV]), fma2(fixm1, one, one));
                        const float4 tp = tab[0], d4 = dtab[0];
                        const float2 f2 = __ldg(fx + e), df2 = __ldg(a.dfix + (size_t)p * E + e);
                        rb = fma2(yb, pack2(-tp.y, -tp.y), rb);
                        pf = fma2(yb, pack2(d4.x, d4.x), pf);
                        psg = fma2(yb, pack2(d4.y, d4.y), psg);
                        pf = fma2(ub, pack2(-df2.x, -df2.x), pf);
                        psg = fma2(ub, pack2(-df2.y, -df2.y), psg);
                        rf_s[e * NT + tid] = fma2(ub, pack2(f2.y, f2.y), rf_s[e * NT + tid]);
                    }
                    const float2 rb2 = unpack2(rb);
                    put(a.rbin + ((size_t)(j - 1) * E + e) * M, rb2.x, rb2.y);
                    par_s[2 * e * NT + tid] = fma2(pf, one, par_s[2 * e * NT + tid]);
                    par_s[(2 * e + 1) * NT + tid] = fma2(psg, one, par_s[(2 * e + 1) * NT + tid]);
                    if (e > 0) {
                        const float2 l2 = unpack2(mul2(chib, chi));
                        put(a.lbin + ((size_t)(j - 1) * E + e) * M, l2.x, l2.y);
                        lb0 += l2.x;
                        lb1 += l2.y;
                    }
                }
                put(a.lbin + (size_t)(j - 1) * E * M, lb0, lb1);
            }
        }
    });
    if (REV)
        for (int e = 0; e < E; ++e) {
            const float2 v = unpack2(rf_s[e * NT + tid]);
            put(a.fixin + ((size_t)blockIdx.y * E + e) * M, v.x, v.y);
        }
    // block sums in FP64, fixed order: a warp per value
    j_s[tid] = (double)J.hi + (double)J.lo;
    __syncthreads();
    double *out = a.part_p + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (2 * E + 1);
    const int lane = tid & 31;
    for (int v = REV ? tid >> 5 : 2 * E + (tid >> 5); v <= 2 * E; v += NT / 32) {
        double s = 0.0;
        for (int i = lane; i < NT; i += 32) {
            if (v < 2 * E) {
                const float2 x = unpack2(par_s[v * NT + i]);
                const uint32_t k = blockIdx.x * 2u * NT + (uint32_t)i;
                s += (k < a.M ? (double)x.x : 0.0) + (k + NT < a.M ? (double)x.y : 0.0);
            } else {
                s += j_s[i];
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) out[v] = s;
    }
}

// Block: 32 outer paths (lane = path), NW warps with the factors split over them as in
// sim_kernel; the economy of index 0 alone needs the others, through the sum of their
// log-FX adjoints, which adj_price_kernel provides. Bound by HBM (80 floats a (path, step)):
// 321 us for 2^15 paths and 100 steps, 3.3 TB/s, with eight warps; 4 warps leave too few loads
// in flight.
template <int E, int C, int CS, int NW>
__global__ void __launch_bounds__(32 * NW) adj_reverse_kernel(AdjSplitArgs a, int splits)
{
    constexpr int F = 2 * E - 1 + CS, NPAR = 3 * E - 1 + 3 * C;
    constexpr int ME = (E + NW - 1) / NW, MC = (C + NW - 1) / NW;
    constexpr int PF = 0, PSR = E, PSX = 2 * E - 1, PK = 3 * E - 1, PT = PK + C, PN = PT + C;   // PSX + e for e >= 1
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t kl = blockIdx.x * 32u + (uint32_t)lane;
    const bool live = kl < a.M;
    const size_t M = a.M;
    const uint32_t kr = live ? kl : 0u;   // a valid path to read for a lane past M
    const int n = c_sim.n, S = c_sim.S, ppp = c_sim.ppp;
    const float ds = c_sim.ds, sqds = c_sim.sqds;
    auto has_e = [&](int i) { return NW * (i + 1) <= E || warp + NW * i < E; };
    auto has_c = [&](int i) { return NW * (i + 1) <= C || warp + NW * i < C; };
    float rb[ME], lb[ME], pf[ME], psr[ME], psx[ME], gb[MC], Lb[MC], Vn[MC], pk[MC], pt[MC], pn[MC];
    float Ib = 0.f, lbs = 0.f;
#pragma unroll
    for (int i = 0; i < ME; ++i) rb[i] = lb[i] = pf[i] = psr[i] = psx[i] = 0.f;
#pragma unroll
    for (int i = 0; i < MC; ++i) gb[i] = Lb[i] = Vn[i] = pk[i] = pt[i] = pn[i] = 0.f;
    // what a fine step and a date read, requested one ahead of their use: nothing in the
    // recursions' inputs depends on them, and a step's own work is short
    float We[ME] = {}, Wx[ME] = {}, Wc[MC] = {}, gq[MC] = {}, ri[ME] = {}, li[ME] = {}, sv[MC] = {}, vv[MC] = {}, ibn = 0.f,
          lsn = 0.f;
    auto load_step = [&](int q) {
        const float *W = a.inc + (size_t)q * F * M + kr, *g = a.gpre + (size_t)q * C * M + kr;
#pragma unroll
        for (int i = 0; i < ME; ++i)
            if (has_e(i)) {
                const int e = warp + NW * i;
                We[i] = __ldg(W + (size_t)e * M);
                Wx[i] = e > 0 ? __ldg(W + (size_t)(E - 1 + e) * M) : 0.f;
            }
#pragma unroll
        for (int i = 0; i < MC; ++i)
            if (has_c(i)) {
                const int c = warp + NW * i;
                gq[i] = __ldg(g + (size_t)c * M);
                Wc[i] = NW * (i + 1) <= CS || c < CS ? __ldg(W + (size_t)(2 * E - 1 + c) * M) : 0.f;
            }
    };
    auto load_date = [&](int j) {
        const float *rin = a.rbin + (size_t)(j - 1) * E * M + kr, *lin = a.lbin + (size_t)(j - 1) * E * M + kr;
        const float *s = a.surv + (size_t)j * C * M + kr, *v = a.V + (size_t)j * C * M + kr;
#pragma unroll
        for (int i = 0; i < ME; ++i)
            if (has_e(i)) {
                const int e = warp + NW * i;
                ri[i] = __ldg(rin + (size_t)e * M);
                li[i] = e > 0 ? __ldg(lin + (size_t)e * M) : 0.f;
            }
        if (warp == 0) {
            ibn = __ldg(a.ibin + (size_t)(j - 1) * M + kr);
            lsn = __ldg(lin);
        }
#pragma unroll
        for (int i = 0; i < MC; ++i)
            if (has_c(i)) {
                const int c = warp + NW * i;
                sv[i] = __ldg(s + (size_t)c * M);
                vv[i] = __ldg(v + (size_t)c * M);
            }
    };
    load_date(n);
    load_step(n * S - 1);
    for (int j = n; j >= 1; --j) {
        // what the pricing at t_j adds, and the survival terms
#pragma unroll
        for (int i = 0; i < ME; ++i) {
            rb[i] += ri[i];
            lb[i] += li[i];
        }
        Ib += ibn;
        lbs += lsn;
#pragma unroll
        for (int i = 0; i < MC; ++i) {
            Lb[i] += sv[i] * (vv[i] - Vn[i]);
            Vn[i] = vv[i];
        }
        if (j > 1) load_date(j - 1);
        for (int s = S - 1; s >= 0; --s) {   // Euler sub-steps of (t_{j-1}, t_j], in reverse
            const int q = (j - 1) * S + s;
            float we[ME], wx[ME], wc[MC], g_[MC];
#pragma unroll
            for (int i = 0; i < ME; ++i) {
                we[i] = We[i];
                wx[i] = Wx[i];
            }
#pragma unroll
            for (int i = 0; i < MC; ++i) {
                wc[i] = Wc[i];
                g_[i] = gq[i];
            }
            if (q > 0) load_step(q - 1);
            const float2 *dd = a.ddrift + (size_t)q * E;
#pragma unroll
            for (int i = 0; i < ME; ++i)
                if (has_e(i)) {
                    const int e = warp + NW * i;
                    const float2 d2 = __ldg(dd + e);
                    pf[i] += rb[i] * d2.x;
                    psr[i] += rb[i] * fmaf(sqds, we[i], d2.y);
                    float v = rb[i] - rb[i] * c_sim.hw_a_ds[e];
                    if (e > 0) {
                        const float sx = __ldg(a.sig + E + e), sr = __ldg(a.sig + e);
                        psx[i] += lb[i] * fmaf(sqds, wx[i], -sx * ds) - rb[i] * __ldg(a.rho + e) * sr * ds;
                        v -= lb[i] * ds;
                    } else {
                        v += fmaf(lbs, ds, Ib * ds);
                    }
                    rb[i] = v;
                }
#pragma unroll
            for (int i = 0; i < MC; ++i)
                if (has_c(i)) {
                    const int c = warp + NW * i;
                    const float g = g_[i], gp = fmaxf(g, 0.f);
                    float gbn = gb[i];
                    if (NW * (i + 1) <= CS || c < CS) {
                        const float kap = __ldg(a.sig + 2 * E + c), th = __ldg(a.sig + 2 * E + C + c);
                        pk[i] += gb[i] * (th - gp) * ds;
                        pt[i] += gb[i] * kap * ds;
                        pn[i] += gb[i] * sqrtf(gp) * sqds * wc[i];
                        if (g > 0.f)
                            gbn = gb[i] * (1.f - c_sim.cir_kds[c] + c_sim.cir_nu_sqds[c] * wc[i] * 0.5f * rsqrtf(g));
                    }
                    if (g > 0.f) gbn += Lb[i] * ds;
                    gb[i] = gbn;
                }
        }
        // the state at t_{j-1}: a reset date receives the adjoints of its fixing
        if ((j - 1) % ppp == 0) {
            const int p = (j - 1) / ppp;
#pragma unroll
            for (int i = 0; i < ME; ++i)
                if (has_e(i))
                    for (int b = 0; b < splits; ++b)
                        rb[i] += __ldg(a.fixin + ((size_t)(p * splits + b) * E + warp + NW * i) * M + kr);
        }
    }
    // sums over the block's paths, FP64
    double *out = a.part_r + (size_t)blockIdx.x * NPAR;
    auto total = [&](float x, int at) {
        double s = live ? (double)x : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) out[at] = s;
    };
#pragma unroll
    for (int i = 0; i < ME; ++i)
        if (has_e(i)) {
            const int e = warp + NW * i;
            total(pf[i] + rb[i], PF + e);   // r_0 = f
            total(psr[i], PSR + e);
            if (e > 0) total(psx[i], PSX + e);
        }
#pragma unroll
    for (int i = 0; i < MC; ++i)
        if (has_c(i)) {
            const int c = warp + NW * i;
            total(pk[i], PK + c);
            total(pt[i], PT + c);
            total(pn[i], PN + c);
        }
}

}  // namespace
}  // namespace cva
