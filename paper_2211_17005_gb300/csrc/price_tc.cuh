// Pricing of every portfolio on the tensor cores (included by outer.cuh, inside its
// anonymous namespace; uses its constant tables, OuterArgs, PriceShape and with_live).
//
// For a pricing date, the date-bucketed MtM of App. B regrouped by (counterparty,
// currency, reset date) is a contraction over (economy e, live reset date g):
//   MtM_{pf,c} = sum_e sum_g ( chi_e D_e[g] wA[pf][c][e][g] - chi_e Z_e[g] wK[pf][c][e][g] ),
// the path's bond-price differences D and bond prices Z (times the FX rate chi) against
// the weights, which do not depend on the path or the date. With X the paths' rows
// [chi_e D_e | chi_e Z_e] (K = 2 LV columns per economy padded to a multiple of 8, LV the
// live reset dates of the period) and W the weights [NPF C][K], the MtM of 128 paths is
// the 128 x (NPF C) product X W^T.
//
// The product runs on tcgen05 in TF32 with the FP32 accuracy of the CUDA-core form
// recovered by splitting each operand into a TF32 head and a TF32 tail (x = hi + lo,
// lo = tf32(x - hi), 21 significant bits): X W^T ~ Xhi Whi^T + Xhi Wlo^T + Xlo Whi^T,
// three MMAs per K step accumulating in FP32 in tensor memory (the dropped Xlo Wlo^T
// term is below 2^-22 of each product). The CUDA cores compute the bond prices of
// their path (one thread per path, the chained expm1 differences of price_kernel) and
// write the X row of one economy at a time into shared memory, while the tensor core
// multiplies the previous economies'.
//
// Blocks of four independent slots of 128 threads (16 warps, so that the bond-price
// chains of one slot hide the latencies of the others), for the dates of one part of a
// period (blockIdx.y), so that the block runs the instantiation for the period's live
// reset dates: dead columns are neither computed nor multiplied (at 12 dates a year over
// ten years an economy's K falls from 24 to 14.4 on average). Slot s of block b takes path
// tiles 4 b + s, 4 b + s + 4 gridDim.x, ... and for each the part's dates, whose fixing it
// shares. Each slot has two X buffers (one where K = 24 leaves no room), so that an
// economy's row is written while the tensor core works on the last one, and two
// accumulators, so that a date's MtM is read while the next date's is accumulated. With one
// economy a row has no last one to hide behind: one buffer, and two blocks a multiprocessor
// (50001 paths, 50 dates: 120 us with two buffers, 70 so).
//
// Shared memory: W hi | W lo ([NN][KT] each, K-major core matrices), the X buffers
// (Xhi | Xlo, [128][GK] each) of every slot, the coupons at the fixing [E][512], the bond
// tables of the block's dates (the rest of the multiprocessor's memory is too small an L1 to
// hold them). TMEM: two 128 x NN FP32 accumulators per slot.
//
// Bound by the latency of a slot's chain (bond prices, operand split, stores to shared memory,
// the multiplication behind them) at 16 warps a multiprocessor. Six portfolios (50 to 2000
// swaps), 2^18 paths, 120 dates: 9.94 ms with every reset date, one X buffer and a block
// barrier and vote per economy, 7.99 ms by period with two, 5.74 ms with the tables and
// coupons in shared memory.
constexpr uint32_t kPriceMbarPolls = 1u << 26;   // limit of a wait for the tensor core
constexpr int kPriceSlots = 4;
constexpr int kPriceTcDates = 6;                 // dates of a block at most

template <int E, int NPF, int C, int LV>
struct PriceTc {
    static constexpr int GK = (2 * LV + 7) / 8 * 8;      // K of one economy: LV differences, LV prices, padding
    static constexpr int KT = E * GK;                     // K of the whole product
    static constexpr int NN = (NPF * C + 15) / 16 * 16;   // N: every (portfolio, counterparty), padded
    static constexpr uint32_t acc_cols = NN <= 32 ? 32u : 64u;
    static constexpr uint32_t tmem_cols = kPriceSlots * 2 * acc_cols;
    static constexpr int sWhi = 0, sWlo = NN * KT * 4;
    static constexpr int sX = 2 * NN * KT * 4;            // buffer b of slot s at sX + (s bufs + b) xbuf
    static constexpr int xbuf = 2 * 128 * GK * 4;         // Xhi, then Xlo at + 128 GK 4
    static constexpr int sFixBytes = E * 128 * kPriceSlots * 4, sTabBytes = kPriceTcDates * E * LV * 16;
    static constexpr int bufs = E > 1 && sX + 2 * kPriceSlots * xbuf + sFixBytes + sTabBytes <= 224 * 1024 ? 2 : 1;
    static constexpr int sTab = sX + bufs * kPriceSlots * xbuf;
    static constexpr int sFix = sTab + sTabBytes;
    static constexpr int bytes = sFix + sFixBytes;
    static_assert(NN <= 64 && tmem_cols <= 512, "tensor memory");
    static_assert(bytes <= 224 * 1024, "shared memory");
};

// shared memory of the widest period of at most G live reset dates
template <int E, int NPF, int C, int LV>
constexpr int price_tc_bytes()
{
    if constexpr (LV == 0) return 0;
    else return std::max(PriceTc<E, NPF, C, LV>::bytes, price_tc_bytes<E, NPF, C, LV - 1>());
}

// one answer per slot (its 128 threads, named barrier 1 + slot)
__device__ __forceinline__ bool slot_all(bool p, int slot)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, %2, 128, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(1 + slot)
        : "memory");
    return r != 0;
}

// the bond prices of one economy for one path (price_kernel's chain), times the FX
// rate: x = [chi D | chi Z | 0]
template <int LV, int GK>
__device__ __forceinline__ void price_row(float (&x)[GK], const float4 *tab, float re, float fixm1, float chi)
{
    const float4 tp = tab[0];
    float zp = expf(fmaf(-tp.y, re, tp.x));
    x[0] = chi * (zp * fixm1);
    x[LV] = chi * zp;
#pragma unroll
    for (int g = 1; g < LV; ++g) {
        const float4 t4 = tab[g];
        const float em = expm1_small(fmaf(-t4.w, re, t4.z));
        x[g] = chi * (-zp * em);
        zp = fmaf(zp, em, zp);
        x[LV + g] = chi * zp;
    }
#pragma unroll
    for (int g = 2 * LV; g < GK; ++g) x[g] = 0.f;
}

template <int E, int C, int CS, int G, int NPF>
__global__ void __launch_bounds__(128 * kPriceSlots, E > 1 ? 1 : 2) price_tc_kernel(OuterArgs a, uint32_t tiles, PriceShape ps)
{
    constexpr int F = 2 * E - 1 + CS, R = NPF * C;
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_mbar[3 * kPriceSlots];   // [slot][X buffer], then each slot's last
    const int tid = threadIdx.x, warp = tid >> 5, slot = tid >> 7, row = tid & 127;
    const size_t M = a.M;
    const int n = c_sim.n, ppp = c_sim.ppp;
    const int p = (int)blockIdx.y / ps.splits, part = (int)blockIdx.y % ps.splits;
    const int jp = p * ppp + 1 + part * ps.dates_per_block, j0 = max(jp, ps.start + 1);
    const int j1 = min(min(jp + ps.dates_per_block, (p + 1) * ppp + 1), n + 1);   // dates [j0, j1)
    if (j0 >= j1 && blockIdx.y > 0) return;
    const uint32_t tile0 = blockIdx.x * kPriceSlots + slot, step = gridDim.x * kPriceSlots;
    auto zeros = [&](int j) {
        for (uint32_t t = tile0; t < tiles; t += step) {
            const uint32_t kl = t * 128u + (uint32_t)row;
            if (kl < a.M)
                for (int q = 0; q < R; ++q) {
                    const size_t o = ((size_t)((q / C) * (n + 1) + j) * C + q % C) * M + kl;
                    a.expo[o] = 0.f;
                    if (a.mtm) a.mtm[o] = 0.f;
                }
        }
    };
    if (blockIdx.y == 0) zeros(0);   // no default at t_0: exposures of date 0 are never used
    with_live<G>(p < G ? G - p : 0, [&](auto lv_) {
        constexpr int LV = decltype(lv_)::value;
        if constexpr (LV == 0) {   // every swap has matured
            for (int j = j0; j < j1; ++j) zeros(j);
        } else {
            using P = PriceTc<E, NPF, C, LV>;
            constexpr int GK = P::GK, KT = P::KT, NN = P::NN, P0 = G - LV, BUFS = P::bufs;   // P0 = p
            if (warp == 0) {
                umma::tmem_alloc(&s_tmem, P::tmem_cols);
                umma::tmem_relinquish();
            }
            if (tid == 0) {
                for (int q = 0; q < 3 * kPriceSlots; ++q) umma::mbar_init(&s_mbar[q], 1);
                umma::fence_mbar_init();
            }
            // the weights as TF32 head and tail: row r = pf C + c, column e GK + g: wA (g < LV),
            // then -wK (LV <= g < 2 LV), then zeros
            for (int i = tid; i < NN * KT; i += blockDim.x) {
                const int r = i / KT, k = i % KT, e = k / GK, g = k % GK;
                float w = 0.f;
                if (r < R && g < 2 * LV) {
                    const int wrow = (r * E + e) * G + P0;
                    w = g < LV ? __ldg(a.w_glob + wrow + g) : -__ldg(a.w_glob + kMaxW + wrow + (g - LV));
                }
                const float hi = umma::tf32_round(w);
                const uint32_t off = umma::kmajor_offset32((uint32_t)r, (uint32_t)k, KT);
                *reinterpret_cast<float *>(tsm + P::sWhi + off) = hi;
                *reinterpret_cast<float *>(tsm + P::sWlo + off) = umma::tf32_round(w - hi);
            }
            float4 *tab_s = reinterpret_cast<float4 *>(tsm + P::sTab);   // [date - j0][E][LV]
            for (int i = tid; i < (j1 - j0) * E * LV; i += blockDim.x)
                tab_s[i] = __ldg(a.zc + ((size_t)j0 * E + i / LV) * G + P0 + i % LV);
            // the X columns past the live ones stay zero
            for (int b = 0; b < BUFS; ++b)
                for (int h = 0; h < 2; ++h)
                    for (int k = (2 * LV + 3) / 4 * 4; k < GK; k += 4)
                        *reinterpret_cast<float4 *>(tsm + P::sX + (slot * BUFS + b) * P::xbuf + h * 128 * GK * 4 +
                                                    umma::kmajor_offset32((uint32_t)row, (uint32_t)k, GK)) =
                            make_float4(0.f, 0.f, 0.f, 0.f);
            umma::fence_proxy_async();
            umma::fence_before_sync();
            __syncthreads();
            umma::fence_after_sync();
            const uint32_t tmem = s_tmem + (uint32_t)slot * 2u * P::acc_cols;
            const uint32_t sbase = umma::smem_u32(tsm);
            const uint32_t idesc = umma::idesc_tf32_f32(128u, (uint32_t)NN);
            float *fix_s = reinterpret_cast<float *>(tsm + P::sFix) + tid;   // [E], stride 512
            uint32_t uses = 0;        // X buffers filled so far by this slot
            uint32_t item = 0;        // dates priced so far by this slot
            bool ok = true;
            // the X buffer of use u is free (the MMAs of use u - BUFS have completed)
            auto wait_use = [&](uint32_t u) {   // completion of use u
                if (ok) ok = umma::mbar_wait(&s_mbar[2 * slot + (int)(u % BUFS)], (u / BUFS) & 1u, kPriceMbarPolls);
            };
            for (uint32_t t = tile0; t < tiles && ok; t += step) {
                const uint32_t kl = t * 128u + (uint32_t)row;
                const bool live = kl < a.M;
                const uint32_t kr = live ? kl : 0u;      // a valid path to read for a row past M
                {   // the running coupon's 1/ZC_{t_-}(t_+) - 1 of every economy
                    const float *ffix = a.features + (size_t)(p * ppp) * F * M + kr;   // state at the last reset
#pragma unroll 2
                    for (int e = 0; e < E; ++e) {
                        const float2 f2 = __ldg(a.fix + (size_t)p * E + e);
                        fix_s[e * 128 * kPriceSlots] = expm1f(fmaf(f2.y, __ldg(ffix + (size_t)e * M), -f2.x));
                    }
                }
                for (int j = j0; j < j1 && ok; ++j, ++item) {
                    const float *fe = a.features + (size_t)j * F * M + kr;
                    const float4 *tab = tab_s + (j - j0) * E * LV;
                    const float beta = expf(-__ldg(a.disc + (size_t)j * M + kr));
                    const uint32_t acc = tmem + (item & 1u) * P::acc_cols;
                    {   // the next date's states (the next tile's first), for its loads to find in the L2 cache
                        const bool more = j + 1 < j1;
                        const size_t jn = more ? (size_t)(j + 1) : (size_t)j0;
                        const uint64_t kn = (uint64_t)(more ? t : t + step) * 128u + (uint32_t)(row & ~31);
                        if (kn < a.M)
                            prefetch_state<E>(a.features + jn * F * M, a.disc + jn * M, M, (uint32_t)kn, a.M);
                    }
                    // an economy's state is requested two economies ahead (rate, log chi)
                    float n_r[2], n_l[2];
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int e = i < E ? i : 0;
                        n_r[i] = __ldg(fe + (size_t)e * M);
                        n_l[i] = e > 0 ? __ldg(fe + (size_t)(E - 1 + e) * M) : 0.f;
                    }
#pragma unroll 1
                    for (int e = 0; e < E; ++e, ++uses, tab += LV) {
                        const float re = n_r[0], chi = e == 0 ? 1.f : expf(n_l[0]);
                        n_r[0] = n_r[1];
                        n_l[0] = n_l[1];
                        if (e + 2 < E) {
                            n_r[1] = __ldg(fe + (size_t)(e + 2) * M);
                            n_l[1] = __ldg(fe + (size_t)(E + 1 + e) * M);   // log chi^{e+2}
                        }
                        float x[GK];
                        price_row<LV, GK>(x, tab, re, fix_s[e * 128 * kPriceSlots], chi);
                        if (uses >= (uint32_t)BUFS) wait_use(uses - BUFS);
                        const int xo = P::sX + (slot * BUFS + (int)(uses % BUFS)) * P::xbuf;
#pragma unroll
                        for (int q = 0; q < (2 * LV + 3) / 4; ++q) {
                            float4 h, l;
                            h.x = umma::tf32_round(x[4 * q + 0]);
                            h.y = umma::tf32_round(x[4 * q + 1]);
                            h.z = umma::tf32_round(x[4 * q + 2]);
                            h.w = umma::tf32_round(x[4 * q + 3]);
                            l.x = umma::tf32_round(x[4 * q + 0] - h.x);
                            l.y = umma::tf32_round(x[4 * q + 1] - h.y);
                            l.z = umma::tf32_round(x[4 * q + 2] - h.z);
                            l.w = umma::tf32_round(x[4 * q + 3] - h.w);
                            const uint32_t off = umma::kmajor_offset32((uint32_t)row, (uint32_t)(4 * q), GK);
                            *reinterpret_cast<float4 *>(tsm + xo + off) = h;
                            *reinterpret_cast<float4 *>(tsm + xo + 128 * GK * 4 + off) = l;
                        }
                        umma::fence_proxy_async();
                        umma::fence_before_sync();
                        asm volatile("bar.sync %0, 128;" ::"r"(1 + slot) : "memory");
                        if (row == 0) {
                            umma::fence_after_sync();
                            const uint32_t ah = sbase + (uint32_t)xo, al = ah + 128u * GK * 4u;
                            const uint32_t asbo = (GK / 4) * 128u, bsbo = (KT / 4) * 128u;
#pragma unroll
                            for (int s = 0; s < GK / 8; ++s) {
                                const uint32_t bk = (uint32_t)((e * GK + 8 * s) / 4) * 128u;
                                const uint64_t dah = umma::smem_desc(ah + s * 256u, 128u, asbo),
                                               dal = umma::smem_desc(al + s * 256u, 128u, asbo),
                                               dbh = umma::smem_desc(sbase + P::sWhi + bk, 128u, bsbo),
                                               dbl = umma::smem_desc(sbase + P::sWlo + bk, 128u, bsbo);
                                umma::mma_tf32(acc, dah, dbh, idesc, (e > 0 || s > 0) ? 1u : 0u);
                                umma::mma_tf32(acc, dah, dbl, idesc, 1u);
                                umma::mma_tf32(acc, dal, dbh, idesc, 1u);
                            }
                            umma::commit(&s_mbar[2 * slot + (int)(uses % BUFS)]);
                        }
                    }
                    // the date's last MMAs (and with them all before) have completed
                    wait_use(uses - 1);
                    ok = slot_all(ok, slot);
                    umma::fence_after_sync();
                    // epilogue: this thread's row of the accumulator, exposures of every (pf, c)
                    const size_t o0 = (size_t)j * C * M + kl, pf_stride = (size_t)(n + 1) * C * M;
#pragma unroll
                    for (int c0 = 0; c0 < NN; c0 += 16) {
                        float v[16];
                        umma::tmem_ld16(acc + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
                        umma::tmem_wait_ld();
                        if (live)
#pragma unroll
                            for (int i = 0; i < 16; ++i)
                                if (c0 + i < R) {
                                    const size_t o = o0 + (size_t)((c0 + i) / C) * pf_stride + (size_t)((c0 + i) % C) * M;
                                    const float m = ok ? v[i] : __int_as_float(0x7fc00000);   // a wait that gave up: NaN
                                    a.expo[o] = c_sim.lgd[(c0 + i) % C] * beta * fmaxf(m, 0.f);
                                    if (a.mtm) a.mtm[o] = m;
                                }
                    }
                    // (the other accumulator takes the next date; this one is written again only
                    // after barriers of the next date that follow these reads)
                    umma::fence_before_sync();
                }
            }
            // after a wait that gave up, the slot's MMAs still in flight complete (bounded) before
            // the accumulators are freed: on a barrier of its own, as the parity of the buffers'
            // says nothing once a phase was not waited for
            if (!ok && row == 0) {
                umma::commit(&s_mbar[2 * kPriceSlots + slot]);
                (void)umma::mbar_wait(&s_mbar[2 * kPriceSlots + slot], 0u, kPriceMbarPolls);
            }
            umma::fence_before_sync();
            __syncthreads();
            if (warp == 0) umma::tmem_dealloc(s_tmem, P::tmem_cols);
        }
    });
}
