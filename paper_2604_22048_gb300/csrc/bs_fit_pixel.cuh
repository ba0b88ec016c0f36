// Pixel-space evaluations of the log posterior and its gradient (Appendix C): per-pixel
// weights on the tensor cores, a dense covariance on the CUDA cores.  Included by
// bs_fit_impl.cuh inside namespace bs::(anonymous), after the spectral evaluation
// (eval_logpost) and the table layout it reuses.
#pragma once

// ---- Spatially variable noise (Appendix C): log L = -1/2 sum_x w(x) (d - m)^2 / sigma^2.
// Parseval no longer makes this a sum over k, but the gradient is still sum_k
// Re[conj(R_k) dM_k / dtheta] / (sigma^2 N^2) with R = DFT(w (d - m)), so the half-plane
// pass of eval_logpost gives it when its data spectrum is replaced by the effective
// D' = M + R (scaled as the table).  The transforms run on the tensor cores (the layout
// and operand split are described with PixTc); one CTA evaluates two or four chains (G).

// Per galaxy (all threads): the A operands of the four products for this side into
// tensor memory (warp w writes lanes 32 (w mod 4) .. + 31, the high parts for w < 4 and
// the low parts otherwise), the further chains' copies of the table, and the stamp and
// its weights in shared memory.
template <int G>
__device__ void pix_tc_setup(const FitParams &P, const GalCtx &gc, const SmemView &sm, const PixTc &px, int gal)
{
    using Q = tc::Geo<G>;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = gc.N, c = gc.c, H = gc.H;
    const int row = 32 * (warp & 3) + lane;      // the TMEM lane this thread writes
    const bool lo = warp >= 4;
    const uint32_t tl = *px.tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    auto part = [&](float x) { const float h = tc::tf32_rn(x); return lo ? tc::tf32_rn(x - h) : h; };
    // [[C, -S], [S, C]]: row r = (p, a), column k = (q, b): p = q gives C, else -S (p = 0) or S
    const int p = row >> 6, a = row & 63;
    for (int k0 = 0; k0 < 2 * Q::KV && warp < 8; k0 += 8) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = k0 + j, q = k >= Q::KV, b = k - q * Q::KV;
            float co = 0.f, sn = 0.f;
            if (a < N && b < N) {
                int m = ((a - c) * (b - c)) % N;   // exact reduction of the phase index
                if (m < 0) m += N;
                sincospif(2.0f * (float)m / (float)N, &sn, &co);
            }
            v[j] = part(p == q ? co : (p == 0 ? -sn : sn));
        }
        tc::st8(tl + (lo ? Q::kColAFlo : Q::kColAF) + k0, v);
    }
    // the complex-to-real constant: rows ix < 64, K (re, u | im, u):
    // (w_u / N^2) (cos, -sin)(2 pi u (ix - c) / N); rows 64 + ix again, so that the model image
    // comes out in both halves of the accumulator's lanes
    const float wn = 1.0f / ((float)N * (float)N);
    for (int k0 = 0; k0 < 2 * Q::KU && warp < 8; k0 += 8) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = k0 + j, q = k >= Q::KU, u = k - q * Q::KU;
            float co = 0.f, sn = 0.f;
            if (a < N && u < H) {
                int m = (u * (a - c)) % N;
                if (m < 0) m += N;
                sincospif(2.0f * (float)m / (float)N, &sn, &co);
                const float wu = u ? 2.0f * wn : wn;
                co *= wu;
                sn *= wu;
            }
            v[j] = part(q ? -sn : co);
        }
        tc::st8(tl + (lo ? Q::kColA2lo : Q::kColA2) + k0, v);
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    const int nrow = gc.H * row_floats(P.npad);
    for (int i = tid; i < nrow; i += blockDim.x) {
        const float t = sm.tab[i];
#pragma unroll
        for (int g = 0; g < G - 1; ++g) px.tab1[(size_t)g * P.h_max * row_floats(P.npad) + i] = t;
    }
    const int64_t off = P.offsets[gal];
    const int n = N * N;
    for (int i = tid; i < n; i += blockDim.x) {
        px.dimg[i] = load_pix(P.data, P.data_f64, off + i);
        px.wimg[i] = __ldg(P.pix_w + off + i);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
}

// One 3xTF32 product into TMEM columns [0, N) (all threads; one lane of the first warp issues and
// commits, everyone waits for the given parity).  K runs over n_q halves of nk steps
// of 8: step (q, k) reads A at TMEM column a + q a_q + 8 k (its low part a_lo columns
// further) and B at b + q b_q + 288 k bytes (the data operand: leading offset 144 B,
// row groups sbo_b apart).  `failed` carries whether this thread's last wait gave up: the barrier
// before the issue shares it, and returns false for every thread (nothing issued, the CTA
// aborted with the previous product's parity pending).
struct TcGemm {
    uint32_t a, a_q, a_lo, b, b_q, sbo_b, id;
    int n_q, nk;
};
template <int CG>
__device__ __forceinline__ bool tc_run(const PixTc &px, const TcGemm &G, uint32_t parity, bool &failed)
{
    tc::fence_async_smem();
    tc::fence_before();
    if (__syncthreads_or(failed)) {
        if (threadIdx.x == 0) *px.abort = 2 + (int)(parity ^ 1u);
        return false;
    }
    const uint32_t bar = tc::saddr(px.bar);
    // The first warp as a whole runs the loop and one elected lane issues, so that the
    // descriptors stay in uniform registers: under a test of the thread index each of them was moved
    // there again for every MMA, about 50 cycles an MMA against 21 (400 galaxies of 41 px:
    // 101.0 -> 90.3 ms; unrolling the loop by four gave nothing on either form).
    if (__shfl_sync(BS_FULL_MASK, threadIdx.x >> 5, 0) == 0) {
        tc::fence_after();
        const uint32_t elected = tc::elect_one();
        const uint32_t tmem = __shfl_sync(BS_FULL_MASK, *px.tmem, 0);
        const uint32_t b_lo = tc::Geo<CG>::kBopFloats * 4;
        for (int q = 0; q < G.n_q; ++q) {
            // a k-step advances the B descriptor's start-address field (bytes / 16, the
            // low 14 bits; every address stays below 256 KB, so the field does not carry)
            uint32_t a = tmem + G.a + q * G.a_q;
            const uint32_t b0 = G.b + q * G.b_q;
            uint64_t bh = tc::sdesc(b0, tc::kLboB, G.sbo_b), bl = tc::sdesc(b0 + b_lo, tc::kLboB, G.sbo_b);
#pragma unroll 1
            for (int k = 0; k < G.nk; ++k) {
                tc::mma_ta(elected, tmem, a, bl, G.id, (q | k) ? 1u : 0u);
                tc::mma_ta(elected, tmem, a + G.a_lo, bh, G.id, 1u);
                tc::mma_ta(elected, tmem, a, bh, G.id, 1u);
                a += 8;
                bh += 288 / 16;
                bl += 288 / 16;
            }
        }
        tc::commit(elected, bar);
    }
    failed = !tc::wait_parity(bar, parity);
    tc::fence_after();
    return true;
}

__device__ __forceinline__ double pix_nan(float g[6])
{
#pragma unroll
    for (int i = 0; i < 6; ++i) g[i] = NAN;
    return NAN;
}

// The gradient of the log posterior of this group's chain from the half-plane pass on
// its effective spectrum, with the rows split over the group's four warps: warp j of
// the group sums the terms of its rows u in [r j, r (j + 1)), r even (the pass reads
// rows in pairs); the four warp sums meet in shared memory, where every thread of the
// group adds them in warp order and forms the gradient (the sums and the gradient of
// eval_logpost, exponential profile, no chi^2).  m: the model's shape at th.
template <int NC>
__device__ __forceinline__ void pix_grad(const FitParams &P, const GalCtx &gc, const Shape &m, const float *tab, const float2 *kxr, const PixTc &px,
                         float4 *xph, const float vcol[NC], const float th[6], float g[6])
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = warp >> 2, wj = warp & 3;
    const int per = 2 * ((gc.H + 7) >> 3);
    const int u0 = min(gc.H, wj * per), u1 = min(gc.H, u0 + per);
    float sums[6], chi_hi = 0.f, chi_lo = 0.f;
    spectral_sums<NC, false, 0>(P, gc, m, tab, kxr, xph, vcol, th, u0, u1, sums, chi_hi, chi_lo);
    float *gs = px.gsum + grp * 24;
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 6; ++k) gs[6 * wj + k] = sums[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 6; ++k) sums[k] = ((gs[k] + gs[6 + k]) + gs[12 + k]) + gs[18 + k];
    spectral_grad<0>(P, gc, m, sums, th, g);
}

// One evaluation of the G chains of the CTA (all threads; each group passes its own
// chain's th; a group with skip set passes any finite th and ignores the results).
// Returns the log posterior of the caller's chain if want_ll (the caller's group's
// flag), else 0; *all_done is set when all groups have raised their done flags (the
// evaluation then does nothing).
template <int NC, int G>
__device__ double eval_pix(const FitParams &P, const GalCtx &gc, const SmemView &sm, int gal, float4 *xph,
                           const float vcol[NC], const float th[6], float g[6], bool want_ll, bool *all_done)
{
    using Q = tc::Geo<G>;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = warp >> 2;                        // the chain of this thread's group
    const int L = 32 * (warp & 3) + lane;             // this thread's TMEM lane
    const int tg = tid & 127;                         // thread within the group
    const PixTc px = pix_tc_view<G>(sm.kxr, P.h_max, P.npad, P.max_side);
    const int N = gc.N, H = gc.H, c = gc.c;
    constexpr int npad = 32 * NC, rowf = 96 * NC;
    float *tab = grp ? px.tab1 + (size_t)(grp - 1) * P.h_max * rowf : sm.tab;
    const Shape ms = model_shape<0>(P, th);
    const float F = ms.F, E = ms.E, al = ms.al, be = ms.be, ga = ms.ga;
    __syncthreads();   // the previous evaluation's readers of the tables and buffers are done
    bool done = true;
#pragma unroll
    for (int q = 0; q < G; ++q) done = done && px.done[q];
    if (all_done) *all_done = done;
    if (done) return 0.0;
    if (*px.abort) return pix_nan(g);
    const float sqrt2 = 1.41421356237309515f;
    float *bh = px.bop, *bl = px.bop + Q::kBopFloats;
    constexpr int kLb = tc::kLboB / 4;
    const int ks = (N + 7) >> 3;          // k-steps of 8 covering the side
    const int n8 = 8 * ks;                // columns or rows of one chain over iy (or ix)
    const int h8 = 8 * ((H + 7) >> 3);    // and over u
    // (a) the model's half spectrum Mt into the chain's table D slots, and M = Mt /
    // scale_u as the operand of (1): rows (chain, u < h8), K (re, vi | im, vi); thread
    // tg of the group takes column vi = tg mod 64 and the rows u = tg / 64 + 2 i.  The row
    // phases X(u) are formed a lane each and passed by shuffles
    {
        const int vi = tg & 63, u0 = tg >> 6;
        const bool col = vi < N;
        int ox, oy, ot;
        slot_offsets(npad, col ? vi >> 5 : 0, col ? vi & 31 : 0, ox, oy, ot);
        const float ky = (float)(vi - c) * gc.dk;
        const float cst = fmaf(be * ky, ky, 1.0f), gky = ga * ky;
        float Xs, Xc, sy, cy;
        sincospi_sfu(-2.0f * th[4] * (float)lane * gc.invN, &Xs, &Xc);
        sincospi_sfu(-2.0f * th[5] * (float)(vi - c) * gc.invN, &sy, &cy);
        const float2 Y = make_float2(F * cy, F * sy);
        const float sN = (float)N, sN2 = (float)N * 0.70710678118654752f;
        // operand element (h8 grp + u, vi) of eight-row group ug, u = ug + u0 + 2 j
        const int eo = (vi >> 2) * kLb + (vi & 3) + u0 * 4;
#pragma unroll 1
        for (int ug = 0; ug < h8; ug += 8) {
            const int e0 = eo + ((h8 * grp + ug) >> 3) * (Q::KV / 2) * kLb;
            // every load of the four rows before the first store, which the compiler cannot move them over
            float T[4], kx[4];
            float2 X[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int u = ug + u0 + 2 * j, uc = min(u, H - 1);
                T[j] = tab[uc * rowf + ot];
                kx[j] = sm.kxr[uc].x;
                X[j] = make_float2(__shfl_sync(BS_FULL_MASK, Xc, u), __shfl_sync(BS_FULL_MASK, Xs, u));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int u = ug + u0 + 2 * j;
                const float s = fmaf(fmaf(al, kx[j], gky), kx[j], cst);
                const float rs = rsqrtf(s);
                const float A = T[j] * rs * rs * rs;
                const float mr = A * (X[j].x * Y.x - X[j].y * Y.y), mi = A * (X[j].x * Y.y + X[j].y * Y.x);
                const float inv_scale = u == 0 ? sN : sN2;
                const bool in = col && u < H;
                if (in) {
                    tab[u * rowf + ox] = mr;
                    tab[u * rowf + oy] = mi;
                }
                const float Mr = in ? mr * inv_scale : 0.f, Mi = in ? mi * inv_scale : 0.f;
                if (Q::KV == 64 || vi < Q::KV) {
                    tc::split_store(bh, bl, e0 + 8 * j, Mr);
                    tc::split_store(bh, bl, e0 + 8 * j + (Q::KV / 4) * kLb, Mi);   // K index KV + vi
                }
            }
        }
    }
    const uint32_t bop = tc::saddr(px.bop);
    const uint32_t tl = *px.tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    constexpr uint32_t aflo = Q::kColAFlo - Q::kColAF, a2lo = Q::kColA2lo - Q::kColA2;
    constexpr uint32_t core = tc::kLboB;                            // bytes of a core matrix
    constexpr uint32_t sbo_v2 = Q::KV / 2 * core, sbo_v = Q::KV / 4 * core, sbo_u2 = Q::KU / 2 * core;
    bool failed = false;
    // (1) G = M E for all chains: rows (re, iy | im, iy), columns (chain, u)
    if (!tc_run<G>(px, TcGemm{Q::kColAF, Q::KV, aflo, bop, Q::KV / 4 * core, sbo_v2, tc::idesc(128, G * h8), 2, ks}, 0,
                   failed))
        return pix_nan(g);
    // (1) -> operand of (2): row (chain, iy), K (re, u | im, u), G as it is (the weights
    // are in the constant); this thread's lane (p, iy), its chain's h8 columns
    {
        float v[32];
        tc::ld8n(tl + h8 * grp, h8 >> 3, v);
        const int p = L >> 6, iy = L & 63;
        if (iy < n8) {
            const int e0 = tc::op_index(n8 * grp + iy, p * Q::KU, 2 * Q::KU, kLb);
#pragma unroll
            for (int m = 0; m < 8; ++m)
                if (4 * m < h8)
                    tc::split_store4(bh, bl, e0 + m * kLb, v[4 * m], v[4 * m + 1], v[4 * m + 2], v[4 * m + 3]);
        }
    }
    // (2) m = W G: rows ix (twice), columns (chain, iy)
    if (!tc_run<G>(px, TcGemm{Q::kColA2, Q::KU, a2lo, bop, Q::KU / 4 * core, sbo_u2, tc::idesc(128, G * n8), 2,
                              (H + 7) >> 3},
                   1, failed))
        return pix_nan(g);
    // the residual and the operand of (3): rows (chain, iy), K ix; the group's warps 0 and 1
    // (lanes ix) take the first half of the eight-row groups, warps 2 and 3 (lanes 64 + ix) the rest
    {
        const int ix = L & 63;
        const int g0 = (L >> 6) ? (ks + 1) >> 1 : 0, ng = (L >> 6) ? ks >> 1 : (ks + 1) >> 1;
        const float *dp = px.dimg + 8 * g0 * N + ix, *wp = px.wimg + 8 * g0 * N + ix;
        int e0 = (ix >> 2) * kLb + (ix & 3) + (ks * grp + g0) * (Q::KV / 4) * kLb;
        // eight rows at a time, their loads before the first store.  Here and in the other steps between
        // products the warps waited for chains of shared-memory loads, each behind the last
        // element's stores, which the compiler must not move it over: a round of two chains at 41 px
        // took 17,800 cycles, 15,200 with the loads of a few elements ahead (four chains 10.6 -> 9.0
        // ms a launch of one wave; with the groups unrolled 12.2 ms, for want of registers)
#pragma unroll 1
        for (int q = 0; q < ng; ++q) {
            float m[32], d[8], w[8];
            tc::ld8n(tl + n8 * grp + 8 * (g0 + q), 1, m);
            const int left = ix < N ? N - 8 * (g0 + q) : 0;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                d[t] = t < left ? dp[t * N] : 0.f;
                w[t] = t < left ? wp[t * N] : 0.f;
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float r = t < left ? w[t] * (d[t] - m[t]) : 0.f;
                if (Q::KV == 64 || ix < Q::KV) tc::split_store(bh, bl, e0 + (t << 2), r);
            }
            dp += 8 * N;
            wp += 8 * N;
            e0 += Q::KV / 4 * kLb;
        }
    }
    // chi^2 (warps 0 and 1 of the group, all rows again: one evaluation of a trajectory):
    // compensated FP32 per thread over iy in order, FP64 across threads
    if (want_ll) {
        float c_hi = 0.f, c_lo = 0.f;
        if (L < 64) {
#pragma unroll 1
            for (int g8 = 0; g8 < ks; ++g8) {
                float m[32];
                tc::ld8n(tl + n8 * grp + 8 * g8, 1, m);
                float x[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const bool in = L < N && 8 * g8 + t < N;
                    const int e = in ? (8 * g8 + t) * N + L : 0;
                    const float res = px.dimg[e] - m[t];
                    x[t] = px.wimg[e] * res * res;
                }
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    if (L < N && 8 * g8 + t < N) {
                        float t_hi, t_lo;
                        two_sum(c_hi, x[t], t_hi, t_lo);
                        c_hi = t_hi;
                        c_lo += t_lo;
                    }
                }
            }
        }
        const double cw = warp_sum_d((double)c_hi + (double)c_lo);
        if (lane == 0) px.chi[warp] = cw;
    }
    // (3) conj Q = [C; S] r: rows (re, a | im, a), columns (chain, iy)
    if (!tc_run<G>(px, TcGemm{Q::kColAF, 0u, aflo, bop, 0u, sbo_v, tc::idesc(128, G * n8), 1, ks}, 0, failed))
        return pix_nan(g);
    // (3) -> operand of (4): row (chain, u = a - c < h8), K (re, iy | im, iy); this
    // thread's lane (q, a), its chain's n8 columns iy
    {
        const int q = L >> 6, u = (L & 63) - c;
#pragma unroll 1
        for (int y0 = 0; y0 < n8; y0 += 16) {
            float v[16];
            tc::ld16(tl + n8 * grp + y0, v);
            if (u >= 0 && u < h8) {
                const int e0 = tc::op_index(h8 * grp + u, q * Q::KV + y0, 2 * Q::KV, kLb);
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    if (y0 + 4 * m < n8)
                        tc::split_store4(bh, bl, e0 + m * kLb, v[4 * m], v[4 * m + 1], v[4 * m + 2], v[4 * m + 3]);
            }
        }
    }
    // (4) conj R = E conj Q: rows (re, vi | im, vi), columns (chain, u)
    if (!tc_run<G>(px, TcGemm{Q::kColAF, Q::KV, aflo, bop, Q::KV / 4 * core, sbo_v2, tc::idesc(128, G * h8), 2, ks}, 1,
                   failed))
        return pix_nan(g);
    // D' = Mt + scale_u R in the chain's table D slots; this thread's lane (p, vi), its
    // chain's columns u
    {
        const int p = L >> 6, vi = L & 63;
        float v[32];
        tc::ld8n(tl + h8 * grp, h8 >> 3, v);
        if (vi < N) {
            int ox, oy, ot;
            slot_offsets(npad, vi >> 5, vi & 31, ox, oy, ot);
            const int os = p ? oy : ox;
            const float sg = p ? -gc.invN : gc.invN;
#pragma unroll
            for (int u0 = 0; u0 < 32; u0 += 8) {
                if (u0 < H) {
                    float o[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (u0 + j < H) o[j] = tab[(u0 + j) * rowf + os];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (u0 + j < H)
                            tab[(u0 + j) * rowf + os] = fmaf((u0 + j ? sqrt2 : 1.0f) * sg, v[u0 + j], o[j]);
                }
            }
        }
    }
    if (__syncthreads_or(failed)) {
        if (threadIdx.x == 0) *px.abort = 2 + 1;
        return pix_nan(g);
    }
    // the gradient from the half-plane pass on the chain's effective spectrum, its rows
    // over the group's four warps
    pix_grad<NC>(P, gc, ms, tab, sm.kxr, px, xph, vcol, th, g);
    if (!want_ll) return 0.0;
    const double chi2 = px.chi[4 * grp] + px.chi[4 * grp + 1];
    const float lprior = P.prior_const - 0.5f * (th[4] * th[4] + th[5] * th[5]) * P.inv_sxy2 +
                         2.0f * log1pf(-E) - 0.5f * E * P.inv_se2;
    return -0.5 * chi2 * (double)gc.inv_b + (double)lprior;
}

// A group whose chain has no further evaluations (all threads of the group): raise
// its done flag, then join the other group's evaluations until both are done.
template <int NC, int G>
__device__ void pix_drain(const FitParams &P, const GalCtx &gc, const SmemView &sm, int gal, float4 *xph,
                          const float vcol[NC])
{
    const PixTc px = pix_tc_view<G>(sm.kxr, P.h_max, P.npad, P.max_side);
    if ((threadIdx.x & 127) == 0) px.done[threadIdx.x >> 7] = 1;
    const float th[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // any finite point: the results are not used
    float g[6];
    for (;;) {
        bool all = false;
        eval_pix<NC, G>(P, gc, sm, gal, xph, vcol, th, g, false, &all);
        if (all) break;
    }
}

// ---- A general dense pixel covariance (Appendix C, Eq. covar-pixel-likelihood):
// log L = -1/2 (d - m)^T P (d - m) with the precision P = Sigma^-1.  Its cost is the
// product y = P (d - m), N^4 multiply-adds per evaluation reading P from L2, beside
// which the two separable transforms are small; and P amplifies rounding errors of
// the rendered model m, so the transforms stay in FP32 on the CUDA cores (kernel
// instance PROF 4).  The gradient is the half-plane pass on the effective spectrum
// D' = M + DFT(y) (scaled as the table).
//
// A CTA runs a galaxy's chains (at most 4, or a share of them where there are SMs to
// spare: dense_chains_per_cta) on 16 warps, or on fewer where small stamps share an SM
// (dense_warps_for), one evaluation of every chain at a time: the first warp of each chain
// (its leader) runs the chain's logic, and all warps meet in dense_round, where one read of P
// serves every chain.  The transforms' rows are split over the warps of the chain, the product's
// columns over all warps; every output is summed by one lane in a fixed order, so a chain's
// draws depend neither on the others nor on the number of warps.  The product is bound by the read of P (778 KB at 21 px,
// from L2): 32 rows of loads are in flight per warp.
// 64 galaxies of 21 px, 4 chains x (100 + 100), L <= 8: 332 ms with a warp per chain that
// evaluated on its own (the product waiting for each row of P, transforms on 11 to 21 of 32
// lanes), 23.8 ms on 64 SMs with all chains of a galaxy in one CTA, 18.2 ms with two per CTA on
// 128, the same draws bit for bit.  The L1 holds part of P between rounds: its first rows kept
// in shared memory instead came out the same or slower (21 px 18.3 -> 19.4 ms, 13 px 8.56 -> 8.56).
//
// After the shared region, in floats: the twiddles exp(+2 pi i m / N) (max_side float2),
// the chains' requests, the residual images of the four chain slots interleaved (max_side^2
// float4), and per chain a private copy of the table ([h_max][3 npad]: the D slots hold the
// evaluation's effective spectrum, the T slots the transfer), the half-transformed
// image ([h_max][max_side] float2) and the product with the precision (max_side^2).
constexpr int kDenseWarps = 16;
constexpr int kDenseChains = 4;
__host__ __device__ __forceinline__ int dense_chain_floats(int h_max, int npad, int max_side)
{
    const int n = h_max * row_floats(npad) + 2 * h_max * max_side + max_side * max_side;
    return (n + 3) & ~3;
}
__host__ __device__ __forceinline__ int dense_tw_floats(int max_side) { return (2 * max_side + 3) & ~3; }
__host__ __device__ __forceinline__ size_t dense_region_bytes(int h_max, int npad, int max_side, int n_chains)
{
    return ((size_t)dense_tw_floats(max_side) + 8 * kDenseChains + 4 * (size_t)max_side * max_side +
            (size_t)n_chains * dense_chain_floats(h_max, npad, max_side)) *
           sizeof(float);
}
struct DenseView {
    float2 *tw;    // [max_side] exp(+2 pi i m / N)
    float *req;    // [4][8] per chain: theta (6), request (0 none, 1 gradient, 2 and log posterior)
    float4 *rb;    // [max_side^2] residuals d - m of the four chain slots
    float *chain0; // the chains' blocks, `stride` floats each:
    int stride, o_G, o_y;
    __device__ __forceinline__ float *tab(int c) const { return chain0 + (size_t)c * stride; }
    __device__ __forceinline__ float2 *G(int c) const   // [h_max][max_side]
    {
        return reinterpret_cast<float2 *>(tab(c) + o_G);
    }
    __device__ __forceinline__ float *yb(int c) const { return tab(c) + o_y; }   // [max_side^2] precision x residual
};
// kxr ends at h_max + 1 float2 after its start; the region follows, 16-byte aligned.
__device__ __forceinline__ DenseView dense_view(float2 *kxr, int h_max, int npad, int max_side)
{
    float *base = reinterpret_cast<float *>(kxr + ((h_max + 2) & ~1));
    DenseView v;
    v.tw = reinterpret_cast<float2 *>(base);
    v.req = base + dense_tw_floats(max_side);
    v.rb = reinterpret_cast<float4 *>(v.req + 8 * kDenseChains);
    v.chain0 = v.req + 8 * kDenseChains + 4 * max_side * max_side;
    v.stride = dense_chain_floats(h_max, npad, max_side);
    v.o_G = h_max * row_floats(npad);
    v.o_y = v.o_G + 2 * h_max * max_side;
    return v;
}

// Per-galaxy set-up of the dense path (all threads): the twiddles, no requests, zero
// residuals of the slots without a chain, and each chain's private table from the staged
// one (transfer, zero spectrum).
__device__ void dense_setup(const FitParams &P, const GalCtx &gc, const SmemView &sm, const DenseView &dv, int n_tables)
{
    const int tid = threadIdx.x, nth = blockDim.x;
    for (int m = tid; m < gc.N; m += nth) {
        float s, co;
        sincospif(2.0f * (float)m * gc.invN, &s, &co);
        dv.tw[m] = make_float2(co, s);
    }
    for (int i = tid; i < 8 * kDenseChains; i += nth) dv.req[i] = 0.f;
    for (int i = tid; i < gc.N * gc.N; i += nth) dv.rb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int nrow = gc.H * row_floats(P.npad);
    for (int t = 0; t < n_tables; ++t) {
        float *dst = dv.tab(t);
        for (int i = tid; i < nrow; i += nth) dst[i] = sm.tab[i];
    }
    __syncthreads();
}

// y = P r of every chain slot (all warps): the precision is symmetric, so y_a = sum_b
// P[b][a] r_b, and a warp takes 32 columns a at a time, each row b of them one coalesced
// load used for all slots (pairs of them in packed arithmetic).
template <int PAIRS>
__device__ __forceinline__ void dense_product(const FitParams &P, const GalCtx &gc, const DenseView &dv, int gal,
                                              int n_slots)
{
    constexpr int kAhead = 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int n = gc.N * gc.N;
    const float *__restrict__ Pg = P.pix_prec + P.prec_offs[gal];
    for (int a0 = 32 * warp; a0 < n; a0 += 32 * nwarp) {
        const int a = a0 + lane;
        const float *col = Pg + min(a, n - 1);
        float2 y[PAIRS];
#pragma unroll
        for (int c = 0; c < PAIRS; ++c) y[c] = make_float2(0.f, 0.f);
        auto term = [&](float p, const float4 &r) {
            y[0] = fma2(f2(p), make_float2(r.x, r.y), y[0]);
            if constexpr (PAIRS > 1) y[1] = fma2(f2(p), make_float2(r.z, r.w), y[1]);
        };
        const float4 *r = dv.rb;
        int b0 = 0;
        for (; b0 + kAhead <= n; b0 += kAhead) {
            float p[kAhead];
#pragma unroll
            for (int t = 0; t < kAhead; ++t) p[t] = __ldg(col + t * n);
            col += kAhead * n;
#pragma unroll
            for (int t = 0; t < kAhead; ++t) term(p[t], r[t]);
            r += kAhead;
        }
        {
            float p[kAhead];
#pragma unroll
            for (int t = 0; t < kAhead; ++t) p[t] = b0 + t < n ? __ldg(col + t * n) : 0.f;
#pragma unroll
            for (int t = 0; t < kAhead; ++t)
                if (b0 + t < n) term(p[t], r[t]);
        }
        if (a < n) {
#pragma unroll
            for (int c = 0; c < 2 * PAIRS; ++c)
                if (c < n_slots) dv.yb(c)[a] = (c & 1) ? y[c >> 1].y : y[c >> 1].x;
        }
    }
}

// The model image's half of a round, of one chain's rows u (all warps of the chain): (a) its
// half spectrum Mt into the D slots of the chain's table, (b1) its column transform into G,
// G(u, iy) of rows u > 0 as (2 Re, -2 Im) (an exact scaling: the row transform's factors).
// Row u = k + r nk of the chain's warp k; UB rows share a twiddle.
template <int UB>
__device__ __forceinline__ void dense_model(const FitParams &P, const GalCtx &gc, const SmemView &sm, const DenseView &dv,
                                            int s, int k, int nk)
{
    constexpr int rowf = 96;
    const int lane = threadIdx.x & 31;
    const int N = gc.N, H = gc.H, c = gc.c;
    float *tab = dv.tab(s);
    float2 *G = dv.G(s);
    const bool own = lane < N;
    const int x = min(lane, N - 1) - c, xs = x < 0 ? x + N : x;   // this lane's row, centred, and mod N
    float th[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) th[i] = dv.req[8 * s + i];
    const float F = exp10f(th[0]);
    const float r0 = exp10f(th[1]) * (1.0f / kHlrOverR0);
    const float r02 = r0 * r0;
    const float e1 = th[2], e2 = th[3];
    const float E = e1 * e1 + e2 * e2;
    const float Pq = 1.0f / (1.0f - E);
    const float al = r02 * (1.0f + E + 2.0f * e1) * Pq;
    const float be = r02 * (1.0f + E - 2.0f * e1) * Pq;
    const float ga = r02 * 4.0f * e2 * Pq;
    const float v = (float)(lane - c);
    float sy, cy;
    sincospi_sfu(-2.0f * th[5] * v * gc.invN, &sy, &cy);
    const float Yr = F * cy, Yi = F * sy;
    const float ky = v * gc.dk;
    const float cst = fmaf(be * ky, ky, 1.0f), gky = ga * ky;
    for (int ub = k; ub < H; ub += UB * nk) {
#pragma unroll
        for (int r = 0; r < UB; ++r) {
            const int u = ub + r * nk;
            if (u < H) {
                float *row = tab + u * rowf;
                const float kx = sm.kxr[u].x;
                const float sarg = fmaf(fmaf(al, kx, gky), kx, cst);
                const float rs = rsqrtf(sarg);
                const float A = row[64 + lane] * rs * rs * rs;
                float sx, cx;
                sincospi_sfu(-2.0f * th[4] * (float)u * gc.invN, &sx, &cx);
                const float Pr = cx * Yr - sx * Yi, Pi = cx * Yi + sx * Yr;
                const float mr = own ? A * Pr : 0.0f, mi = own ? A * Pi : 0.0f;
                *reinterpret_cast<float2 *>(row + 2 * lane) = make_float2(mr, mi);
                const float inv_scale = (float)N * (u == 0 ? 1.0f : 0.70710678118654752f);
                if (own) G[u * N + lane] = make_float2(mr * inv_scale, mi * inv_scale);
            }
        }
        __syncwarp();
        // G(u, iy) = sum_v M(u, v) exp(+2 pi i v (iy - c) / N), in place (lane = iy)
        float re[UB], im[UB];
        const float2 *g[UB];
#pragma unroll
        for (int r = 0; r < UB; ++r) {
            re[r] = im[r] = 0.f;
            g[r] = G + min(ub + r * nk, H - 1) * N;
        }
        int i1 = ((N - xs) * c) % N;     // -c (iy - c) mod N
#pragma unroll 2
        for (int vi = 0; vi < N; ++vi) {
            const float2 t = dv.tw[i1];
#pragma unroll
            for (int r = 0; r < UB; ++r) {
                const float2 mv = g[r][vi];
                re[r] = fmaf(mv.x, t.x, fmaf(-mv.y, t.y, re[r]));
                im[r] = fmaf(mv.x, t.y, fmaf(mv.y, t.x, im[r]));
            }
            i1 += xs;
            if (i1 >= N) i1 -= N;
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < UB; ++r) {
            const int u = ub + r * nk;
            if (u < H && own) G[u * N + lane] = u ? make_float2(2.0f * re[r], -2.0f * im[r]) : make_float2(re[r], im[r]);
        }
    }
}

// (b2) The chain's rows iy of m (lane = ix) and the residual r = d - m.
template <int UB>
__device__ __forceinline__ void dense_residual(const FitParams &P, const GalCtx &gc, const DenseView &dv, int gal, int s,
                                               int k, int nk)
{
    const int lane = threadIdx.x & 31;
    const int N = gc.N, H = gc.H, c = gc.c;
    const float2 *G = dv.G(s);
    const int x = min(lane, N - 1) - c, xs = x < 0 ? x + N : x;
    const int64_t off = P.offsets[gal];
    const float invN2 = gc.invN * gc.invN;
    for (int yb = k; yb < N; yb += UB * nk) {
        float acc[UB];
        const float2 *g[UB];
#pragma unroll
        for (int r = 0; r < UB; ++r) {
            g[r] = G + min(yb + r * nk, N - 1);
            acc[r] = g[r]->x;                    // u = 0 (real)
        }
        int i1 = xs;                             // u (ix - c) mod N, advanced per u
#pragma unroll 2
        for (int u = 1; u < H; ++u) {
            const float2 t = dv.tw[i1];
#pragma unroll
            for (int r = 0; r < UB; ++r) {
                const float2 gv = g[r][u * N];
                acc[r] = fmaf(gv.x, t.x, fmaf(gv.y, t.y, acc[r]));
            }
            i1 += xs;
            if (i1 >= N) i1 -= N;
        }
#pragma unroll
        for (int r = 0; r < UB; ++r) {
            const int iy = yb + r * nk;
            if (iy < N && lane < N)
                reinterpret_cast<float *>(dv.rb + iy * N + lane)[s] =
                    load_pix(P.data, P.data_f64, off + (int64_t)iy * N + lane) - acc[r] * invN2;
        }
    }
}

// The way back, of the chain's rows u: Q(u, iy) = sum_ix y(ix, iy) exp(-2 pi i u (ix - c) / N)
// (lane = iy), then (b3) D' = Mt + scale_u R(u, v), R(u, v) = sum_iy Q(u, iy) exp(-2 pi i v (iy - c)
// / N) (lane = v).
template <int UB>
__device__ __forceinline__ void dense_back(const GalCtx &gc, const DenseView &dv, int s, int k, int nk)
{
    constexpr int rowf = 96;
    const int lane = threadIdx.x & 31;
    const int N = gc.N, H = gc.H, c = gc.c;
    float *tab = dv.tab(s);
    float2 *G = dv.G(s);
    const bool own = lane < N;
    const int xl = min(lane, N - 1), x = xl - c, xs = x < 0 ? x + N : x;
    const float *yrow = dv.yb(s) + xl * N;
    for (int ub = k; ub < H; ub += UB * nk) {
        float re[UB], im[UB];
        int i1[UB], d1[UB];
        float2 *g[UB];
#pragma unroll
        for (int r = 0; r < UB; ++r) {
            const int u = min(ub + r * nk, H - 1);
            re[r] = im[r] = 0.f;
            i1[r] = (u * c) % N;                 // -u (ix - c) at ix = 0
            d1[r] = u ? N - u : 0;
            g[r] = G + u * N;
        }
#pragma unroll 2
        for (int ix = 0; ix < N; ++ix) {
            const float y = yrow[ix];
#pragma unroll
            for (int r = 0; r < UB; ++r) {
                const float2 t = dv.tw[i1[r]];
                re[r] = fmaf(y, t.x, re[r]);
                im[r] = fmaf(y, t.y, im[r]);
                i1[r] += d1[r];
                if (i1[r] >= N) i1[r] -= N;
            }
        }
#pragma unroll
        for (int r = 0; r < UB; ++r)
            if (ub + r * nk < H && own) g[r][lane] = make_float2(re[r], im[r]);
        __syncwarp();
        const int dk = xs ? N - xs : 0;
        int i2 = (xs * c) % N;                   // -v (iy - c) at iy = 0
#pragma unroll
        for (int r = 0; r < UB; ++r) re[r] = im[r] = 0.f;
#pragma unroll 2
        for (int iy = 0; iy < N; ++iy) {
            const float2 t = dv.tw[i2];
#pragma unroll
            for (int r = 0; r < UB; ++r) {
                const float2 q = g[r][iy];
                re[r] = fmaf(q.x, t.x, fmaf(-q.y, t.y, re[r]));
                im[r] = fmaf(q.x, t.y, fmaf(q.y, t.x, im[r]));
            }
            i2 += dk;
            if (i2 >= N) i2 -= N;
        }
#pragma unroll
        for (int r = 0; r < UB; ++r) {
            const int u = ub + r * nk;
            if (u < H && own) {
                const float scale = (u == 0 ? 1.0f : 1.41421356237309515f) * gc.invN;
                float2 *d = reinterpret_cast<float2 *>(tab + u * rowf) + lane;
                *d = make_float2(fmaf(scale, re[r], d->x), fmaf(scale, im[r], d->y));
            }
        }
    }
}

// One evaluation of every chain that asks for one (all threads of the CTA).  A leader
// (the first warp of chain `mine`) has its theta in th and passes active = true; every other warp,
// and a leader whose chain has ended, passes active = false.  Returns false when no
// chain asked (the evaluations of the galaxy are over); the leader receives its chain's
// log posterior in lp (if want_ll) and its lane's component of the gradient in gi.
template <int NC>
__device__ bool dense_round(const FitParams &P, const GalCtx &gc, const SmemView &sm, int gal, int n_slots, bool active,
                            int mine, const float vcol[NC], const float th[6], float &gi, bool want_ll, double &lp)
{
    static_assert(NC == 1, "stamps of at most 31 px: a lane is a row or a column of the stamp");
    const DenseView dv = dense_view(sm.kxr, P.h_max, P.npad, P.max_side);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int N = gc.N, H = gc.H;
    if (lane == 0 && warp < n_slots && warp == mine) {   // the leader of slot `mine` is warp `mine`
        float *q = dv.req + 8 * mine;
#pragma unroll
        for (int i = 0; i < 6; ++i) q[i] = active ? th[i] : 0.f;
        q[6] = active ? (want_ll ? 2.f : 1.f) : 0.f;
    }
    __syncthreads();
    bool any = false;
    for (int s = 0; s < n_slots; ++s) any = any || dv.req[8 * s + 6] != 0.f;
    if (!any) return false;
    // this warp's share of one chain: member k of the nk warps of chain s (warps past
    // nk n_slots take part in the product only); rows are taken in passes of as many as
    // share them evenly, four at most
    const int s = warp % n_slots, k = warp / n_slots, nk = nwarp / n_slots;
    const bool in = k < nk && dv.req[8 * s + 6] != 0.f;
    const int ub = (H + nk - 1) / nk;
    if (in) {
        if (ub <= 2) dense_model<2>(P, gc, sm, dv, s, k, nk);
        else if (ub == 3) dense_model<3>(P, gc, sm, dv, s, k, nk);
        else dense_model<4>(P, gc, sm, dv, s, k, nk);
    }
    __syncthreads();
    if (in) {
        if (ub <= 2) dense_residual<2>(P, gc, dv, gal, s, k, nk);
        else if (ub == 3) dense_residual<3>(P, gc, dv, gal, s, k, nk);
        else dense_residual<4>(P, gc, dv, gal, s, k, nk);
    }
    __syncthreads();
    if (n_slots <= 2) dense_product<1>(P, gc, dv, gal, n_slots);
    else dense_product<2>(P, gc, dv, gal, n_slots);
    __syncthreads();
    if (in) {
        if (ub <= 2) dense_back<2>(gc, dv, s, k, nk);
        else if (ub == 3) dense_back<3>(gc, dv, s, k, nk);
        else dense_back<4>(gc, dv, s, k, nk);
    }
    __syncthreads();
    if (!active) return true;
    // (c) the leader: the gradient from the half-plane pass on the effective spectrum, and
    // chi^2 = r.y
    float4 *xph = sm.xph + (size_t)mine * phase_stride(P.h_max);
    eval_logpost<NC, 0>(P, gc, dv.tab(mine), sm.kxr, xph, vcol, th, gi, false);
    lp = 0.0;
    if (want_ll) {
        double chi = 0.0;
        const float *yb = dv.yb(mine), *rb = reinterpret_cast<const float *>(dv.rb) + mine;
        for (int a = lane; a < N * N; a += 32) chi += (double)rb[4 * a] * (double)yb[a];
        const double chi2 = warp_sum_d(chi);
        const float E = th[2] * th[2] + th[3] * th[3];
        const float lprior = P.prior_const - 0.5f * (th[4] * th[4] + th[5] * th[5]) * P.inv_sxy2 +
                             2.0f * log1pf(-E) - 0.5f * E * P.inv_se2;
        lp = -0.5 * chi2 * (double)gc.inv_b + (double)lprior;
    }
    return true;
}

// Rounds without a chain of one's own, until no chain asks (a warp that leads none, or a
// leader whose chain has ended).
template <int NC>
__device__ void dense_join(const FitParams &P, const GalCtx &gc, const SmemView &sm, int gal, int n_slots, int mine,
                           const float vcol[NC])
{
    const float th[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float gi;
    double lp;
    while (dense_round<NC>(P, gc, sm, gal, n_slots, false, mine, vcol, th, gi, false, lp)) {
    }
}
