// Shear sampling phase on sm_103a (Sec. 3.2): one streaming pass over the
// interim samples evaluates Eq. likelihood-shear and its gradient.
//
// Per sample, with eps = (eps' - g)/(1 - g* eps') (inverse of
// Eq. shear-transform), U = |1 - g* eps'|^2, Q = |eps|^2 = |eps' - g|^2 / U and
// the identity 1 - |eps|^2 = (1 - |g|^2)(1 - |eps'|^2) / U, the log weight
// log p_e(eps | alpha) + log|d eps/d eps'| - log P0_e(eps') + b splits into a
// per-galaxy constant and
//   x = -kappa ln U - Q / (2 alpha^2) + |eps'|^2 / (2 sigma_e0^2)
//       [- 2 ln(1 - |eps'|^2) for the truncated Gaussian] + b,
// kappa = 4 for the (1-|e|^2)^2 exp(-|e|^2/2 alpha^2) family (2 from that
// factor, 2 from the Jacobian (1-|g|^2)^2 / U^2 of
// Eq. true-prior-jacobian-shear) and 2 for the truncated Gaussian.  Its
// derivatives are dx/dg_i = (-2/U) [du_i (Q/(2 alpha^2) - kappa) - n_i/(2 alpha^2)]
// with du_1 = ur e1 - vi e2, du_2 = ur e2 + vi e1, n = eps' - g, and
// dx/dalpha = Q / alpha^3.
//
// Each galaxy's K samples are read by a group of lanes: when K % 4 == 0 and the
// rows are 16-byte aligned, 4 lanes per galaxy read 12-sample chunks from tiles
// of 64 galaxies x 48 samples that the tensor memory accelerator streams into
// shared memory; otherwise 8 lanes per galaxy with scalar loads one chunk ahead.  The
// arithmetic runs on pairs of samples in packed FP32x2 instructions, x is
// kept in log2 units for the MUFU exp2, and the group keeps
// an online log-sum-exp (a reference log weight that may lag the running
// maximum by up to 32, sum of weights and weighted derivative sums), merged
// with shuffles.  Per-galaxy totals are
// accumulated in FP64 and written as per-block partials; a one-block kernel
// sums the partials in a fixed order (deterministic) and adds the
// per-galaxy constants.
#include <algorithm>
#include <atomic>
#include <cmath>

#include <cuda.h>            // CUtensorMap and its enums (types only: the encoder is looked up at run time)
#include <cudaTypedefs.h>    // PFN_cuTensorMapEncodeTiled

#include "bs_device.cuh"
#include "bs_internal.h"

namespace bs {

namespace {

constexpr int kGroup = 8;          // lanes per galaxy
constexpr int kShearThreads = 256;

// Hardware approximations with denormal flushing.  Their arguments here are
// normal numbers (U in (0, 4], 1 - |eps'|^2 >= 2^-24, sums of weights >= 1),
// or, for ex2, non-positive differences whose flushed results are weights
// below 2^-126 of the largest; so no range fix-ups are needed around them.
__device__ __forceinline__ float ex2_ftz(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float lg2_ftz(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_ftz(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Packed FP32x2 arithmetic: two samples per instruction, each half rounded
// like the scalar operation.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

// The point's constants from the launch's parameters into registers.  Left to the compiler they
// are loaded again at every use (two per packed operand), which took a fifth of the
// one-point pass's issue slots.
__device__ __forceinline__ void hold(float2 &v) { asm volatile("" : "+f"(v.x), "+f"(v.y)); }
__device__ __forceinline__ ShearConst held(const ShearConst &k)
{
    ShearConst c = k;
    hold(c.g1);
    hold(c.g2);
    hold(c.a2n);
    hold(c.an);
    hold(c.nan);
    hold(c.nk);
    hold(c.c0);
    hold(c.gg);
    return c;
}

// Two samples: the weight split as exp2(x) f, with x = c0 |eps'|^2 -
// a2 Q (+ b log2 e) the exponent and f the power of U the log term stands for:
//   BA14:               -4 log2 U                    -> f = (1/U)^4
//   truncated Gaussian: -2 log2 U - 2 log2(1 - |eps'|^2) -> f = (1/(U (1 - |eps'|^2)))^2
// (f lies in about [0.004, 16], so it cannot overflow a weight; no logarithm
// per sample), and the factors of the derivatives,
//   dx/dg_i = -2 rU c_i,  c_i = du_i (a Q - kappa) - a n_i,  n = eps' - g,
//   du_i = eps'_i - g_i |eps'|^2  (-1/2 dU/dg_i),
// regrouped as c_i = eps'_i p - g_i r with p = a Q - kappa - a and
// r = |eps'|^2 (a Q - kappa) - a, so that a galaxy's weighted sum of c_i is
// sum(w rU p eps'_i) - g_i sum(w rU r): three running sums instead of two
// per-sample factors c_i (2 fewer packed operations per pair of samples);
// the -2 is applied once per galaxy.  U = |1 - conj(g) eps'|^2 is taken in the
// Lagrange form 1 - 2 g.eps' + |g|^2 |eps'|^2 (U is near 1: no cancellation);
// n is formed explicitly (not expanded through |eps'|^2 - 2 g.eps' + |g|^2,
// which cancels when eps' is near g).
template <int FAMILY, bool HAS_B>
__device__ __forceinline__ void pair_terms(const ShearConst &c, float2 e1, float2 e2, float2 bv, float2 &x,
                                           float2 &fw, float2 &ru, float2 &pp, float2 &rr, float2 &q)
{
    const float2 Ep = fma2(e1, e1, mul2(e2, e2));
    const float2 ge = fma2(c.g1, e1, mul2(c.g2, e2));            // g.eps'
    const float2 U = fma2(c.gg, Ep, fma2(c.m2, ge, f2(1.0f)));
    const float2 n1 = sub2(e1, c.g1), n2 = sub2(e2, c.g2);
    const float2 Nn = fma2(n1, n1, mul2(n2, n2));
    float2 rU, f;
    if (FAMILY == BS_EPRIOR_TRUNC_GAUSS) {
        const float2 om = sub2(f2(1.0f), Ep);
        const float2 uo = mul2(U, om);
        const float2 r = make_float2(rcp_ftz(uo.x), rcp_ftz(uo.y));   // 1 / (U (1 - |eps'|^2))
        rU = mul2(r, om);
        f = mul2(r, r);
    } else {
        rU = make_float2(rcp_ftz(U.x), rcp_ftz(U.y));
        const float2 r2 = mul2(rU, rU);
        f = mul2(r2, r2);
    }
    const float2 Q = mul2(Nn, rU);
    float2 xx = fma2(c.c0, Ep, mul2(c.a2n, Q));
    if (FAMILY == BS_EPRIOR_TRUNC_GAUSS) {
        if (!(Q.x < c.r2)) xx.x = -INFINITY;
        if (!(Q.y < c.r2)) xx.y = -INFINITY;
    }
    if (HAS_B) xx = fma2(f2(kLog2e), bv, xx);
    const float2 aqk = fma2(c.an, Q, c.nk);
    pp = add2(aqk, c.nan);
    rr = fma2(Ep, aqk, c.nan);
    fw = f;
    ru = rU;
    q = Q;
    x = xx;
}

// One chunk: 4 consecutive samples of this lane.
struct Chunk {
    float4 e1, e2, b;
    bool full;     // all four samples exist
    int nvalid;
};

// Scalar loads of one chunk (any K, any alignment); missing samples are zero.
template <bool HAS_B>
__device__ __forceinline__ void load_chunk(const ShearLaunch &s, long long base, int k0, int K, Chunk &ch)
{
    ch.nvalid = k0 < K ? min(4, K - k0) : 0;
    ch.full = ch.nvalid == 4;
    float t1[4] = {0.f, 0.f, 0.f, 0.f}, t2[4] = {0.f, 0.f, 0.f, 0.f}, tb[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (r < ch.nvalid) {
            const long long j = base + k0 + r;
            t1[r] = __ldg(s.e1 + j);
            t2[r] = __ldg(s.e2 + j);
            if (HAS_B) tb[r] = __ldg(s.b + j);
        }
    }
    ch.e1 = make_float4(t1[0], t1[1], t1[2], t1[3]);
    ch.e2 = make_float4(t2[0], t2[1], t2[2], t2[3]);
    ch.b = make_float4(tb[0], tb[1], tb[2], tb[3]);
}

// Online log-sum-exp state of one lane (both halves share the reference).
struct Lse {
    float m;                 // the reference log2 weight
    float2 sw, t1, t2, tq;   // t_i: sum of weight rU p eps'_i
    float2 tr;               // sum of weight rU r
};

constexpr float kNoReference = -1e30f;

// Samples missing from a chunk (past K) get log weight -inf.
__device__ __forceinline__ void mask_missing(const Chunk &ch, float2 (&x)[2])
{
    if (ch.nvalid < 4) x[1].y = -INFINITY;
    if (ch.nvalid < 3) x[1].x = -INFINITY;
    if (ch.nvalid < 2) x[0].y = -INFINITY;
    if (ch.nvalid < 1) x[0].x = -INFINITY;
}

// The sums of a pair with weights e.
__device__ __forceinline__ void add_pair(Lse &L, float2 e, float2 e1, float2 e2, float2 ru, float2 pp, float2 rr,
                                         float2 qq)
{
    const float2 er = mul2(e, ru);
    const float2 erp = mul2(er, pp);
    L.sw = add2(L.sw, e);
    L.t1 = fma2(erp, e1, L.t1);
    L.t2 = fma2(erp, e2, L.t2);
    L.tr = fma2(er, rr, L.tr);
    L.tq = fma2(e, qq, L.tq);
}

// exp2(x + nm) f
__device__ __forceinline__ float2 pair_weight(float2 x, float2 nm, float2 f)
{
    const float2 d = add2(x, nm);
    return mul2(make_float2(ex2_ftz(d.x), ex2_ftz(d.y)), f);
}

// The first four samples of a galaxy (L as lse_reset leaves it): their largest log2 weight is the
// reference, unless every weight is zero.
template <int FAMILY, bool HAS_B>
__device__ __forceinline__ void eval_first(const ShearConst &c, const Chunk &ch, Lse &L)
{
    float2 x[2], fw[2], ru[2], pp[2], rr[2], qq[2];
    const float2 e1[2] = {make_float2(ch.e1.x, ch.e1.y), make_float2(ch.e1.z, ch.e1.w)};
    const float2 e2[2] = {make_float2(ch.e2.x, ch.e2.y), make_float2(ch.e2.z, ch.e2.w)};
    const float2 bb[2] = {make_float2(ch.b.x, ch.b.y), make_float2(ch.b.z, ch.b.w)};
#pragma unroll
    for (int h = 0; h < 2; ++h)
        pair_terms<FAMILY, HAS_B>(c, e1[h], e2[h], bb[h], x[h], fw[h], ru[h], pp[h], rr[h], qq[h]);
    const float mloc = fmaxf(fmaxf(x[0].x, x[0].y), fmaxf(x[1].x, x[1].y));
    if (mloc - L.m > 32.0f) L.m = mloc;
    const float2 nm = f2(-L.m);
#pragma unroll
    for (int h = 0; h < 2; ++h) add_pair(L, pair_weight(x[h], nm, fw[h]), e1[h], e2[h], ru[h], pp[h], rr[h], qq[h]);
}

template <int FAMILY, bool HAS_B>
__device__ __forceinline__ void eval_chunk(const ShearConst &c, const Chunk &ch, Lse &L)
{
    float2 x[2], fw[2], ru[2], pp[2], rr[2], qq[2];
    const float2 e1[2] = {make_float2(ch.e1.x, ch.e1.y), make_float2(ch.e1.z, ch.e1.w)};
    const float2 e2[2] = {make_float2(ch.e2.x, ch.e2.y), make_float2(ch.e2.z, ch.e2.w)};
    const float2 bb[2] = {make_float2(ch.b.x, ch.b.y), make_float2(ch.b.z, ch.b.w)};
#pragma unroll
    for (int h = 0; h < 2; ++h)
        pair_terms<FAMILY, HAS_B>(c, e1[h], e2[h], bb[h], x[h], fw[h], ru[h], pp[h], rr[h], qq[h]);
    if (!ch.full) mask_missing(ch, x);
    // The weights are taken against the lane's reference L.m, which may lag the
    // largest log2 weight seen by up to 32 (weights below 2^32 f, so sums of any
    // realistic K stay finite), so that the exponentials need not wait for this
    // chunk's maximum; only a larger jump (the first chunk of a galaxy, whose
    // reference starts at -1e30) rescales the sums and recomputes the chunk's
    // weights (from the samples: the first pass's exponents are not kept).
    const float2 nm = f2(-L.m);
    float2 ew[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 d = add2(x[h], nm);
        ew[h] = mul2(make_float2(ex2_ftz(d.x), ex2_ftz(d.y)), fw[h]);
    }
    const float mloc = fmaxf(fmaxf(x[0].x, x[0].y), fmaxf(x[1].x, x[1].y));
    if (mloc - L.m > 32.0f) {
        const float2 sc = f2(ex2_ftz(L.m - mloc));
        L.sw = mul2(L.sw, sc);
        L.t1 = mul2(L.t1, sc);
        L.t2 = mul2(L.t2, sc);
        L.tq = mul2(L.tq, sc);
        L.tr = mul2(L.tr, sc);
        L.m = mloc;
        float2 x2[2], f2w[2], u0, u1, u2, u3;
#pragma unroll
        for (int h = 0; h < 2; ++h) pair_terms<FAMILY, HAS_B>(c, e1[h], e2[h], bb[h], x2[h], f2w[h], u0, u1, u2, u3);
        if (!ch.full) mask_missing(ch, x2);
        const float2 nl = f2(-mloc);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 d = add2(x2[h], nl);
            ew[h] = mul2(make_float2(ex2_ftz(d.x), ex2_ftz(d.y)), f2w[h]);
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) add_pair(L, ew[h], e1[h], e2[h], ru[h], pp[h], rr[h], qq[h]);
}

// Four samples of a galaxy at one of several points, without a branch, so that consecutive quads and
// points overlap and the time does not depend on the data: the reference moves to the quad's largest
// log weight where that lies above it by more than 32, as in eval_chunk, and the sums are scaled by
// the weight between the two, which is 1 in most quads.  Four points of 50,000 x 300: 107-113 us at any
// alpha; with eval_chunk 107 us at alpha = 0.2 and 123-132 at 0.005, with a lane's samples taken again at
// the galaxy's end where a weight had jumped 101-104 and 305-315.
template <int FAMILY>
__device__ __forceinline__ void eval_quad(const ShearConst &c, const Chunk &ch, Lse &L)
{
    float2 x[2], fw[2], ru[2], pp[2], rr[2], qq[2];
    const float2 e1[2] = {make_float2(ch.e1.x, ch.e1.y), make_float2(ch.e1.z, ch.e1.w)};
    const float2 e2[2] = {make_float2(ch.e2.x, ch.e2.y), make_float2(ch.e2.z, ch.e2.w)};
#pragma unroll
    for (int h = 0; h < 2; ++h)
        pair_terms<FAMILY, false>(c, e1[h], e2[h], f2(0.f), x[h], fw[h], ru[h], pp[h], rr[h], qq[h]);
    const float mloc = fmaxf(fmaxf(x[0].x, x[0].y), fmaxf(x[1].x, x[1].y));
    const float m = mloc - L.m > 32.0f ? mloc : L.m;
    const float2 sc = f2(ex2_ftz(L.m - m)), nm = f2(-m);
    L.m = m;
    L.sw = mul2(L.sw, sc);
    L.t1 = mul2(L.t1, sc);
    L.t2 = mul2(L.t2, sc);
    L.tq = mul2(L.tq, sc);
    L.tr = mul2(L.tr, sc);
#pragma unroll
    for (int h = 0; h < 2; ++h) add_pair(L, pair_weight(x[h], nm, fw[h]), e1[h], e2[h], ru[h], pp[h], rr[h], qq[h]);
}

// Four samples of a galaxy after its first four, against the reference as it stands, for points whose weights
// cannot jump: an ellipticity in the unit disk has 0 <= Q < 1, so that x lies in (-a2, c0), and with
// a2 + c0 <= kMaxSpan (alpha >= 0.173 at sigma_e0 = 0.3) no sample is above another by more than eval_quad
// allows.  The bits are eval_quad's.  Four points of 50,000 x 300: 98-105 us.
constexpr float kMaxSpan = 32.0f;
template <int FAMILY>
__device__ __forceinline__ void eval_plain(const ShearConst &c, const Chunk &ch, Lse &L)
{
    const float2 nm = f2(-L.m);
    const float2 e1[2] = {make_float2(ch.e1.x, ch.e1.y), make_float2(ch.e1.z, ch.e1.w)};
    const float2 e2[2] = {make_float2(ch.e2.x, ch.e2.y), make_float2(ch.e2.z, ch.e2.w)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float2 x, fw, ru, pp, rr, qq;
        pair_terms<FAMILY, false>(c, e1[h], e2[h], f2(0.f), x, fw, ru, pp, rr, qq);
        add_pair(L, pair_weight(x, nm, fw), e1[h], e2[h], ru, pp, rr, qq);
    }
}

// A galaxy's first chunk (e1 at r, e2 a tile further) by eval_chunk, for a lane whose first four samples have no
// weight (the truncated Gaussian's far samples) and set no reference for eval_plain.
template <int FAMILY>
__device__ __noinline__ Lse first_chunk(const ShearConst &c, const float *r, int n_quads);

// A galaxy's sum of weights that is not below this (or NaN) has left the range of a float all the same: the
// whole first chunk of a lane had no weight (the truncated Gaussian's far samples), or samples lie on or
// outside the unit circle.  The galaxy is then taken again by eval_chunk (replay_galaxy).
constexpr float kMost = 0x1p100f;

// Merge the lanes of a galaxy's group and add the galaxy's terms, times the galaxy's weight
// w[n] (1 when w is NULL; a zero weight drops the galaxy), to the accumulators of the
// group's first four lanes: lane 0 the log-sum-exp (log2), lanes 1-3 the softmax-weighted
// derivative sums, each lane one of them: the FP64 pipe takes 16 cycles an operation for the
// whole SM, so the four go through it side by side.  (g1, g2) is the shear of the evaluation.  Returns the
// galaxy's sum of weights.
template <int G = kGroup>
__device__ __forceinline__ float finish_galaxy(const Lse &L, float g1, float g2, unsigned gmask, int sub,
                                              const float *w, long long n, double &acc)
{
    float m = L.m;
    const float tr = L.tr.x + L.tr.y;
    float sw = L.sw.x + L.sw.y, tq = L.tq.x + L.tq.y;
    float t1 = fmaf(-g1, tr, L.t1.x + L.t1.y), t2 = fmaf(-g2, tr, L.t2.x + L.t2.y);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        const float mo = __shfl_xor_sync(gmask, m, o, G);
        const float so = __shfl_xor_sync(gmask, sw, o, G);
        const float o1 = __shfl_xor_sync(gmask, t1, o, G);
        const float o2 = __shfl_xor_sync(gmask, t2, o, G);
        const float oq = __shfl_xor_sync(gmask, tq, o, G);
        const float mn = fmaxf(m, mo);
        const float ca = ex2_ftz(m - mn), cb = ex2_ftz(mo - mn);
        sw = sw * ca + so * cb;
        t1 = t1 * ca + o1 * cb;
        t2 = t2 * ca + o2 * cb;
        tq = tq * ca + oq * cb;
        m = mn;
    }
    if (sub >= 4) return sw;
    const float wf = w ? __ldg(w + n) : 1.0f;
    if (wf == 0.0f) return sw;
    if (sw > 0.f) {
        const float inv = 1.0f / sw;
        const float d = sub == 1 ? -2.0f * t1 * inv : sub == 2 ? -2.0f * t2 * inv : tq * inv;
        // lane 0: m + log2(sw), the other lanes d + 0
        int e;
        // log2 of the sum of weights: the exponent exactly and the mantissa's logarithm, in [-1, 0),
        // to about 6e-8 by the accurate log2f.  The hardware approximation's absolute error
        // (about 2^-22, the same sign for sums of the same size) would add up over
        // 10^6 galaxies to a shift of the total of a few tenths of a nat.
        const float l = log2f(frexpf(sw, &e));
        double v = (double)(sub == 0 ? m : d);
        if (sub == 0) v += (double)e + (double)l;
        if (w) v *= (double)wf;
        acc += v;
    } else if (sub == 0) {
        acc = -INFINITY;
    }
    return sw;
}

__device__ __forceinline__ void lse_reset(Lse &L)
{
    L.m = kNoReference;
    L.sw = L.t1 = L.t2 = L.tq = L.tr = f2(0.f);
}

// Galaxy n at point p by the group's lanes, each its samples of the tile kernels' assignment (12 of every 48)
// by eval_chunk; this lane's term as finish_galaxy adds it.
template <int FAMILY>
__device__ __noinline__ double replay_galaxy(const ShearMultiLaunch &m, int p, long long n, int sub, unsigned gmask);

// Block reduction of the lanes' FP64 accumulators (quantity = lane of the group of G, the
// first four) into this block's partials.
template <int G>
__device__ __forceinline__ void block_partials(const ShearLaunch &s, double acc)
{
    __shared__ double red[kShearThreads / 32][4];
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o >= G; o >>= 1) acc += __shfl_xor_sync(BS_FULL_MASK, acc, o);
    if (lane < 4) red[threadIdx.x >> 5][lane] = acc;
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = 0.0;
        for (int i = 0; i < kShearThreads / 32; ++i) t += red[i][threadIdx.x];
        s.partials[(size_t)blockIdx.x * 4 + threadIdx.x] = t;
    }
}

// Any K and alignment: scalar loads into two register buffers in turn (the
// next chunk's loads in flight while the current one is evaluated).
template <int FAMILY, bool HAS_B>
__global__ void __launch_bounds__(kShearThreads, 3) shear_kernel(const __grid_constant__ ShearLaunch s)
{
    const int lane = threadIdx.x & 31;
    const int sub = lane & (kGroup - 1);
    const unsigned gmask = 0xFFu << (lane & ~(kGroup - 1));
    const long long group = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kGroup;
    const long long ngroups = (long long)gridDim.x * blockDim.x / kGroup;
    const ShearConst c = s.c;      // (a copy: read through a reference the constants cost 116 bytes of spills, not 52)
    const int K = s.K;
    double acc = 0.0;

    for (long long n = group; n < s.n_gal; n += ngroups) {
        const long long base = n * (long long)K;
        Lse L;
        lse_reset(L);
        Chunk A, B;
        int k0 = 4 * sub;
        load_chunk<HAS_B>(s, base, k0, K, A);
        for (;;) {
            if (k0 >= K) break;
            load_chunk<HAS_B>(s, base, k0 + 4 * kGroup, K, B);
            eval_chunk<FAMILY, HAS_B>(c, A, L);
            k0 += 4 * kGroup;
            if (k0 >= K) break;
            load_chunk<HAS_B>(s, base, k0 + 4 * kGroup, K, A);
            eval_chunk<FAMILY, HAS_B>(c, B, L);
            k0 += 4 * kGroup;
        }
        finish_galaxy(L, s.g1, s.g2, gmask, sub, s.w, n, acc);
    }
    block_partials<kGroup>(s, acc);
}

constexpr int kAGroup = 4;     // lanes per galaxy of the tile-streamed kernels
constexpr int kChunk = 12;     // samples per lane per chunk
constexpr int kQuads = kChunk / 4;

// ---- Tensor-memory-accelerator tiles (K a multiple of 4, 16-byte aligned rows): a CTA streams
// tiles of kTileG consecutive galaxies x kTileK samples of e1 and e2 (and b) with 2-D
// cp.async.bulk.tensor loads into a ring of three stages; one thread issues the
// loads of a stage and arms the stage's mbarrier with their byte count, and the
// others wait on it.  Thread t serves galaxy t / 4 of the tile and its samples
// [12 (t mod 4), + 12) of each chunk.  Galaxies past n_gal and samples past K arrive zero-filled and
// are masked by index.  A wait gives up after two seconds: the CTA then writes NaN
// partials, so that the pass's value is NaN.
constexpr int kTileG = kShearThreads / kAGroup;   // 64 galaxies per tile
constexpr int kTileK = kChunk * kAGroup;          // 48 samples per chunk
constexpr int kTmaStages = 3;
// Launch bounds for 2 CTAs per SM, of whose 128 registers the compiler takes 78: without b 3 CTAs are
// resident and nothing is rebuilt or spilled.  10^6 x 300: 446 us so (5.4 TB/s), 472 us bounded
// for 3 CTAs, 476 us before the constants were held, 539 us with 4 stages (2 CTAs fit).
// With b, 3.6 GB, 2 CTAs fit: 580-600 us; 610 us with two stages, which let 3 in; 709 us through
// per-lane cp.async copies, whose kernel this replaced.  What is left is the memory: the
// warps' waits find their tile late, and deeper rings per warp or L2 prefetches of whole tiles made
// the pass without b slower (516-690 us).
constexpr int kTmaBlocks = 2;
constexpr int kTileFloats = kTileG * kTileK;      // one array's box, 12 KB

__host__ __device__ constexpr size_t tma_smem_bytes(bool has_b)
{
    return (size_t)kTmaStages * (has_b ? 3 : 2) * kTileFloats * sizeof(float) + 128;   // + alignment of the ring
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Wait for the phase of the given parity.  Each try_wait may suspend the warp
// in hardware for up to 20 us until the phase completes (no busy loop taking
// issue slots from the computing warps).  The clock for the limit of two seconds is
// read only once a try has failed: most waits find their phase complete.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    uint64_t t0 = 0;
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(20000u)
            : "memory");
        if (ok) return true;
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t0 == 0) t0 = t;
        if (t - t0 > 2000000000ull) return false;
    }
}

// The CTA's ring of kStages stages, each one tile-chunk of NV arrays (e1, e2 and b), with a
// "full" mbarrier per stage (armed by the producer with the stage's byte count) and an
// "empty" one (one arrival per warp once the warp has read the stage).  Thread 0 is
// the producer: it issues item i (tile blockIdx.x + t gridDim.x, chunk c) after the
// stage's previous item has been released.  Every wait gives up after two seconds.
template <int NV>
struct TmaRing {
    static constexpr int kStages = kTmaStages;
    float *ring;
    uint64_t *full, *empty;
    int cpg, n_items;
    // producer state (thread 0): next item to load, its tile and chunk
    int p_item = 0, p_chunk = 0;
    long long p_tile;
    bool p_ok = true;

    __device__ void init(unsigned char *raw, uint64_t *f, uint64_t *e, long long n_gal, int K)
    {
        constexpr int kWarps = kShearThreads / 32;
        ring = reinterpret_cast<float *>(raw + ((128u - (smem_u32(raw) & 127u)) & 127u));
        full = f;
        empty = e;
        cpg = (K + kTileK - 1) / kTileK;   // chunks per tile
        const long long n_tiles = (n_gal + kTileG - 1) / kTileG;
        const int my_tiles = blockIdx.x < n_tiles ? (int)((n_tiles - 1 - blockIdx.x) / gridDim.x + 1) : 0;
        n_items = my_tiles * cpg;
        p_tile = blockIdx.x;
        if (threadIdx.x == 0) {
            for (int st = 0; st < kStages; ++st) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[st])) : "memory");
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&empty[st])), "r"(kWarps)
                             : "memory");
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();
    }
    __device__ void issue(const CUtensorMap *m1, const CUtensorMap *m2, const CUtensorMap *m3)
    {
        if (p_item >= n_items || !p_ok) return;
        const int st = p_item % kStages;
        if (p_item >= kStages) {   // the stage's previous item has been read by every warp
            if (!mbar_wait(smem_u32(&empty[st]), (uint32_t)((p_item / kStages - 1) & 1))) {
                p_ok = false;
                return;
            }
        }
        const uint32_t bar = smem_u32(&full[st]);
        const uint32_t d = smem_u32(ring + (size_t)st * NV * kTileFloats);
        const int x = p_chunk * kTileK, y = (int)(p_tile * kTileG);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"((uint32_t)(NV * kTileFloats * 4))
                     : "memory");
        const CUtensorMap *maps[3] = {m1, m2, m3};
#pragma unroll
        for (int v = 0; v < NV; ++v)
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
                    "r"(d + v * kTileFloats * 4),
                "l"(maps[v]), "r"(x), "r"(y), "r"(bar)
                : "memory");
        ++p_item;
        if (++p_chunk == cpg) {
            p_chunk = 0;
            p_tile += gridDim.x;
        }
    }
    // all threads: wait until item's stage has landed (false, in every lane, on a timeout)
    __device__ bool wait_full(int item) const
    {
        return __all_sync(BS_FULL_MASK,
                          mbar_wait(smem_u32(&full[item % kStages]), (uint32_t)((item / kStages) & 1)));
    }
    // all threads of a warp, after reading item's stage
    __device__ void release(int item) const
    {
        __syncwarp();
        if ((threadIdx.x & 31) == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&empty[item % kStages]))
                         : "memory");
    }
    // all threads, at the end: loads still in flight land in the ring (waited for, with the limit)
    __device__ void drain() const
    {
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int it = p_item - kStages; it < p_item; ++it)
                if (it >= 0) mbar_wait(smem_u32(&full[it % kStages]), (uint32_t)((it / kStages) & 1));
        }
    }
};

// Quad h (4 consecutive samples) of this thread's part of a chunk of its galaxy (4 lanes
// per galaxy, 12 samples each) in item's stage, and how many quads of it lie below K.
template <int NV>
__device__ __forceinline__ const float *tma_row(const TmaRing<NV> &R, int item)
{
    const int tid = threadIdx.x, sub = tid & (kAGroup - 1), gl = tid / kAGroup;
    return R.ring + (size_t)(item % TmaRing<NV>::kStages) * NV * kTileFloats + gl * kTileK + kChunk * sub;
}
template <int NV>
__device__ __forceinline__ Chunk tma_quad(const TmaRing<NV> &R, int item, int h)
{
    const float *r1 = tma_row(R, item) + 4 * h;
    Chunk ch;
    ch.nvalid = 4;
    ch.full = true;
    ch.e1 = *reinterpret_cast<const float4 *>(r1);
    ch.e2 = *reinterpret_cast<const float4 *>(r1 + kTileFloats);
    ch.b = NV == 3 ? *reinterpret_cast<const float4 *>(r1 + 2 * kTileFloats) : make_float4(0.f, 0.f, 0.f, 0.f);
    return ch;
}
__device__ __forceinline__ int tma_quads(int K, int chunk)
{
    const int left = (K - chunk * kTileK - kChunk * (int)(threadIdx.x & (kAGroup - 1)) + 3) >> 2;
    return left < 0 ? 0 : left < kQuads ? left : kQuads;
}

template <int FAMILY, bool HAS_B>
__global__ void __launch_bounds__(kShearThreads, kTmaBlocks)
    shear_kernel_tma(const __grid_constant__ ShearLaunch s, const __grid_constant__ CUtensorMap m1,
                     const __grid_constant__ CUtensorMap m2, const __grid_constant__ CUtensorMap m3)
{
    extern __shared__ __align__(128) unsigned char tma_raw[];
    constexpr int NV = HAS_B ? 3 : 2, NS = kTmaStages;
    __shared__ __align__(8) uint64_t full[NS], empty[NS];
    __shared__ int s_fail;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int sub = tid & (kAGroup - 1), gl = tid / kAGroup;
    const unsigned gmask = ((1u << kAGroup) - 1u) << (lane & ~(kAGroup - 1));
    const ShearConst c = held(s.c);
    const int K = s.K;
    if (tid == 0) s_fail = 0;
    TmaRing<NV> R;
    R.init(tma_raw, full, empty, s.n_gal, K);   // (its barrier also orders the reset above)
    if (tid == 0)
        for (int t = 0; t < NS - 1; ++t) R.issue(&m1, &m2, &m3);
    double acc = 0.0;
    Lse L;
    lse_reset(L);
    bool failed = false;
    int chunk = 0;
    long long tile = blockIdx.x;
    for (int item = 0; item < R.n_items; ++item) {
        if (tid == 0) R.issue(&m1, &m2, &m3);
        if (!R.wait_full(item)) {
            failed = true;
            break;
        }
        const long long n = tile * kTileG + gl;
        if (n < s.n_gal) {
            const int nq = tma_quads(K, chunk);
            if (chunk == 0) {
                if (nq > 0) eval_first<FAMILY, HAS_B>(c, tma_quad(R, item, 0), L);
            } else if (nq > 0) {
                eval_chunk<FAMILY, HAS_B>(c, tma_quad(R, item, 0), L);
            }
#pragma unroll
            for (int h = 1; h < kQuads; ++h)
                if (h < nq) eval_chunk<FAMILY, HAS_B>(c, tma_quad(R, item, h), L);
        }
        R.release(item);
        if (++chunk == R.cpg) {
            if (n < s.n_gal) finish_galaxy<kAGroup>(L, s.g1, s.g2, gmask, sub, s.w, n, acc);
            lse_reset(L);
            chunk = 0;
            tile += gridDim.x;
        }
    }
    if (failed || (tid == 0 && !R.p_ok)) s_fail = 1;
    R.drain();                                  // (begins with a barrier)
    block_partials<kAGroup>(s, s_fail ? NAN : acc);
}

template <int FAMILY>
__device__ __noinline__ Lse first_chunk(const ShearConst &c, const float *r, int n_quads)
{
    Lse L;
    lse_reset(L);
    Chunk ch;
    ch.nvalid = 4;
    ch.full = true;
    ch.b = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int h = 0; h < n_quads; ++h) {
        ch.e1 = *reinterpret_cast<const float4 *>(r + 4 * h);
        ch.e2 = *reinterpret_cast<const float4 *>(r + kTileFloats + 4 * h);
        eval_chunk<FAMILY, false>(c, ch, L);
    }
    return L;
}

template <int FAMILY>
__device__ __noinline__ double replay_galaxy(const ShearMultiLaunch &m, int p, long long n, int sub, unsigned gmask)
{
    const ShearLaunch &s = m.s;
    Lse L;
    lse_reset(L);
    const long long base = n * (long long)s.K;
    for (int k0 = kChunk * sub; k0 < s.K; k0 += kTileK)
        for (int k = k0; k < k0 + kChunk && k < s.K; k += 4) {
            Chunk ch;
            load_chunk<false>(s, base, k, s.K, ch);
            eval_chunk<FAMILY, false>(m.c[p], ch, L);
        }
    __syncwarp(gmask);
    double t = 0.0;
    finish_galaxy<kAGroup>(L, m.g1[p], m.g2[p], gmask, sub, s.w, n, t);
    return t;
}

// The tensor-map encoder of the driver, looked up once through the runtime
// (no link to the driver library).
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// A [n_gal][K] FP32 row-major array as a 2-D tensor map with kTileK x kTileG boxes.
bool make_sample_map(CUtensorMap &m, const float *base, long long n_gal, int K)
{
    auto enc = tensor_map_encoder();
    if (!enc || n_gal <= 0 || n_gal > 0xFFFFFFFFll) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)n_gal};
    const cuuint64_t strides[1] = {(cuuint64_t)K * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)kTileK, (cuuint32_t)kTileG};
    const cuuint32_t estr[2] = {1, 1};
    return enc(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Sum the partials of a point (n_part blocks of 4) and add the per-galaxy constants: a warp per
// quantity, so that the blocks' partials are read in one round trip and no barrier is
// needed; a fixed order.
__device__ __forceinline__ void finalize_point(const double *partials, int n_part, const double *add, double alpha_scale,
                                               double *out)
{
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double t = 0.0;
#pragma unroll 8
    for (int i = lane; i < n_part; i += 32) t += partials[(size_t)i * 4 + k];
    t = warp_sum_d(t);
    if (lane == 0) out[k] = t * (k == 0 ? 0.6931471805599453 : k == 3 ? alpha_scale : 1.0) + add[k];
}

struct ShearFinalize {
    double add[4], alpha_scale;
};
__global__ void __launch_bounds__(128) shear_finalize_kernel(const double *partials, int n_part,
                                                             const __grid_constant__ ShearFinalize f, double *out)
{
    finalize_point(partials, n_part, f.add, f.alpha_scale, out);
}

__global__ void __launch_bounds__(128) shear_finalize_batch_kernel(const double *partials, size_t part_stride, int n_part,
                                                                   const __grid_constant__ ShearFinalizeBatch f,
                                                                   double *out)
{
    const int q = blockIdx.x;
    finalize_point(partials + q * part_stride, n_part, f.add[q], f.alpha_scale[q], out + 4 * q);
}

// ---- all properties free ----------------------------------------------------

// log Phi(t) and the inverse Mills ratio phi(t)/Phi(t) of the standard normal,
// through erfcx on the left tail so that neither underflows.  On the right, 1 - Phi = q below
// 2^-25 makes 1 - q round to 1 and log1p(-q) to -q (from t = 6), and from t = 14.5 on both q
// and phi underflow to 0: the shorter forms give the bits of the general one.
__device__ __forceinline__ void log_ndtr_mills(float t, float &lphi, float &r)
{
    if (t < 0.0f) {
        const float u = -t * 0.70710678118654752f;
        const float ex = erfcxf(u);                 // exp(u^2) erfc(u)
        lphi = logf(0.5f * ex) - u * u;
        r = 0.79788456080286536f / ex;              // sqrt(2/pi) / erfcx
    } else if (t >= 14.5f) {
        lphi = -0.0f;
        r = 0.0f;
    } else {
        const float q = 0.5f * erfcf(t * 0.70710678118654752f);   // 1 - Phi(t)
        const float ph = 0.39894228040143268f * expf(-0.5f * t * t);
        if (t >= 6.0f) {
            lphi = -q;
            r = ph;
        } else {
            lphi = log1pf(-q);
            r = ph / (1.0f - q);
        }
    }
}

// The running sums of one lane, in pairs for the packed arithmetic: the reference log2 weight, the
// sum of weights, (t1, t2) on the shear, (sum w Q, sum w y), and sum w of (z - a r, z (z - a r)),
// (r z, y^2).
struct FullAcc {
    float m, sw;
    float2 t, qy, h01, h24;
};

// Two samples of a lane in packed arithmetic (each half rounded like the scalar
// operation): log2 weight of the ellipticity part (as pair_terms, with the logarithm) plus
// the flux/size log prior ratio up to per-galaxy constants,
//   -z^2/2 + log Phi(a z) - y^2/2,  z = (lf - mu_f)/sigma_f, y = (ls - mu_s)/sigma_s,
// and the factors of its derivatives (times sigma where that is constant):
//   (z - a r), z (z - a r), r z, y, y^2,  r = phi(a z)/Phi(a z);
// then the two samples in turn into the sums.  na, nb: (log Phi, r, z) of the two.
template <int FAMILY>
__device__ __forceinline__ void full_pair(const ShearFullLaunch &f, const ShearConst &c, float2 e1, float2 e2, float2 ls,
                                          const float4 &na, const float4 &nb, int n_valid, FullAcc &A)
{
    const float2 Ep = fma2(e1, e1, mul2(e2, e2));
    const float2 ge = fma2(c.g1, e1, mul2(c.g2, e2));
    const float2 U = fma2(c.gg, Ep, fma2(f2(-2.0f), ge, f2(1.0f)));   // Lagrange form
    const float2 n1 = sub2(e1, c.g1), n2 = sub2(e2, c.g2);
    const float2 rU = make_float2(rcp_ftz(U.x), rcp_ftz(U.y));
    const float2 Q = mul2(fma2(n1, n1, mul2(n2, n2)), rU);
    const float2 larg = FAMILY == BS_EPRIOR_TRUNC_GAUSS ? mul2(U, sub2(f2(1.0f), Ep)) : U;
    const float lgk = FAMILY == BS_EPRIOR_TRUNC_GAUSS ? -2.0f : -4.0f;    // -kappa of the family
    const float2 lg = make_float2(lg2_ftz(larg.x), lg2_ftz(larg.y));
    float2 x = fma2(c.c0, Ep, fma2(f2(lgk), lg, mul2(c.a2n, Q)));
    if (FAMILY == BS_EPRIOR_TRUNC_GAUSS) {
        if (!(Q.x < c.r2)) x.x = -INFINITY;
        if (!(Q.y < c.r2)) x.y = -INFINITY;
    }
    const float2 aqk = fma2(c.an, Q, c.nk);
    const float2 du1 = fma2(f2(-f.s.g1), Ep, e1), du2 = fma2(f2(-f.s.g2), Ep, e2);
    const float2 c1 = fma2(du1, aqk, mul2(c.nan, n1)), c2 = fma2(du2, aqk, mul2(c.nan, n2));
    const float2 lphi = make_float2(na.x, nb.x), r = make_float2(na.y, nb.y), z = make_float2(na.z, nb.z);
    const float2 y = mul2(sub2(ls, f2(f.mu_s)), f2(f.inv_ss));
    const float2 yy = mul2(y, y);
    x = fma2(f2(kLog2e), fma2(f2(-0.5f), fma2(z, z, yy), lphi), x);
    const float2 h0 = fma2(f2(-f.a_f), r, z);
    const float2 zh = mul2(z, h0), rz = mul2(r, z);
    auto add = [&](float xs, float q, float ru, float d1, float d2, float v0, float v1, float v2, float vy, float vyy) {
        if (xs > A.m) {
            const float2 sc = f2(ex2_ftz(A.m - xs));
            A.sw *= sc.x;
            A.t = mul2(A.t, sc);
            A.qy = mul2(A.qy, sc);
            A.h01 = mul2(A.h01, sc);
            A.h24 = mul2(A.h24, sc);
            A.m = xs;
        }
        const float e = ex2_ftz(xs - A.m);
        A.sw += e;
        A.t = fma2(f2(e * ru), make_float2(d1, d2), A.t);
        A.qy = fma2(f2(e), make_float2(q, vy), A.qy);
        A.h01 = fma2(f2(e), make_float2(v0, v1), A.h01);
        A.h24 = fma2(f2(e), make_float2(v2, vyy), A.h24);
    };
    if (n_valid > 0) add(x.x, Q.x, rU.x, c1.x, c2.x, h0.x, zh.x, rz.x, y.x, yy.x);
    if (n_valid > 1) add(x.y, Q.y, rU.y, c1.y, c2.y, h0.y, zh.y, rz.y, y.y, yy.y);
}

// A warp takes four galaxies, eight lanes each (lane j of eight: samples j, j + 8, ...), in blocks
// of 32 samples.  The normal-CDF terms of a block are formed first, one galaxy at a time over
// all 32 lanes: a galaxy's samples are mostly on one side of mu_f, so that the branches
// of log_ndtr_mills seldom diverge, which four galaxies side by side do; they pass through
// shared memory to the lanes that sum them.  Bound by instruction issue.
// 100,000 x 300: 0.45 ms with the terms formed where they are summed, in scalar arithmetic, an
// output at a time through the FP64 pipe; 0.30 ms now (0.40 with prefetched loads and the FP64
// sums side by side alone).
template <int FAMILY>
__global__ void __launch_bounds__(kShearThreads, 3) shear_full_kernel(const __grid_constant__ ShearFullLaunch f)
{
    __shared__ float4 s_norm[kShearThreads / 32][4][33];   // (log Phi, r, z) per galaxy and sample of the block
    const ShearLaunch &s = f.s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = lane & (kGroup - 1), g = lane / kGroup;
    const unsigned gmask = 0xFFu << (lane & ~(kGroup - 1));
    const long long ngroups = (long long)gridDim.x * blockDim.x / kGroup;
    const ShearConst c = held(s.c);
    const int K = s.K;
    double acc = 0.0, acc8 = 0.0;   // output `sub` of the first eight; the ninth (lane 0)

    for (long long n0 = ((long long)blockIdx.x * (kShearThreads / 32) + warp) * 4; n0 < s.n_gal; n0 += ngroups) {
        const long long n = n0 + g;                        // this lane's galaxy
        const bool live = n < s.n_gal;
        const float *p1 = s.e1 + n * (long long)K, *p2 = s.e2 + n * (long long)K;
        const float *pf = f.lf + n0 * (long long)K, *ps = f.ls + n * (long long)K;
        const int ng = s.n_gal - n0 < 4 ? (int)(s.n_gal - n0) : 4;
        FullAcc A;
        A.m = -1e30f;
        A.sw = 0.f;
        A.t = A.qy = A.h01 = A.h24 = f2(0.f);
        for (int kb = 0; kb < K; kb += 32) {
            float v1[4], v2[4], vs[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int k = kb + 8 * t + sub;
                const bool in = live && k < K;
                v1[t] = in ? __ldg(p1 + k) : 0.f;
                v2[t] = in ? __ldg(p2 + k) : 0.f;
                vs[t] = in ? __ldg(ps + k) : 0.f;
            }
            float vf[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                vf[j] = j < ng && kb + lane < K ? __ldg(pf + (long long)j * K + kb + lane) : f.mu_f;
#pragma unroll 1
            for (int j = 0; j < ng; ++j) {
                const float lf = j == 0 ? vf[0] : j == 1 ? vf[1] : j == 2 ? vf[2] : vf[3];
                const float z = (lf - f.mu_f) * f.inv_sf;
                float lphi = 0.f, r = 0.f;
                if (kb + lane < K) log_ndtr_mills(f.a_f * z, lphi, r);
                s_norm[warp][j][lane] = make_float4(lphi, r, z, 0.f);
            }
            __syncwarp();
            if (live) {
                const float4 *sn = s_norm[warp][g];
#pragma unroll
                for (int t = 0; t < 4; t += 2) {
                    const int k = kb + 8 * t + sub;
                    if (k < K)
                        full_pair<FAMILY>(f, c, make_float2(v1[t], v1[t + 1]), make_float2(v2[t], v2[t + 1]),
                                          make_float2(vs[t], vs[t + 1]), sn[8 * t + sub], sn[8 * t + 8 + sub],
                                          k + 8 < K ? 2 : 1, A);
                }
            }
            __syncwarp();
        }
        if (!live) continue;
    // merge the 8 lanes of the group
        float u[10] = {A.m, A.sw, A.t.x, A.t.y, A.qy.x, A.h01.x, A.h01.y, A.h24.x, A.qy.y, A.h24.y};
#pragma unroll
        for (int o = kGroup / 2; o > 0; o >>= 1) {
            float w[10];
#pragma unroll
            for (int i = 0; i < 10; ++i) w[i] = __shfl_xor_sync(gmask, u[i], o, kGroup);
            const float mn = fmaxf(u[0], w[0]);
            const float ca = ex2_ftz(u[0] - mn), cb = ex2_ftz(w[0] - mn);
#pragma unroll
            for (int i = 1; i < 10; ++i) u[i] = u[i] * ca + w[i] * cb;
            u[0] = mn;
        }
        // lane 0 takes the log-sum-exp and the last derivative sum, lanes 1-7 a derivative sum
        // each (one pass through the FP64 pipe for the eight)
        const float wf = s.w ? __ldg(s.w + n) : 1.0f;
        if (wf != 0.0f) {
            if (u[1] > 0.f) {
                const float inv = 1.0f / u[1];
                float d = -2.0f * u[2] * inv;
                if (sub == 2) d = -2.0f * u[3] * inv;
#pragma unroll
                for (int i = 4; i < 9; ++i)
                    if (sub == i - 1) d = u[i] * inv;
                int e;
                const float l = log2f(frexpf(u[1], &e));   // as finish_galaxy
                double t = (double)(sub == 0 ? u[0] : d);
                if (sub == 0) t += (double)e + (double)l;
                acc += s.w ? (double)wf * t : t;
                if (sub == 0) {
                    const double t8 = (double)(u[9] * inv);
                    acc8 += s.w ? (double)wf * t8 : t8;
                }
            } else if (sub == 0) {
                acc = -INFINITY;
            }
        }
    }
    __shared__ double red[kShearThreads / 32][kShearFullOut];
#pragma unroll
    for (int o = 16; o >= kGroup; o >>= 1) {
        acc += __shfl_xor_sync(BS_FULL_MASK, acc, o);
        acc8 += __shfl_xor_sync(BS_FULL_MASK, acc8, o);
    }
    const int w = threadIdx.x >> 5;
    if (lane < kGroup) red[w][lane] = acc;
    if (lane == 0) red[w][kShearFullOut - 1] = acc8;
    __syncthreads();
    if (threadIdx.x < kShearFullOut) {
        double t = 0.0;
        for (int i = 0; i < kShearThreads / 32; ++i) t += red[i][threadIdx.x];
        s.partials[(size_t)blockIdx.x * kShearFullOut + threadIdx.x] = t;
    }
}

struct FinalizeN {
    double scale[kShearFullOut], add[kShearFullOut];
};

// A warp per output, as finalize_point.
__global__ void __launch_bounds__(32 * kShearFullOut) shear_finalize_n_kernel(const double *partials, int n_part, int n_out,
                                                                              const __grid_constant__ FinalizeN c,
                                                                              double *out)
{
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double t = 0.0;
#pragma unroll 8
    for (int i = lane; i < n_part; i += 32) t += partials[(size_t)i * n_out + k];
    t = warp_sum_d(t);
    if (lane == 0) out[k] = t * c.scale[k] + c.add[k];
}

template <int FAMILY, bool HAS_B>
cudaError_t launch_fb(const ShearLaunch &s, int grid, bool vec, cudaStream_t st)
{
    if (vec) {
        // the samples as tensor maps, streamed in tiles by the tensor memory accelerator
        CUtensorMap m1, m2, m3;
        if (make_sample_map(m1, s.e1, s.n_gal, s.K) && make_sample_map(m2, s.e2, s.n_gal, s.K) &&
            make_sample_map(m3, HAS_B ? s.b : s.e1, s.n_gal, s.K)) {
            constexpr size_t smem = tma_smem_bytes(HAS_B);
            const cudaError_t e = cudaFuncSetAttribute(shear_kernel_tma<FAMILY, HAS_B>,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            shear_kernel_tma<FAMILY, HAS_B><<<grid, kShearThreads, smem, st>>>(s, m1, m2, m3);
            return cudaGetLastError();
        }
    }
    shear_kernel<FAMILY, HAS_B><<<grid, kShearThreads, 0, st>>>(s);
    return cudaGetLastError();
}

// ---- Several points per pass.  One read of the samples serves up to
// kMultiPoints (g1, g2, alpha) points: each sample's weight and derivative
// factors are formed for every point (the same per-sample arithmetic as
// shear_kernel), so the pass turns from HBM-bound into ALU-bound; the shear
// estimate's batches (central differences of its Hessian, Gauss-Hermite nodes)
// then cost about their arithmetic alone.  A galaxy group's FP64 totals go to
// its own shared-memory slot (one writer), summed over the block in a fixed
// order; partials are laid out per point so that each point is finalized as
// a single-point pass.
template <int FAMILY>
__global__ void __launch_bounds__(kShearThreads, 2) shear_kernel_multi(const __grid_constant__ ShearMultiLaunch m)
{
    constexpr int NP = kMultiPoints;
    constexpr int kGroups = kShearThreads / kGroup;
    __shared__ double acc[kGroups][NP][4];
    const ShearLaunch &s = m.s;
    const int lane = threadIdx.x & 31;
    const int sub = lane & (kGroup - 1);
    const int gi = threadIdx.x / kGroup;
    const unsigned gmask = 0xFFu << (lane & ~(kGroup - 1));
    const long long group = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kGroup;
    const long long ngroups = (long long)gridDim.x * blockDim.x / kGroup;
    const int K = s.K;
    if (sub == 0)
        for (int p = 0; p < NP; ++p)
            for (int i = 0; i < 4; ++i) acc[gi][p][i] = 0.0;

    for (long long n = group; n < s.n_gal; n += ngroups) {
        const long long base = n * (long long)K;
        Lse L[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) lse_reset(L[p]);
        Chunk A, B;
        int k0 = 4 * sub;
        auto eval_all = [&](const Chunk &ch) {
#pragma unroll
            for (int p = 0; p < NP; ++p)
                if (p < m.n_points) eval_chunk<FAMILY, false>(m.c[p], ch, L[p]);
        };
        load_chunk<false>(s, base, k0, K, A);
        for (;;) {
            if (k0 >= K) break;
            load_chunk<false>(s, base, k0 + 4 * kGroup, K, B);
            eval_all(A);
            k0 += 4 * kGroup;
            if (k0 >= K) break;
            load_chunk<false>(s, base, k0 + 4 * kGroup, K, A);
            eval_all(B);
            k0 += 4 * kGroup;
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (p < m.n_points) {
                double t = 0.0;
                finish_galaxy(L[p], m.g1[p], m.g2[p], gmask, sub, s.w, n, t);
                if (sub < 4) acc[gi][p][sub] += t;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < NP * 4) {
        const int p = threadIdx.x >> 2, i = threadIdx.x & 3;
        double t = 0.0;
        for (int k = 0; k < kGroups; ++k) t += acc[k][p][i];
        m.partials[((size_t)p * gridDim.x + blockIdx.x) * 4 + i] = t;
    }
}

}  // namespace

namespace {

// SMs x resident CTAs of a kernel on the current device, asked of the runtime once per device
// (every evaluation of a likelihood needs it).
struct GridCache {
    std::atomic<int> blocks[64] = {};
};
template <typename K>
int resident_grid(GridCache &cache, K kernel, size_t smem)
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64) {
        const int known = cache.blocks[dev].load(std::memory_order_relaxed);
        if (known > 0) return known;
    }
    int sms = 0, nb = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kShearThreads, smem);
    if (sms <= 0 || nb <= 0) return sms > 0 ? sms : 1;      // not kept: the next call asks again
    if (dev >= 0 && dev < 64) cache.blocks[dev].store(sms * nb, std::memory_order_relaxed);
    return sms * nb;
}

GridCache g_grid_one, g_grid_b, g_grid_scalar, g_grid_scalar_b, g_grid_full, g_grid_multi;

// Whether a one-point pass streams its samples in tiles.
bool shear_vec(const ShearLaunch &s)
{
    return (s.K % 4 == 0) && ((reinterpret_cast<uintptr_t>(s.e1) & 15) == 0) &&
           ((reinterpret_cast<uintptr_t>(s.e2) & 15) == 0) &&
           (s.b == nullptr || (reinterpret_cast<uintptr_t>(s.b) & 15) == 0);
}

// Each pass is sized by its own kernel: with offsets the tile kernel holds 2 CTAs per SM, the scalar
// one 3 (100,000 x 250 with b: 68-70 us, 78-95 us with 2 per SM).
int shear_grid_resident(bool has_b, bool vec)
{
    if (vec)
        return has_b ? resident_grid(g_grid_b, shear_kernel_tma<BS_EPRIOR_TRUNC_GAUSS, true>, tma_smem_bytes(true))
                     : resident_grid(g_grid_one, shear_kernel_tma<BS_EPRIOR_TRUNC_GAUSS, false>, tma_smem_bytes(false));
    return has_b ? resident_grid(g_grid_scalar_b, shear_kernel<BS_EPRIOR_TRUNC_GAUSS, true>, 0)
                 : resident_grid(g_grid_scalar, shear_kernel<BS_EPRIOR_TRUNC_GAUSS, false>, 0);
}

}  // namespace

int shear_grid_blocks()
{
    int most = 0;
    for (int i = 0; i < 4; ++i) most = std::max(most, shear_grid_resident(i & 1, i & 2));
    return most;
}

int shear_grid_for(const ShearLaunch &s)
{
    const int full = shear_grid_resident(s.b != nullptr, shear_vec(s));
    const long long want = (s.n_gal + 31) / 32;
    return want < 1 ? 1 : want < full ? (int)want : full;
}

cudaError_t launch_shear(const ShearLaunch &s, int grid, cudaStream_t stream)
{
    const bool vec = shear_vec(s), hb = s.b != nullptr;
    if (s.family == BS_EPRIOR_BA14)
        return hb ? launch_fb<BS_EPRIOR_BA14, true>(s, grid, vec, stream)
                  : launch_fb<BS_EPRIOR_BA14, false>(s, grid, vec, stream);
    return hb ? launch_fb<BS_EPRIOR_TRUNC_GAUSS, true>(s, grid, vec, stream)
              : launch_fb<BS_EPRIOR_TRUNC_GAUSS, false>(s, grid, vec, stream);
}

int shear_full_grid_blocks() { return resident_grid(g_grid_full, shear_full_kernel<BS_EPRIOR_BA14>, 0); }

cudaError_t launch_shear_full(const ShearFullLaunch &f, int grid, cudaStream_t stream)
{
    if (f.s.family == BS_EPRIOR_BA14)
        shear_full_kernel<BS_EPRIOR_BA14><<<grid, kShearThreads, 0, stream>>>(f);
    else
        shear_full_kernel<BS_EPRIOR_TRUNC_GAUSS><<<grid, kShearThreads, 0, stream>>>(f);
    return cudaGetLastError();
}

cudaError_t launch_shear_finalize_n(const double *partials, int n_part, int n_out, const double *scale,
                                    const double *add, double *out, cudaStream_t stream)
{
    if (n_out < 1 || n_out > kShearFullOut) return cudaErrorInvalidValue;
    FinalizeN c;
    for (int i = 0; i < kShearFullOut; ++i) {
        c.scale[i] = i < n_out ? scale[i] : 0.0;
        c.add[i] = i < n_out ? add[i] : 0.0;
    }
    shear_finalize_n_kernel<<<1, 32 * n_out, 0, stream>>>(partials, n_part, n_out, c, out);
    return cudaGetLastError();
}

int shear_multi_grid_blocks() { return resident_grid(g_grid_multi, shear_kernel_multi<BS_EPRIOR_BA14>, 0); }

// Several points per pass with the samples streamed in tiles (K a multiple of 4,
// 16-byte aligned rows, no b): the one-point tile kernel's ring and lane layout, each
// quad of samples evaluated for every point, each point keeping its own log-sum-exp
// state; a galaxy's 4 lanes put their FP64 totals per point in their own shared-memory
// slot, summed over the block in a fixed order.  On a wait that gives up, the block's
// partials are NaN.
// FULL: all kMultiPoints points are asked for (no test between them).  BOUNDED: eval_plain's bound
// holds for every point.
template <int FAMILY, bool FULL, bool BOUNDED>
__global__ void __launch_bounds__(kShearThreads, 2)
    shear_kernel_tma_multi(const __grid_constant__ ShearMultiLaunch m, const __grid_constant__ CUtensorMap m1,
                           const __grid_constant__ CUtensorMap m2)
{
    constexpr int NP = kMultiPoints;
    extern __shared__ __align__(128) unsigned char tma_raw[];
    __shared__ __align__(8) uint64_t full[kTmaStages], empty[kTmaStages];
    __shared__ double acc[kTileG][NP][4];
    __shared__ int s_fail;
    const ShearLaunch &s = m.s;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int sub = tid & (kAGroup - 1), gl = tid / kAGroup;
    const unsigned gmask = ((1u << kAGroup) - 1u) << (lane & ~(kAGroup - 1));
    const int K = s.K;
    if (sub == 0)
        for (int p = 0; p < NP; ++p)
            for (int i = 0; i < 4; ++i) acc[gl][p][i] = 0.0;
    if (tid == 0) s_fail = 0;
    TmaRing<2> R;
    R.init(tma_raw, full, empty, s.n_gal, K);   // (its barrier also orders the resets above)
    if (tid == 0)
        for (int t = 0; t < kTmaStages - 1; ++t) R.issue(&m1, &m2, nullptr);
    Lse L[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) lse_reset(L[p]);
    bool failed = false;
    int chunk = 0;
    long long tile = blockIdx.x;
    for (int item = 0; item < R.n_items; ++item) {
        if (tid == 0) R.issue(&m1, &m2, nullptr);
        if (!R.wait_full(item)) {
            failed = true;
            break;
        }
        const long long n = tile * kTileG + gl;
        if (n < s.n_gal) {
            const int nq = tma_quads(K, chunk);
#pragma unroll
            for (int h = 0; h < kQuads; ++h) {
                if (h < nq) {
                    const Chunk ch = tma_quad(R, item, h);
                    auto all = [&](auto eval) {
#pragma unroll
                        for (int p = 0; p < NP; ++p)
                            if (FULL || p < m.n_points) eval(p);
                    };
                    if (h == 0 && chunk == 0)
                        all([&](int p) { eval_first<FAMILY, false>(m.c[p], ch, L[p]); });
                    else if constexpr (BOUNDED)
                        all([&](int p) { eval_plain<FAMILY>(m.c[p], ch, L[p]); });
                    else
                        all([&](int p) { eval_quad<FAMILY>(m.c[p], ch, L[p]); });
                }
            }
            if (BOUNDED && FAMILY == BS_EPRIOR_TRUNC_GAUSS && chunk == 0 && nq > 0) {
#pragma unroll
                for (int p = 0; p < NP; ++p)
                    if ((FULL || p < m.n_points) && L[p].m == kNoReference)
                        L[p] = first_chunk<FAMILY>(m.c[p], tma_row(R, item), nq);
            }
        }
        R.release(item);
        if (++chunk == R.cpg) {
            if (n < s.n_gal) {
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    if (p < m.n_points) {
                        double t = 0.0;
                        const float sw = finish_galaxy<kAGroup>(L[p], m.g1[p], m.g2[p], gmask, sub, s.w, n, t);
                        if (BOUNDED && !(sw < kMost)) t = replay_galaxy<FAMILY>(m, p, n, sub, gmask);
                        acc[gl][p][sub] += t;
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < NP; ++p) lse_reset(L[p]);
            chunk = 0;
            tile += gridDim.x;
        }
    }
    if (failed || (tid == 0 && !R.p_ok)) s_fail = 1;
    R.drain();
    __syncthreads();
    if (tid < NP * 4) {
        const int p = tid >> 2, i = tid & 3;
        double t = 0.0;
        for (int k = 0; k < kTileG; ++k) t += acc[k][p][i];
        m.partials[((size_t)p * gridDim.x + blockIdx.x) * 4 + i] = s_fail ? NAN : t;
    }
}

namespace {

using MultiKernel = void (*)(const ShearMultiLaunch, const CUtensorMap, const CUtensorMap);
template <int FAMILY>
MultiKernel tma_multi_kernel(bool full, bool bounded)
{
    if (bounded) return full ? shear_kernel_tma_multi<FAMILY, true, true> : shear_kernel_tma_multi<FAMILY, false, true>;
    return full ? shear_kernel_tma_multi<FAMILY, true, false> : shear_kernel_tma_multi<FAMILY, false, false>;
}

}  // namespace

bool weights_bounded(const ShearLaunch &s) { return s.a2 + s.c0 <= kMaxSpan; }

cudaError_t launch_shear_multi(const ShearMultiLaunch &m, int grid, cudaStream_t stream)
{
    const ShearLaunch &s = m.s;
    const bool vec = (s.K % 4 == 0) && ((reinterpret_cast<uintptr_t>(s.e1) & 15) == 0) &&
                     ((reinterpret_cast<uintptr_t>(s.e2) & 15) == 0) && s.b == nullptr;
    CUtensorMap m1, m2;
    if (vec && make_sample_map(m1, s.e1, s.n_gal, s.K) && make_sample_map(m2, s.e2, s.n_gal, s.K)) {
        auto k = s.family == BS_EPRIOR_BA14 ? tma_multi_kernel<BS_EPRIOR_BA14>(m.n_points == kMultiPoints, m.bounded)
                                            : tma_multi_kernel<BS_EPRIOR_TRUNC_GAUSS>(m.n_points == kMultiPoints, m.bounded);
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)tma_smem_bytes(false));
        if (e != cudaSuccess) return e;
        k<<<grid, kShearThreads, tma_smem_bytes(false), stream>>>(m, m1, m2);
        return cudaGetLastError();
    }
    if (m.s.family == BS_EPRIOR_BA14)
        shear_kernel_multi<BS_EPRIOR_BA14><<<grid, kShearThreads, 0, stream>>>(m);
    else
        shear_kernel_multi<BS_EPRIOR_TRUNC_GAUSS><<<grid, kShearThreads, 0, stream>>>(m);
    return cudaGetLastError();
}

cudaError_t launch_shear_finalize(const double *partials, int n_part, double add_value,
                                  double add_g1, double add_g2, double add_alpha,
                                  double alpha_scale, double *out, cudaStream_t stream)
{
    const ShearFinalize f = {{add_value, add_g1, add_g2, add_alpha}, alpha_scale};
    shear_finalize_kernel<<<1, 128, 0, stream>>>(partials, n_part, f, out);
    return cudaGetLastError();
}

cudaError_t launch_shear_finalize_batch(const double *partials, size_t part_stride, int n_part,
                                        const ShearFinalizeBatch &b, double *out, cudaStream_t stream)
{
    if (b.n_points < 1 || b.n_points > kFinalizePoints) return cudaErrorInvalidValue;
    shear_finalize_batch_kernel<<<b.n_points, 128, 0, stream>>>(partials, part_stride, n_part, b, out);
    return cudaGetLastError();
}

}  // namespace bs
