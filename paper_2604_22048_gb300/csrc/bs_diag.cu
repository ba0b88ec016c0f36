// Chain diagnostics on sm_103a (Sec. 4.1): per galaxy and parameter, the
// classic potential scale reduction R-hat (Gelman & Rubin 1992) and the
// multi-chain effective sample size with Geyer's initial monotone positive
// sequence (Gelman et al., BDA3 Sec. 11.5):
//   var+ = (n-1)/n W + B/n,  rho_t = 1 - (W - mean_c acov_c(t)) / var+,
//   tau = -1 + 2 sum_k P_k (P_k = rho_2k + rho_2k+1 while positive, made
//   monotone), ESS = m n / tau with tau >= 1 / log10(m n).
// One warp per (galaxy, parameter); autocovariances by direct lane-parallel
// sums, computed only until the sequence stops.
#include <cmath>

#include "bs_device.cuh"
#include "bs_internal.h"

namespace bs {

namespace {

// Moments of a galaxy's chains and what follows from them: W, B / n and var+.
struct ChainMoments {
    float W, vp;
};
__device__ __forceinline__ ChainMoments chain_moments(const float (&mean)[kMaxChains], float wsum, float mbar, int C, int S)
{
    const float W = wsum / C;
    mbar /= C;
    float bn = 0.f;
    if (C > 1) {
#pragma unroll
        for (int c = 0; c < kMaxChains; ++c)
            if (c < C) bn += (mean[c] - mbar) * (mean[c] - mbar);
        bn /= (C - 1);
    }
    const float vp = (S - 1.0f) / S * W + bn;
    return {W, vp};
}

// tau from the sum of the monotone positive pairs, into ESS and R-hat.
__device__ __forceinline__ void store_ess(float sum, const ChainMoments &m, int C, int S, size_t out, float *ess, float *rhat)
{
    float tau = -1.0f + 2.0f * sum;
    const float tmin = 1.0f / log10f((float)C * S);
    if (tau < tmin) tau = tmin;
    ess[out] = (float)C * S / tau;
    if (rhat) rhat[out] = sqrtf(m.vp / m.W);
}

// The chains of a warp's (galaxy, parameter) are staged once in shared memory as deviations
// from their means, two chains interleaved (zeros beside the last of an odd number), pair p at
// p (S + kLagBlock) with zeros after it, and their autocovariances are taken kLagBlock lags at a
// time in packed FP32x2, a chain in either half: a lane sums an odd-length run of
// consecutive samples (no bank conflicts between lanes), four samples x eight lags per step
// from four samples and a window of eleven, seven of them kept from the step before: 8
// loads for 32 packed multiply-adds, all chains into the same eight sums, reduced over the warp
// together.  Most sequences stop within one or two blocks of lags.  The samples are
// read once from HBM.  Bound by instruction issue, shared-memory loads and the FMA pipe about
// alike.
// 10,000 galaxies x 4 chains x 300: 493-614 us (with the autocorrelation of the
// chains) re-reading both factors of every product and reducing chain by chain and lag by lag,
// 117 us now at 64 registers (8 CTAs of 4 warps per SM; 120 us for 7 CTAs, 119 for 9).
constexpr int kLagBlock = 8;

__host__ __device__ constexpr size_t ess_warp_floats(int C, int S)
{
    return (size_t)((C + 1) / 2) * 2 * ((size_t)S + kLagBlock);
}

// VEC: S a multiple of 4 and the samples 16-byte aligned (16-byte loads).
template <bool VEC>
__global__ void __launch_bounds__(128, 8) ess_kernel(const float *samples, int n_gal, int C, int S, float *ess, float *rhat)
{
    extern __shared__ __align__(16) float ess_smem[];
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5, warp = threadIdx.x >> 5;
    // grid y: the parameter, so that neighbouring warps read neighbouring galaxies
    const int k = blockIdx.y;
    const long long gl = (long long)blockIdx.x * warps + warp;
    if (gl >= n_gal) return;
    const int gal = (int)gl;
    const float *x = samples + (((size_t)k * n_gal + gal) * C) * S;
    const int stride = S + kLagBlock;
    float2 *d = reinterpret_cast<float2 *>(ess_smem + warp * ess_warp_floats(C, S));
    float mean[kMaxChains], var[kMaxChains];
#pragma unroll
    for (int p = 0; p < kMaxChains / 2; ++p) {
        float sa = 0.f, sb = 0.f;
        if (2 * p < C) {
            const float *xa = x + (size_t)(2 * p) * S;
            const bool two = 2 * p + 1 < C;
            const float *xb = two ? xa + S : xa;
            float2 *dp = d + p * stride;
            if constexpr (VEC) {
                // six loads in flight per round trip
                for (int i0 = 4 * lane; i0 < S; i0 += 384) {
                    float4 a[3], b[3];
#pragma unroll
                    for (int t = 0; t < 3; ++t) {
                        const int i = i0 + 128 * t;
                        a[t] = b[t] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (i < S) {
                            a[t] = __ldg(reinterpret_cast<const float4 *>(xa + i));
                            if (two) b[t] = __ldg(reinterpret_cast<const float4 *>(xb + i));
                        }
                    }
#pragma unroll
                    for (int t = 0; t < 3; ++t) {
                        const int i = i0 + 128 * t;
                        if (i < S) {
                            float4 *o = reinterpret_cast<float4 *>(dp + i);
                            o[0] = make_float4(a[t].x, b[t].x, a[t].y, b[t].y);
                            o[1] = make_float4(a[t].z, b[t].z, a[t].w, b[t].w);
                        }
                        sa += (a[t].x + a[t].y) + (a[t].z + a[t].w);
                        sb += (b[t].x + b[t].y) + (b[t].z + b[t].w);
                    }
                }
            } else {
#pragma unroll 4
                for (int i = lane; i < S; i += 32) {
                    const float a = __ldg(xa + i), b = two ? __ldg(xb + i) : 0.f;
                    dp[i] = make_float2(a, b);
                    sa += a;
                    sb += b;
                }
            }
            if (lane < kLagBlock) dp[S + lane] = make_float2(0.f, 0.f);
        }
        mean[2 * p] = sa;
        mean[2 * p + 1] = sb;
    }
    warp_sum_n(mean);
    __syncwarp();
    float mbar = 0.f, wsum = 0.f;
#pragma unroll
    for (int p = 0; p < kMaxChains / 2; ++p) {
        float2 v = make_float2(0.f, 0.f);
        if (2 * p < C) {
            mean[2 * p] = mean[2 * p] / (float)S;
            mean[2 * p + 1] = mean[2 * p + 1] / (float)S;
            const float2 nm = make_float2(-mean[2 * p], -mean[2 * p + 1]);
            float2 *dp = d + p * stride;
#pragma unroll 4
            for (int i = lane; i < S; i += 32) {
                const float2 e = __fadd2_rn(dp[i], nm);
                dp[i] = e;
                v = __ffma2_rn(e, e, v);
            }
        }
        var[2 * p] = v.x;
        var[2 * p + 1] = v.y;
    }
    warp_sum_n(var);
#pragma unroll
    for (int c = 0; c < kMaxChains; ++c) {
        if (c < C) {
            wsum += var[c] / (float)(S - 1);
            mbar += mean[c];
        }
    }
    __syncwarp();
    ChainMoments m = chain_moments(mean, wsum, mbar, C, S);
    // A variance whose reciprocal, or whose C S-fold sum, a float does not hold: the staged deviations are
    // brought near 1 by a power of two, which no ratio below sees.
    if (!(m.vp >= 0x1p-100f && m.vp <= 0x1p100f)) {
        const float s = m.vp < 1.0f ? 0x1p60f : 0x1p-60f;
        for (int i = lane; i < (C + 1) / 2 * stride; i += 32) d[i] = make_float2(d[i].x * s, d[i].y * s);
        m.W *= s * s;
        m.vp *= s * s;
        __syncwarp();
    }
    const int L = ((S + 31) >> 5) | 1, i0 = lane * L;
    const float inv_n = 1.0f / ((float)C * (float)S), inv_vp = 1.0f / m.vp;
    float sum = 0.f, prev = INFINITY;
    bool go = true;
    for (int t0 = 0; go && t0 + 1 < S; t0 += kLagBlock) {
        float2 acc2[kLagBlock];
#pragma unroll
        for (int j = 0; j < kLagBlock; ++j) acc2[j] = make_float2(0.f, 0.f);
        const int n = min(L, S - t0 - i0);     // samples of this lane with a partner at lag t0
        if (n > 0) {
            for (int p = 0; 2 * p < C; ++p) {
                const float2 *a0 = d + p * stride + i0, *q = a0 + t0;
                float2 w[kLagBlock + 3];
#pragma unroll
                for (int j = 0; j < kLagBlock - 1; ++j) w[j] = q[j];
                int i = 0;
                float2 a[4];
                for (; i + 4 <= n; i += 4) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        a[r] = a0[i + r];
                        w[kLagBlock - 1 + r] = q[i + r + kLagBlock - 1];
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int j = 0; j < kLagBlock; ++j) acc2[j] = __ffma2_rn(a[r], w[r + j], acc2[j]);
#pragma unroll
                    for (int j = 0; j < kLagBlock - 1; ++j) w[j] = w[j + 4];
                }
                // the last samples of the run, three at most
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const bool in = i + r < n;
                    a[r] = in ? a0[i + r] : make_float2(0.f, 0.f);
                    w[kLagBlock - 1 + r] = in ? q[i + r + kLagBlock - 1] : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int j = 0; j < kLagBlock; ++j) acc2[j] = __ffma2_rn(a[r], w[r + j], acc2[j]);
            }
        }
        float acc[kLagBlock];
#pragma unroll
        for (int j = 0; j < kLagBlock; ++j) acc[j] = acc2[j].x + acc2[j].y;
        warp_sum_n(acc);
#pragma unroll
        for (int j = 0; j < kLagBlock; j += 2) {
            if (go && t0 + j + 1 < S) {
                const float r0 = t0 + j == 0 ? 1.0f : 1.0f - (m.W - acc[j] * inv_n) * inv_vp;
                const float P = r0 + (1.0f - (m.W - acc[j + 1] * inv_n) * inv_vp);
                if (P > 0.f) {
                    const float Pm = P > prev ? prev : P;
                    sum += Pm;
                    prev = Pm;
                } else {
                    go = false;
                }
            }
        }
    }
    if (lane == 0) store_ess(sum, m, C, S, (size_t)gal * 6 + k, ess, rhat);
}

// Chains too long for shared memory, those whose number rounded up to even times S + 8 is above 57,344: read
// per lag.
__global__ void __launch_bounds__(128) ess_kernel_global(const float *samples, int n_gal, int C, int S,
                                                         float *ess, float *rhat)
{
    const int lane = threadIdx.x & 31;
    const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (wid >= (long long)n_gal * 6) return;
    const int gal = (int)(wid / 6), k = (int)(wid % 6);
    const float *x = samples + (((size_t)k * n_gal + gal) * C) * S;
    float mean[kMaxChains];
    float wsum = 0.f, mbar = 0.f;
    for (int c = 0; c < C; ++c) {
        const float *xc = x + (size_t)c * S;
        float s = 0.f;
        for (int i = lane; i < S; i += 32) s += xc[i];
        s = warp_sum(s) / (float)S;
        float v = 0.f;
        for (int i = lane; i < S; i += 32) {
            const float d = xc[i] - s;
            v = fmaf(d, d, v);
        }
        v = warp_sum(v) / (float)(S - 1);
        mean[c] = s;
        wsum += v;
        mbar += s;
    }
    const ChainMoments cm = chain_moments(mean, wsum, mbar, C, S);
    const float W = cm.W, vp = cm.vp;
    auto rho = [&](int t) -> float {
        float a = 0.f;
        for (int c = 0; c < C; ++c) {
            const float *xc = x + (size_t)c * S;
            float s = 0.f;
            for (int i = lane; i + t < S; i += 32) s = fmaf(xc[i] - mean[c], xc[i + t] - mean[c], s);
            a += warp_sum(s) / (float)S;
        }
        a /= C;
        return 1.0f - (W - a) / vp;
    };
    float sum = 0.f, prev = INFINITY;
    for (int kk = 0; 2 * kk + 1 < S; ++kk) {
        const float r0 = (kk == 0) ? 1.0f : rho(2 * kk);
        const float P = r0 + rho(2 * kk + 1);
        if (!(P > 0.f)) break;
        const float Pm = P > prev ? prev : P;
        sum += Pm;
        prev = Pm;
    }
    if (lane == 0) store_ess(sum, cm, C, S, (size_t)gal * 6 + k, ess, rhat);
}

// FP32 FMA throughput: eight independent chains per thread of x = x a + b on
// float pairs, as scalar FFMA or as packed FFMA2 (16 FMAs per iteration either
// way); the sum is stored so the chains are not removed.
template <bool PACKED>
__global__ void __launch_bounds__(256) ffma_kernel(float *out, int iters, float a, float b)
{
    float2 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = make_float2(1e-3f * (float)threadIdx.x + (float)i, 0.5f * (float)i);
    const float2 av = make_float2(a, a), bv = make_float2(b, b);
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (PACKED) {
                x[i] = __ffma2_rn(x[i], av, bv);
            } else {
                x[i].x = fmaf(x[i].x, a, b);
                x[i].y = fmaf(x[i].y, a, b);
            }
        }
    }
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) sum += x[i].x + x[i].y;
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

// FP64 FMA throughput: sixteen independent DFMA chains per thread.
__global__ void __launch_bounds__(256) dfma_kernel(float *out, int iters, double a, double b)
{
    double x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = 1e-3 * (double)threadIdx.x + (double)i;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = fma(x[i], a, b);
    }
    double sum = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) sum += x[i];
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = (float)sum;
}

}  // namespace

cudaError_t measure_fma_peak(int kind, double &tflops, cudaStream_t stream)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int grid = sms * 8, block = 256, iters = kind == 2 ? 512 : 16384;
    float *out = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    e = cudaMallocAsync(&out, sizeof(float) * (size_t)grid * block, stream);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    float best = 0.f;
    for (int rep = 0; rep < 3 && e == cudaSuccess; ++rep) {
        e = cudaEventRecord(e0, stream);
        if (kind == 1)
            ffma_kernel<true><<<grid, block, 0, stream>>>(out, iters, 1.0000001f, 1e-7f);
        else if (kind == 2)
            dfma_kernel<<<grid, block, 0, stream>>>(out, iters, 1.0000000001, 1e-10);
        else
            ffma_kernel<false><<<grid, block, 0, stream>>>(out, iters, 1.0000001f, 1e-7f);
        count_launches(1);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaEventRecord(e1, stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e == cudaSuccess && rep > 0 && (best == 0.f || ms < best)) best = ms;
    }
    if (out) cudaFreeAsync(out, stream);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (e != cudaSuccess) return e;
    const double flops = 2.0 * 16.0 * (double)iters * grid * block;
    tflops = flops / (best * 1e-3) / 1e12;
    return cudaStreamSynchronize(stream);
}

constexpr size_t kEssSmemMax = 224 * 1024, kEssSmemCta = 56 * 1024;

cudaError_t launch_chain_ess(const float *samples, int n_gal, int n_chains, int n_samples,
                             float *ess, float *rhat, cudaStream_t stream)
{
    const long long warps = (long long)n_gal * 6;
    if (warps == 0) return cudaSuccess;
    const size_t per_warp = ess_warp_floats(n_chains, n_samples) * sizeof(float);
    if (per_warp <= kEssSmemMax) {
        // warps per CTA: up to four that take 56 KB together (four CTAs per SM), else two or one
        const int wpc = per_warp > kEssSmemCta / 2 ? 1 : per_warp > kEssSmemCta / 4 ? 2 : 4;
        const bool vec = n_samples % 4 == 0 && (reinterpret_cast<uintptr_t>(samples) & 15) == 0;
        auto kernel = vec ? ess_kernel<true> : ess_kernel<false>;
        // the same limit from every call: one that followed the size of the call could be lowered by
        // another host thread between here and the launch
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEssSmemMax);
        if (e != cudaSuccess) return e;
        const dim3 grid((unsigned)(((long long)n_gal + wpc - 1) / wpc), 6);
        kernel<<<grid, 32 * wpc, wpc * per_warp, stream>>>(samples, n_gal, n_chains, n_samples, ess, rhat);
    } else {
        ess_kernel_global<<<(unsigned)((warps + 3) / 4), 128, 0, stream>>>(samples, n_gal, n_chains, n_samples, ess, rhat);
    }
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace bs
