// Spergel and Gaussian galaxy profiles of the image-sampling kernels
// (Appendix B: the forward model with a Spergel profile of fixed index nu, or
// a Gaussian), compiled apart from the exponential instances of bs_fit.cu.
#include <cmath>

#include "bs_fit_impl.cuh"

namespace bs {

namespace {

using FitKernel = void (*)(const FitParams);
using PointsKernel = void (*)(const FitParams, int, const int32_t *, const float *, double *, float *);

template <int PROF>
FitKernel prof_kernel(int max_side)
{
    switch ((max_side + 31) / 32) {
        case 1: return fit_kernel_r128<1, PROF>;
        case 2: return fit_kernel_r128<2, PROF>;
        case 3: return fit_kernel_r128<3, PROF>;
        default: return fit_kernel_r128<4, PROF>;
    }
}

// Per-pixel weights (profile 3), exponential: stamps of at most 63 px, two or four chains
// per CTA, the transforms on the tensor cores.
bool pix_quad(int max_side, int cc) { return cc == 4 && max_side <= kPixQuadSide; }   // cc: chains of a CTA

FitKernel pix_kernel(int max_side, bool quad)
{
    if (quad) return max_side <= 31 ? fit_kernel_pix<1, 5> : fit_kernel_pix<2, 5>;
    return max_side <= 31 ? fit_kernel_pix<1, 3> : fit_kernel_pix<2, 3>;
}
static_assert(tc::Geo<4>::KV == kPixQuadSide + 1 && tc::Geo<2>::kThreads == 256, "the chain layouts");

bool is_pix(int profile) { return profile == 3; }

FitKernel kernel_for(int profile, int max_side, int cc)
{
    if (profile == 3) return pix_kernel(max_side, pix_quad(max_side, cc));
    if (profile == 4) return fit_kernel_dense<1>;   // a dense covariance: at most 31 px
    return profile == BS_PROFILE_SPERGEL ? prof_kernel<1>(max_side) : prof_kernel<2>(max_side);
}

template <int PROF>
PointsKernel prof_points(int max_side)
{
    switch ((max_side + 31) / 32) {
        case 1: return logpost_points_kernel<1, PROF>;
        case 2: return logpost_points_kernel<2, PROF>;
        case 3: return logpost_points_kernel<3, PROF>;
        default: return logpost_points_kernel<4, PROF>;
    }
}

PointsKernel points_for(int profile, int max_side)
{
    if (is_pix(profile)) return max_side <= 31 ? logpost_points_pix_kernel<1> : logpost_points_pix_kernel<2>;
    if (profile == 4) return logpost_points_dense_kernel<1>;
    return profile == BS_PROFILE_SPERGEL ? prof_points<1>(max_side) : prof_points<2>(max_side);
}

// Dynamic shared memory of a launch: the pixel-weight path adds the transforms'
// region after the row table, the dense-covariance path its twiddles and
// per-chain scratch.
size_t smem_for(int profile, int max_side, int cc)
{
    if (is_pix(profile)) {
        const int h = (max_side + 1) / 2, npad = 32 * ((max_side + 31) / 32);
        return pix_quad(max_side, cc) ? fit_smem_bytes(max_side, 4) + 16 + pix_tc_bytes<4>(max_side, h, npad)
                                      : fit_smem_bytes(max_side, 2) + 16 + pix_tc_bytes<2>(max_side, h, npad);
    }
    size_t b = fit_smem_bytes(max_side, cc);
    if (profile == 4) {
        const int h = (max_side + 1) / 2, npad = 32 * ((max_side + 31) / 32);
        b += 16 + dense_region_bytes(h, npad, max_side, cc);
    }
    return b;
}

// A kernel's limit of dynamic shared memory: that of the largest stamp and chain count it takes, the
// same from every host thread (as for the white-noise kernels).
cudaError_t allow_smem(const void *kernel, int profile, int max_side, int cc)
{
    const size_t most = is_pix(profile)  ? smem_for(profile, pix_quad(max_side, cc) ? kPixQuadSide : 63, cc)
                        : profile == 4 ? smem_for(profile, kDenseMaxSide, kDenseChains)
                                       : smem_for(profile, BS_MAX_SIDE, kMaxChains);
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

int threads_for(int profile, int cc, int max_side, int dense_warps)
{
    if (is_pix(profile)) return 128 * (pix_quad(max_side, cc) ? 4 : 2);
    return 32 * (profile == 4 ? (dense_warps > 0 ? dense_warps : kDenseWarps) : cc);
}

// Warps of a CTA of dense-covariance points (its runs of points are not known on the host): four, one
// for each chain slot, where the points are more than a CTA of 16 per SM takes at once and the stamps
// small.  2,000 points of 7 px, one per galaxy: 136 us with
// 16 warps, 44 with four.
int dense_point_warps(int n_points, int max_side)
{
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return max_side <= 15 && n_points > (max_side <= 9 ? 1 : 4) * sms ? kDenseChains : kDenseWarps;
}

// K_mu(x) = int_0^inf exp(-x cosh t) cosh(mu t) dt by the trapezoidal rule
// (step 1/64; the integrand falls off doubly exponentially).
double bessel_k(double mu, double x)
{
    const double h = 1.0 / 64.0;
    double sum = 0.5 * std::exp(-x);
    for (int j = 1; j < 4096; ++j) {
        const double t = j * h;
        const double term = std::exp(-x * std::cosh(t)) * std::cosh(mu * t);
        sum += term;
        if (term < 1e-18 * sum) break;
    }
    return sum * h;
}

}  // namespace

double profile_hlr_over_r0(int profile, double nu)
{
    if (profile == BS_PROFILE_GAUSSIAN) return std::sqrt(2.0 * std::log(2.0));
    if (profile != BS_PROFILE_SPERGEL) return 1.6783469900166608;
    // enclosed flux of the Spergel profile, 1 - x^(1+nu) K_(1+nu)(x) / (2^nu Gamma(1+nu)),
    // increases from 0 to 1: bisect for 1/2
    const double norm = std::pow(2.0, nu) * std::tgamma(1.0 + nu);
    auto enclosed = [&](double x) { return 1.0 - std::pow(x, 1.0 + nu) * bessel_k(1.0 + nu, x) / norm; };
    double lo = 1e-6, hi = 50.0;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (enclosed(mid) < 0.5) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

// Warps of a dense-covariance CTA: all 16 while every CTA finds an SM of its own.  Small stamps in larger
// numbers are worth more CTAs per SM (16 warps in all, which the 128 registers of a thread allow) than
// warps per CTA, whose barriers outweigh 4 to 8 rows of work; no fewer than the CTA's chains, and
// from 15 px no fewer than four; from 17 px the product with the precision fills 16.
// 2,000 galaxies of 7 px, one chain of 20 + 20 iterations: 12.1 ms with 16 warps per CTA, 6.2 with
// four, 2.2 with one.
int dense_warps_for(long long ctas, int cc, int max_side, int sms)
{
    if (max_side > 15) return kDenseWarps;
    const long long per_sm = (ctas + sms - 1) / sms;
    int least = max_side > 13 ? 4 : 1;
    while (least < cc) least *= 2;
    int w = kDenseWarps;
    while (w > least && w * per_sm > kDenseWarps) w /= 2;
    return w;
}

int fit_blocks_per_sm_profile(int profile, int cc, int max_side, int dense_warps)
{
    int nb = 0;
    const size_t smem = smem_for(profile, max_side, cc);
    FitKernel k = kernel_for(profile, max_side, cc);
    allow_smem((const void *)k, profile, max_side, cc);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, threads_for(profile, cc, max_side, dense_warps), smem) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_fit_profile(const FitParams &p, int grid, cudaStream_t stream)
{
    const int cc = cta_chains(p);
    const size_t smem = smem_for(p.profile, p.max_side, cc);
    FitKernel k = kernel_for(p.profile, p.max_side, cc);
    cudaError_t e = allow_smem((const void *)k, p.profile, p.max_side, cc);
    if (e != cudaSuccess) return e;
    k<<<grid, threads_for(p.profile, cc, p.max_side, p.dense_warps), smem, stream>>>(p);
    bs::count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_logpost_points_profile(const FitParams &p, int n_points, const int32_t *gal_index,
                                          const float *theta, double *logp, float *grad, cudaStream_t stream)
{
    const int warps = is_pix(p.profile) ? 8 : p.profile == 4 ? dense_point_warps(n_points, p.max_side) : point_warps(p);
    // (the dense path's CTA holds its four chain slots whatever its warps)
    const size_t smem = smem_for(p.profile, p.max_side, is_pix(p.profile) ? 2 : p.profile == 4 ? kDenseChains : warps);
    PointsKernel k = points_for(p.profile, p.max_side);
    cudaError_t e = allow_smem((const void *)k, p.profile, p.max_side, 2);
    if (e != cudaSuccess) return e;
    const int grid = is_pix(p.profile) && n_points > 4096 ? 4096 : n_points;   // the others: a CTA per point
    k<<<grid, 32 * warps, smem, stream>>>(p, n_points, gal_index, theta, logp, grad);
    bs::count_launches(1);
    return cudaGetLastError();
}

}  // namespace bs
