// Forward model on sm_103a (Sec. 3.3): analytic k-space model of an
// exponential galaxy sheared in the reduced-shear convention
// (Eq. shear-transform), convolved with a known PSF and the pixel response,
// drawn on the stamp's periodic grid by a separable inverse DFT.
//
// One CTA per stamp.  With every index taken from the stamp's centre (y = iy - c, x =
// ix - c, v = -c..c) the two passes of the transform keep only what symmetry leaves:
//   S+-(u, a) = M(u, a) +- M(u, -a), a = 0..c (S+(u, 0) = M(u, 0), S-(u, 0) = 0);
//   C(u, y) = sum_a S+ cos(2 pi a y / N), D(u, y) = sum_a S- sin(2 pi a y / N), y = 0..c;
//   A(u, +-y) = C +- i D: two rows of the column pass for 4 multiply-adds per (u, a, y);
//   P = sum_u Re A cos(2 pi u x / N), Q = sum_u Im A sin(2 pi u x / N), x = 0..c;
//   m(y, +-x) = P -+ Q, the weights w_u / N^2 (w_0 = 1, w_u = 2) folded into M:
//     two pixels for 2 multiply-adds per (u, y, x).
// The column pass thus costs a quarter and the row pass half of the direct sums.  Rows go
// through shared memory in blocks of RB values of y (2 RB rows), so that A takes H x RB
// entries instead of H x N and more CTAs fit an SM; a thread sums four rows u of two y
// (column pass) or eight rows of two x (row pass), so that a load serves several packed
// FP32x2 multiply-adds.
// The PSF depends on |k| alone: it is formed for the H (H + 1) / 2 pairs (u, a <= u) and
// read for (u, +-a) and (a, +-u).
// Bound by instruction issue and by the CTAs that shared memory allows (24 warps per SM).
// 20,000 stamps of 25-101 px with a Moffat PSF each: 2.7 ms with direct sums over a stamp's N^2 pixels, the PSF integrated at every grid
// point and one shared-memory load per two multiply-adds; 0.51 ms now (error against
// 64 bits 3.6e-7 and 2.8e-7).
#include "bs_device.cuh"
#include "bs_internal.h"

namespace bs {

namespace {

constexpr int kNodes = 96;       // nodes t_j = j / 8 of the Moffat integral held in shared memory

// (x/2)^nu K_nu(x) by the trapezoidal rule with step 1/4, the factor folded into the
// exponent: any nu and x.
__device__ float r_half_x_pow_knu(float nu, float x)
{
    const float lx = logf(0.5f * x);
    const float h = 0.25f;
    float sum = 0.5f * expf(-x + nu * lx);
    for (int j = 1; j < 400; ++j) {
        const float t = j * h;
        const float ch = coshf(t);
        const float a = -x * ch;
        const float term = 0.5f * (expf(a + nu * (lx + t)) + expf(a + nu * (lx - t)));
        sum += term;
        if (x * ch > nu * t + 40.f && term <= 1e-9f * sum) break;
    }
    return sum * h;
}

// The stamp's PSF: Gaussian sigma or the Moffat's rd, nu = beta - 1, 2 / Gamma(nu).
struct RenderPsf {
    int kind;
    float width, nu, norm;
};

__device__ RenderPsf render_psf(const bs_psf &ps)
{
    RenderPsf q;
    q.kind = ps.kind;
    q.nu = q.norm = 0.0f;
    if (ps.kind == BS_PSF_GAUSSIAN) {
        q.width = ps.fwhm * (1.0f / 2.3548200450309493f);
        return q;
    }
    q.width = ps.fwhm / (2.0f * sqrtf(exp2f(1.0f / ps.beta) - 1.0f));
    q.nu = ps.beta - 1.0f;
    q.norm = 2.0f / tgammaf(q.nu);
    return q;
}

// Transform of the unit-flux PSF at |k|.  The Moffat's is norm (x/2)^nu K_nu(x), x = k rd:
// K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt by the trapezoidal rule, whose nodes'
// cosh t_j and cosh(nu t_j) do not depend on x, so that a node costs one exponential.
// The rule's relative error is about 2 |Gamma(nu + 2 pi i / step)| / Gamma(nu) for small x:
// 1e-9 at nu = 2 and 6e-8 at nu = 4 with step 3/8 (6e-7 at nu = 2 with step 1/2), and
// nothing a float holds with step 1/4, taken from x = 2 on, where the integrand narrows,
// and for larger nu.  Sums stop below 1e-9 of the total.  Very large nu or tiny x,
// whose factors leave the range of a float, take the folded form.
__device__ float render_psf_transfer(const RenderPsf &ps, float k, const float2 *nodes)
{
    if (ps.kind == BS_PSF_GAUSSIAN) return expf(-0.5f * k * k * ps.width * ps.width);
    const float x = k * ps.width;
    if (x == 0.0f) return 1.0f;
    if (!(ps.nu > 0.0f && ps.nu <= 6.0f && x > 1e-3f)) return ps.norm * r_half_x_pow_knu(ps.nu, x);
    const int step = x < 2.0f && ps.nu <= 4.0f ? 3 : 2;   // in eighths
    float sum = 0.5f * expf(-x);
    for (int j = step; j < kNodes; j += step) {
        const float2 n = nodes[j];                 // cosh t_j, cosh(nu t_j)
        const float term = expf(-x * n.x) * n.y;
        sum += term;
        if (term <= 1e-9f * sum) break;
    }
    return ps.norm * powf(0.5f * x, ps.nu) * sum * (0.125f * (float)step);
}

__device__ __forceinline__ float r_sincpi(float x)
{
    return x == 0.0f ? 1.0f : sinpif(x) / (3.14159265358979f * x);
}

struct RenderSmem {
    float4 *S;       // [H][H] (Re S+, Im S+, Re S-, Im S-)
    float4 *A;       // [H][RB] (Re A(+y), Im A(+y), Re A(-y), Im A(-y)); the PSF values before that
    float2 *tw;      // [N] (cos, sin)(2 pi m / N)
    float2 *X, *Y;   // [H] centroid phases exp(-2 pi i u dx / N), exp(-2 pi i a dy / N)
    float *snc;      // [H] sinc(u / N), the pixel's factor per axis
    float2 *nodes;   // [kNodes] cosh t_j, cosh(nu t_j), t_j = j / 8
};

__host__ __device__ __forceinline__ size_t render_smem_bytes(int max_side, int RB)
{
    const size_t h = (max_side + 1) / 2;
    return (h * h + h * RB) * sizeof(float4) + ((size_t)max_side + 2 * h + kNodes) * sizeof(float2) +
           h * sizeof(float);
}

// Stamps of side in (min_side, max_side], the others are left to another launch.
template <int NT, int RB>
__global__ void __launch_bounds__(NT) render_kernel(int n, const float *theta, const float *shear,
                                                    const int64_t *offsets, const int32_t *side, int min_side,
                                                    int max_side, const bs_psf *psf, int n_psf, float p, float *out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RenderSmem sm;
    {
        const int hm = (max_side + 1) / 2;
        sm.S = reinterpret_cast<float4 *>(smem_raw);
        sm.A = sm.S + (size_t)hm * hm;
        sm.tw = reinterpret_cast<float2 *>(sm.A + (size_t)hm * RB);
        sm.X = sm.tw + max_side;
        sm.Y = sm.X + hm;
        sm.nodes = sm.Y + hm;
        sm.snc = reinterpret_cast<float *>(sm.nodes + kNodes);
    }
    const int tid = threadIdx.x;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        const int N = side[i];
        if (N < 3 || N <= min_side || N > max_side || !(N & 1)) continue;   // uniform per CTA; stamp left untouched
        const int c = (N - 1) / 2, H = c + 1;
        const float *th = theta + (size_t)i * 6;
        const float F = exp10f(th[0]);
        const float r0 = exp10f(th[1]) * (1.0f / kHlrOverR0);
        float e1 = th[2], e2 = th[3];
        if (shear) {
            // eps' = (eps + g) / (1 + conj(g) eps)
            const float g1 = shear[2 * i], g2 = shear[2 * i + 1];
            const float nr = e1 + g1, ni = e2 + g2;
            const float dr = 1.0f + g1 * e1 + g2 * e2, di = g1 * e2 - g2 * e1;
            const float inv = 1.0f / (dr * dr + di * di);
            e1 = (nr * dr + ni * di) * inv;
            e2 = (ni * dr - nr * di) * inv;
        }
        const float E = e1 * e1 + e2 * e2;
        const float Pq = 1.0f / (1.0f - E);
        const float r02 = r0 * r0;
        const float al = r02 * (1.0f + E + 2.0f * e1) * Pq;
        const float be = r02 * (1.0f + E - 2.0f * e1) * Pq;
        const float ga = r02 * 4.0f * e2 * Pq;
        const float dk = 6.283185307179586f / ((float)N * p);
        const float invN = 1.0f / (float)N;
        const RenderPsf ps = render_psf(psf[n_psf == 1 ? 0 : i]);
        for (int m = tid; m < N; m += NT) {
            float s, co;
            sincospif(2.0f * (float)m * invN, &s, &co);
            sm.tw[m] = make_float2(co, s);
        }
        for (int u = tid; u < H; u += NT) {
            float s, co;
            sincospif(-2.0f * (float)u * th[4] * invN, &s, &co);
            sm.X[u] = make_float2(co, s);
            sincospif(-2.0f * (float)u * th[5] * invN, &s, &co);
            sm.Y[u] = make_float2(co, s);
            sm.snc[u] = r_sincpi((float)u * invN);
        }
        if (ps.kind != BS_PSF_GAUSSIAN)
            for (int j = tid; j < kNodes; j += NT)
                sm.nodes[j] = make_float2(coshf(0.125f * j), coshf(0.125f * j * fminf(ps.nu, 6.0f)));
        __syncthreads();
        // the PSF at (u, a <= u), into both (u, a) and (a, u); rows H - 1 - r and r of the
        // triangle hold H + 1 values together
        float *T = reinterpret_cast<float *>(sm.A);
        for (int it = tid; it < ((H + 1) >> 1) * (H + 1); it += NT) {
            const int r = it / (H + 1), q = it - r * (H + 1);
            const bool first = q < H - r;
            if (!first && 2 * r == H - 1) continue;   // the middle row has no partner
            const int u = first ? H - 1 - r : r, a = first ? q : q - (H - r);
            const float kx = u * dk, ky = a * dk;
            const float f = render_psf_transfer(ps, sqrtf(kx * kx + ky * ky), sm.nodes);
            T[u * H + a] = f;
            T[a * H + u] = f;
        }
        __syncthreads();
        for (int o = tid; o < H * H; o += NT) {
            const int u = o / H, a = o - u * H;
            const float kx = u * dk, ky = a * dk;
            const float q0 = al * kx * kx + be * ky * ky, q1 = ga * kx * ky;
            const float rp = rsqrtf(1.0f + (q0 + q1)), rm = rsqrtf(1.0f + (q0 - q1));
            const float f = F * T[o] * sm.snc[u] * sm.snc[a] * ((u ? 2.0f : 1.0f) * invN * invN);
            const float ap = f * rp * rp * rp, am = f * rm * rm * rm;
            const float2 X = sm.X[u], Y = sm.Y[a];
            // X Y and X conj(Y)
            const float rr = X.x * Y.x, ii = X.y * Y.y, ri = X.x * Y.y, ir = X.y * Y.x;
            const float pr = ap * (rr - ii), pi = ap * (ri + ir);
            const float mr = am * (rr + ii), mi = am * (ir - ri);
            sm.S[o] = a ? make_float4(pr + mr, pi + mi, pr - mr, pi - mi) : make_float4(pr, pi, 0.f, 0.f);
        }
        float *img = out + offsets[i];
        const int ut = (H + 3) >> 2;
        for (int y0 = 0; y0 < H; y0 += RB) {
            const int ny = min(RB, H - y0);
            __syncthreads();   // S is complete (first block), A's readers are done (later ones)
            // column pass: four rows u of two y (the second one half a block further)
            const int hy = (ny + 1) >> 1;
            for (int it = tid; it < ut * hy; it += NT) {
                const int tile = it / hy, yi = it - tile * hy;
                const int y1 = y0 + yi, y2 = min(y1 + hy, H - 1);
                const float4 *s[4];
                float2 C[4], D[4], C2[4], D2[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    s[r] = sm.S + (size_t)min(4 * tile + r, H - 1) * H;
                    C[r] = D[r] = C2[r] = D2[r] = make_float2(0.f, 0.f);
                }
                int i1 = 0, i2 = 0;
#pragma unroll 2
                for (int a = 0; a < H; ++a) {
                    const float2 t1 = sm.tw[i1], t2 = sm.tw[i2];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float4 v = s[r][a];
                        const float2 vp = make_float2(v.x, v.y), vm = make_float2(v.z, v.w);
                        C[r] = __ffma2_rn(vp, make_float2(t1.x, t1.x), C[r]);
                        D[r] = __ffma2_rn(vm, make_float2(t1.y, t1.y), D[r]);
                        C2[r] = __ffma2_rn(vp, make_float2(t2.x, t2.x), C2[r]);
                        D2[r] = __ffma2_rn(vm, make_float2(t2.y, t2.y), D2[r]);
                    }
                    i1 += y1;
                    if (i1 >= N) i1 -= N;
                    i2 += y2;
                    if (i2 >= N) i2 -= N;
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (4 * tile + r >= H) break;
                    float4 *A = sm.A + (4 * tile + r) * RB + yi;   // C + i D and C - i D
                    A[0] = make_float4(C[r].x - D[r].y, C[r].y + D[r].x, C[r].x + D[r].y, C[r].y - D[r].x);
                    if (yi + hy < ny)
                        A[hy] = make_float4(C2[r].x - D2[r].y, C2[r].y + D2[r].x, C2[r].x + D2[r].y, C2[r].y - D2[r].x);
                }
            }
            __syncthreads();
            // row pass: four values of y (eight rows) of two x (the second one H / 2 further)
            const int nq = (ny + 3) >> 2, hx = (H + 1) >> 1;
            for (int it = tid; it < nq * hx; it += NT) {
                const int q = it / hx, x1 = it - q * hx, x2 = min(x1 + hx, H - 1);
                float2 up[2][4], dn[2][4];   // (P, Q) of the rows +y and -y
#pragma unroll
                for (int r = 0; r < 4; ++r) up[0][r] = dn[0][r] = up[1][r] = dn[1][r] = make_float2(0.f, 0.f);
                const float4 *a = sm.A + 4 * q;
                int i1 = 0, i2 = 0;
#pragma unroll 2
                for (int u = 0; u < H; ++u) {
                    const float2 t1 = sm.tw[i1], t2 = sm.tw[i2];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float4 v = a[u * RB + r];
                        const float2 vu = make_float2(v.x, v.y), vd = make_float2(v.z, v.w);
                        up[0][r] = __ffma2_rn(vu, t1, up[0][r]);
                        dn[0][r] = __ffma2_rn(vd, t1, dn[0][r]);
                        up[1][r] = __ffma2_rn(vu, t2, up[1][r]);
                        dn[1][r] = __ffma2_rn(vd, t2, dn[1][r]);
                    }
                    i1 += x1;
                    if (i1 >= N) i1 -= N;
                    i2 += x2;
                    if (i2 >= N) i2 -= N;
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int y = y0 + 4 * q + r;
                    if (4 * q + r >= ny) break;
                    float *top = img + (c + y) * N + c, *bot = img + (c - y) * N + c;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int x = h ? x2 : x1;
                        if (h && x1 + hx >= H) break;
                        top[x] = up[h][r].x - up[h][r].y;
                        if (x) top[-x] = up[h][r].x + up[h][r].y;
                        if (y) {
                            bot[x] = dn[h][r].x - dn[h][r].y;
                            if (x) bot[-x] = dn[h][r].x + dn[h][r].y;
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace

// Shared memory follows the largest side of a launch (34 KB at 63 px, 70 KB at 101 px), and a
// block's tiles of the two passes keep about 2 H threads busy: stamps up to 63 px run in
// CTAs of 128 threads (24 warps per SM), larger ones in their own launch in CTAs of 256.  The
// launches pass over each other's stamps.  20,000 stamps of 25-101 px through the binding: 735 us;
// 64 and 128 threads with blocks of 16 rows 798 us (16 warps per SM); one launch of 128
// threads for all sides, with half as much work per thread and load, 847 us.
constexpr int kSmallSide = 63;

template <int NT, int RB>
static cudaError_t launch_class(int grid, int n, const float *theta, const float *shear, const int64_t *offsets,
                                const int32_t *side, int min_side, int max_side, const bs_psf *psf, int n_psf,
                                float pixel_scale, float *out, cudaStream_t stream)
{
    const size_t smem = render_smem_bytes(max_side, RB);
    // the limit is that of the largest stamp, the same from every host thread
    const cudaError_t e = cudaFuncSetAttribute(render_kernel<NT, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)render_smem_bytes(BS_MAX_SIDE, RB));
    if (e != cudaSuccess) return e;
    render_kernel<NT, RB><<<grid, NT, smem, stream>>>(n, theta, shear, offsets, side, min_side, max_side, psf, n_psf,
                                                  pixel_scale, out);
    bs::count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_render(int n, const float *theta, const float *shear, const int64_t *offsets,
                          const int32_t *side, int max_side, const bs_psf *psf, int n_psf,
                          float pixel_scale, float *out, cudaStream_t stream)
{
    if (n <= 0) return cudaSuccess;
    const int grid = n < 65535 ? n : 65535;
    if (max_side > kSmallSide) {
        const cudaError_t e = launch_class<256, 32>(grid, n, theta, shear, offsets, side, kSmallSide, max_side, psf, n_psf,
                                                pixel_scale, out, stream);
        if (e != cudaSuccess) return e;
    }
    return launch_class<128, 32>(grid, n, theta, shear, offsets, side, 0, max_side < kSmallSide ? max_side : kSmallSide,
                            psf, n_psf, pixel_scale, out, stream);
}

}  // namespace bs
