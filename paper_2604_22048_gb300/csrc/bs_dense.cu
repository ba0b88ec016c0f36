// Appendix C with a general pixel covariance Sigma (Eq. covar-pixel-likelihood):
// the fit needs its inverse, the precision P = Sigma^-1, once per galaxy.
//
// In FP64, in a scratch of the galaxy's own, n = N^2 pixels:
//   L = chol(Sigma)   right-looking, kPivot columns at a time: the pivot block, the rows
//                     below it, then a rank-kPivot update of the trailing tiles;
//   W = L^-1          row blocks in ascending order: a block's rows are finished by forward
//                     substitution, a column per thread, then subtracted from the rows below
//                     in tiles of the same kind;
//   P = W^T W         a tile per CTA at a time, stored as FP32 in the galaxy's block.
// Every element goes through the operations of the column-by-column algorithms (a product,
// rounded, then a sum or difference, rounded; in ascending order of the summation index), so
// the blocking, and the number of CTAs, do not change a bit of P.
//
// A cluster of CTAs takes a galaxy (several CTAs when there are fewer galaxies than SMs): they
// share the rows, columns and 64 x 64 tiles of every step and meet between steps; the pivot
// blocks each factors for itself.  Bound by the FP64 pipe (two operations a cycle and SM,
// n^3 of them); a tile's operands pass through shared memory, an element of it stays in a
// register over kPivot (or, for P, all) terms.
// 64 galaxies of 21 px: 50.1 ms a column at a time through global memory, one CTA per galaxy;
// 18.5 ms in clusters of two (128 SMs, FP64 pipe 73% active), 17.2 ms with the entries that are
// not needed left out of the tiles; 2,000 of 7 px 3.67, 4.53 and 3.29 ms.  Block sweeps with fused
// multiply-adds took 9 ms but round differently: some elements of P moved by an FP32 ulp.
#include <cmath>

#include <cooperative_groups.h>

#include "bs_device.cuh"
#include "bs_internal.h"

namespace bs {

namespace {

namespace cg = cooperative_groups;

constexpr int kDenseThreads = 256;
constexpr int kPivot = 32;           // columns per step
constexpr int kTile = 64;            // tile of an update
constexpr int kMaxCluster = 8;

struct DenseSmem {
    double D[kPivot][kPivot + 1];        // the pivot block and its Cholesky factor
    double rd[kPivot];                   // 1 / sqrt of the pivots
    double X[kPivot][kTile + 2];         // the operands of a tile, k-major
    double Y[kPivot][kTile + 2];
    int bad;
};

// Right-looking Cholesky of the nb x nb pivot block in sm.D (all threads); sets sm.bad where a
// pivot is not positive.  A column per step: the first warp (lane = row) forms the reciprocal and scales
// the column.  One warp, because the FP64 pipe is the SM's and a square root and a division
// cost it as much for every warp that asks: formed by all eight they were two
// microseconds of every column.
__device__ void factor_pivot(DenseSmem &sm, int nb)
{
    const int tid = threadIdx.x;
    bool bad = false;
    for (int j = 0; j < nb; ++j) {
        if (tid < 32) {
            const double d = sm.D[j][j];
            const double rd = d > 0.0 ? 1.0 / sqrt(d) : NAN;
            __syncwarp();
            if (tid == j) {
                sm.D[j][j] = d * rd;
                sm.rd[j] = rd;
            } else if (tid > j && tid < nb) {
                sm.D[tid][j] = sm.D[tid][j] * rd;
            }
        }
        __syncthreads();
        if (isnan(sm.rd[j])) {
            bad = true;
            break;
        }
        // the trailing part of the block: 8 threads per row
        const int i = tid >> 3;
        if (i > j && i < nb) {
            const double l = sm.D[i][j];
            for (int k = j + 1 + (tid & 7); k <= i; k += 8) sm.D[i][k] = sm.D[i][k] - l * sm.D[k][j];
        }
        __syncthreads();
    }
    if (tid == 0) sm.bad = bad;
    __syncthreads();
}

// Column of a tile of a thread's b-th (0..3): two in either half of the warp's 32 columns, ry the first.
__device__ __forceinline__ int tile_col(int ry, int b) { return ry + (b & 1) + 16 * (b >> 1); }

// acc[a][b] = acc[a][b] -+ sum_k X[k][rx + a] Y[k][column b], k0 <= k < nk ascending, product and sum rounded
// apart, of the first NA of a thread's rows and NB of its columns.
template <bool SUB, int NA, int NB>
__device__ __forceinline__ void tile_part(const DenseSmem &sm, int k0, int nk, int rx, int ry, double (&acc)[4][4])
{
#pragma unroll 2
    for (int k = k0; k < nk; ++k) {
        double x[NA], y[NB];
#pragma unroll
        for (int a = 0; a < NA; ++a) x[a] = sm.X[k][rx + a];
#pragma unroll
        for (int b = 0; b < NB; ++b) y[b] = sm.Y[k][tile_col(ry, b)];
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int b = 0; b < NB; ++b) acc[a][b] = SUB ? acc[a][b] - x[a] * y[b] : acc[a][b] + x[a] * y[b];
    }
}
// rows, cols: how many of the warp's 16 rows and 32 columns the matrix, or its lower triangle, has: the FP64
// pipe takes as long for entries that are not needed.  (With n = N^2 the last row block of every
// second side is one row.)
template <bool SUB>
__device__ __forceinline__ void tile_terms(const DenseSmem &sm, int k0, int nk, int rx, int ry, int rows, int cols,
                                           double (&acc)[4][4])
{
    if (rows == 1) tile_part<SUB, 1, 4>(sm, k0, nk, rx, ry, acc);
    else if (cols <= 16) tile_part<SUB, 4, 2>(sm, k0, nk, rx, ry, acc);
    else tile_part<SUB, 4, 4>(sm, k0, nk, rx, ry, acc);
}

// Tile number -> (row, column) of the lower triangle of tiles, row by row.
__device__ __forceinline__ void tile_of(int t, int &ti, int &tj)
{
    ti = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
    while (ti * (ti + 1) / 2 > t) --ti;
    tj = t - ti * (ti + 1) / 2;
}

__global__ void __launch_bounds__(kDenseThreads, 1) dense_precision_kernel(int n_gal, const int32_t *side,
                                                                           int max_side, const float *cov,
                                                                           const int64_t *offs,
                                                                           float *prec, int32_t *status,
                                                                           double *scratch, size_t scratch_per_cta)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DenseSmem &sm = *reinterpret_cast<DenseSmem *>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int G = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int n_clusters = gridDim.x / G, my_cluster = blockIdx.x / G;
    double *A = scratch + (size_t)my_cluster * G * scratch_per_cta;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int gtid = rank * nth + tid, gnth = G * nth;      // thread of the cluster
    // a thread's 4 x 4 entries of a 64 x 64 tile (tile_col): warp w has rows 16 (w mod 4) .. + 15 and columns
    // 32 (w / 4) .. + 31 (the four quarters of the SM, each with its part of the FP64 pipe, take a row
    // block each: the parts above the diagonal, and a small matrix's, leave none of them out)
    const int warp = tid >> 5, lane = tid & 31;
    const int wi = 16 * (warp & 3), wj = 32 * (warp >> 2);
    const int rx = wi + 4 * (lane >> 3), ry = wj + 2 * (lane & 7);
    // whether the warp's 16 x 32 part of the tile at (i0, j0) meets the lower triangle of n rows
    auto part_of = [&](int i0, int j0, int n) {
        const int i1 = i0 + wi, j1 = j0 + wj;
        return i1 < n && i1 + 15 >= j1;
    };
    // and how many of its columns do
    auto cols_of = [&](int i0, int j0, int n) { return min(i0 + wi + 15, n - 1) - (j0 + wj) + 1; };
    for (int gal = my_cluster; gal < n_gal; gal += n_clusters) {
        const int N = side[gal];
        if (N < 3 || N > max_side || !(N & 1)) {      // the scratch holds max_side only
            if (gtid == 0 && status) status[gal] = 2;
            continue;
        }
        const int n = N * N;
        double *W = A + (size_t)n * n;
        const float *S = cov + offs[gal];
        float *Pout = prec + offs[gal];
        for (size_t i = gtid; i < (size_t)n * n; i += gnth) A[i] = (double)S[i];
        cluster.sync();
        // ---- L, in the lower triangle of A
        bool bad = false;
        for (int p0 = 0; p0 < n; p0 += kPivot) {
            const int nb = min(kPivot, n - p0), r1 = p0 + nb;
            for (int e = tid; e < nb * nb; e += nth) {
                const int i = e / nb, j = e - i * nb;
                sm.D[i][j] = j <= i ? A[(size_t)(p0 + i) * n + p0 + j] : 0.0;
            }
            __syncthreads();
            factor_pivot(sm, nb);              // the same block in every CTA of the cluster
            if (sm.bad) {
                bad = true;
                break;
            }
            // the rows below: 32 rows at a time in shared memory, 8 threads per row
            for (int r0 = r1 + 32 * rank; r0 < n; r0 += 32 * G) {
                for (int e = tid; e < 32 * nb; e += nth) {
                    const int i = e / nb, k = e - i * nb;
                    sm.X[k][i] = r0 + i < n ? A[(size_t)(r0 + i) * n + p0 + k] : 0.0;
                }
                __syncthreads();
                const int i = tid >> 3;
                for (int j = 0; j < nb; ++j) {
                    const double l = sm.X[j][i] * sm.rd[j];
                    for (int k = j + 1 + (tid & 7); k < nb; k += 8) sm.X[k][i] = sm.X[k][i] - l * sm.D[k][j];
                    __syncwarp();              // a row's 8 threads are in one warp
                    if ((tid & 7) == 0) sm.X[j][i] = l;
                    __syncwarp();
                }
                __syncthreads();
                for (int e = tid; e < 32 * nb; e += nth) {
                    const int i2 = e / nb, k = e - i2 * nb;
                    if (r0 + i2 < n) A[(size_t)(r0 + i2) * n + p0 + k] = sm.X[k][i2];
                }
                __syncthreads();
            }
            cluster.sync();
            if (rank == 0)
                for (int e = tid; e < nb * nb; e += nth) {
                    const int i = e / nb, j = e - i * nb;
                    if (j <= i) A[(size_t)(p0 + i) * n + p0 + j] = sm.D[i][j];
                }
            // the trailing triangle, from column r1
            const int nt = (n - r1 + kTile - 1) / kTile;
            for (int t = rank; t < nt * (nt + 1) / 2; t += G) {
                int ti, tj;
                tile_of(t, ti, tj);
                const int i0 = r1 + ti * kTile, j0 = r1 + tj * kTile;
                for (int e = tid; e < kTile * nb; e += nth) {
                    const int i = e / nb, k = e - i * nb;
                    sm.X[k][i] = i0 + i < n ? A[(size_t)(i0 + i) * n + p0 + k] : 0.0;
                    sm.Y[k][i] = j0 + i < n ? A[(size_t)(j0 + i) * n + p0 + k] : 0.0;
                }
                __syncthreads();
                if (part_of(i0, j0, n)) {
                    double acc[4][4];
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const int i = i0 + rx + a, j = j0 + tile_col(ry, b);
                            acc[a][b] = i < n && j <= i ? A[(size_t)i * n + j] : 0.0;
                        }
                    tile_terms<true>(sm, 0, nb, rx, ry, n - i0 - wi, cols_of(i0, j0, n), acc);
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const int i = i0 + rx + a, j = j0 + tile_col(ry, b);
                            if (i < n && j <= i) A[(size_t)i * n + j] = acc[a][b];
                        }
                }
                __syncthreads();
            }
            cluster.sync();
        }
        if (bad) {
            if (gtid == 0 && status) status[gal] = 3;
            for (size_t i = gtid; i < (size_t)n * n; i += gnth) Pout[i] = 0.0f;
            cluster.sync();    // the scratch is rewritten by the cluster's next galaxy
            continue;
        }
        // ---- W = L^-1:  W[i][c] = (delta_ic - sum_{c <= k < i} L[i][k] W[k][c]) / L[i][i]
        for (size_t e = gtid; e < (size_t)n * n; e += gnth) W[e] = (int)e % (n + 1) == 0 ? 1.0 : 0.0;
        cluster.sync();
        for (int p0 = 0; p0 < n; p0 += kPivot) {
            const int nb = min(kPivot, n - p0), r1 = p0 + nb;
            for (int e = tid; e < nb * nb; e += nth) {
                const int i = e / nb, j = e - i * nb;
                sm.D[i][j] = A[(size_t)(p0 + i) * n + p0 + j];
            }
            __syncthreads();
            // this block's rows, a column c < r1 per thread
            for (int c = gtid; c < r1; c += gnth) {
                double w[kPivot];
#pragma unroll
                for (int i = 0; i < kPivot; ++i) w[i] = i < nb ? W[(size_t)(p0 + i) * n + c] : 0.0;
#pragma unroll
                for (int i = 0; i < kPivot; ++i) {
                    if (i < nb && p0 + i >= c) {
                        double t = w[i];
#pragma unroll
                        for (int k = 0; k < i; ++k)
                            if (p0 + k >= c) t = t - sm.D[i][k] * w[k];
                        w[i] = t / sm.D[i][i];
                        W[(size_t)(p0 + i) * n + c] = w[i];
                    }
                }
            }
            cluster.sync();
            // the rows below, columns c < r1
            const int ni = (n - r1 + kTile - 1) / kTile, nc = (r1 + kTile - 1) / kTile;
            for (int t = rank; t < ni * nc; t += G) {
                const int i0 = r1 + (t / nc) * kTile, c0 = (t % nc) * kTile;
                for (int e = tid; e < kTile * nb; e += nth) {
                    const int i = e / nb, k = e - i * nb;
                    sm.X[k][i] = i0 + i < n ? A[(size_t)(i0 + i) * n + p0 + k] : 0.0;
                }
                for (int e = tid; e < kTile * nb; e += nth) {
                    const int k = e / kTile, c = e - k * kTile;
                    sm.Y[k][c] = c0 + c < r1 ? W[(size_t)(p0 + k) * n + c0 + c] : 0.0;
                }
                __syncthreads();
                if (c0 + wj < r1 && i0 + wi < n) {
                    double acc[4][4];
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const int i = i0 + rx + a, c = c0 + tile_col(ry, b);
                            acc[a][b] = i < n && c < r1 ? W[(size_t)i * n + c] : 0.0;
                        }
                    tile_terms<true>(sm, 0, nb, rx, ry, n - i0 - wi, r1 - c0 - wj, acc);
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const int i = i0 + rx + a, c = c0 + tile_col(ry, b);
                            if (i < n && c < r1) W[(size_t)i * n + c] = acc[a][b];
                        }
                }
                __syncthreads();
            }
            cluster.sync();
        }
        // ---- P = W^T W: P[a][b] = sum_{k >= a} W[k][a] W[k][b] for b <= a (W is lower triangular)
        const int nt = (n + kTile - 1) / kTile, tiles = nt * (nt + 1) / 2;
        for (int t = rank; t < tiles; t += G) {
            int ti, tj;
            tile_of(t, ti, tj);
            const int i0 = ti * kTile, j0 = tj * kTile;
            double acc[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
            for (int k0 = i0; k0 < n; k0 += kPivot) {
                const int nk = min(kPivot, n - k0);
                __syncthreads();
                for (int e = tid; e < kTile * nk; e += nth) {
                    const int k = e / kTile, c = e - k * kTile;
                    sm.X[k][c] = i0 + c < n ? W[(size_t)(k0 + k) * n + i0 + c] : 0.0;
                    sm.Y[k][c] = j0 + c < n ? W[(size_t)(k0 + k) * n + j0 + c] : 0.0;
                }
                __syncthreads();
                // (the terms before the first row of the warp's part are products with zeros of W)
                if (part_of(i0, j0, n))
                    tile_terms<false>(sm, max(0, i0 + wi - k0), nk, rx, ry, n - i0 - wi, cols_of(i0, j0, n),
                                      acc);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int i = i0 + rx + a, j = j0 + tile_col(ry, b);
                    if (i < n && j <= i) {
                        const float v = (float)acc[a][b];
                        Pout[(size_t)i * n + j] = v;
                        Pout[(size_t)j * n + i] = v;
                    }
                }
        }
        cluster.sync();    // the scratch is rewritten by the cluster's next galaxy
    }
}

}  // namespace

}  // namespace bs

extern "C" {

size_t bs_dense_precision_workspace_bytes(int32_t max_side)
{
    if (max_side < 3 || max_side > bs::kDenseMaxSide || !(max_side & 1)) return 0;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t n = (size_t)max_side * max_side;
    return (size_t)sms * 2 * n * n * sizeof(double);
}

bs_status bs_dense_precision(int32_t n_gal, const int32_t *side, int32_t max_side, const float *cov,
                             const int64_t *cov_offsets, float *prec, int32_t *status, void *workspace,
                             size_t workspace_bytes, void *stream)
{
    if (n_gal < 0) return bs::set_error(BS_ERR_INVALID_ARG, "bs_dense_precision: n_gal < 0");
    if (n_gal == 0) return BS_OK;
    if (!side || !cov || !cov_offsets || !prec)
        return bs::set_error(BS_ERR_INVALID_ARG, "bs_dense_precision: NULL input or output");
    if (max_side < 3 || max_side > bs::kDenseMaxSide || !(max_side & 1))
        return bs::set_error(BS_ERR_INVALID_ARG, "bs_dense_precision: max_side must be odd, 3..%d",
                             bs::kDenseMaxSide);
    const size_t need = bs_dense_precision_workspace_bytes(max_side);
    if (!workspace || workspace_bytes < need)
        return bs::set_error(BS_ERR_OUT_OF_MEMORY, "bs_dense_precision: workspace of %zu bytes needed", need);
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // CTAs per galaxy: as many (a power of two up to a portable cluster) as leave no CTA without an
    // SM of its own, and no more than there are tiles to share (64 galaxies of 21 px: 17.2 ms in
    // clusters of two)
    const size_t n = (size_t)max_side * max_side;
    const int nt = ((int)n + bs::kTile - 1) / bs::kTile;
    int cluster = 1;
    while (cluster < bs::kMaxCluster && (int64_t)n_gal * 2 * cluster <= sms && nt * (nt + 1) / 2 >= 4 * cluster)
        cluster *= 2;
    const int clusters = n_gal < sms / cluster ? n_gal : sms / cluster;
    cudaError_t e = cudaFuncSetAttribute(bs::dense_precision_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(bs::DenseSmem));
    if (e != cudaSuccess)
        return bs::set_error(BS_ERR_CUDA, "bs_dense_precision: %s", cudaGetErrorString(e));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(clusters * cluster);
    lc.blockDim = dim3(bs::kDenseThreads);
    lc.dynamicSmemBytes = sizeof(bs::DenseSmem);
    lc.stream = static_cast<cudaStream_t>(stream);
    lc.attrs = attr;
    lc.numAttrs = 1;
    e = cudaLaunchKernelEx(&lc, bs::dense_precision_kernel, n_gal, side, max_side, cov, cov_offsets, prec, status,
                           static_cast<double *>(workspace), (size_t)(2 * n * n));
    bs::count_launches(1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess)
        return bs::set_error(BS_ERR_CUDA, "bs_dense_precision: launch: %s", cudaGetErrorString(e));
    return BS_OK;
}

}  // extern "C"
