// State build: sigma, O = I - sigma_Q^{-1} and log det sigma_Q of the lossy
// Gaussian output state (Methods, "Model"; "Partition function" normalisation).
//
// Uniform loss commutes with the interferometer, so with the orthogonal
// xp-form R of U,
//     sigma   = R diag(s) R^T,         s = eta sigma_in + (1 - eta)/2,
//     sigma_Q = R diag(s + 1/2) R^T,   sigma_Q^{-1} = R diag(1/(s + 1/2)) R^T,
//     log det sigma_Q = sum_j log1p(eta (2 - eta) sinh^2 r_j).
// Every entry is an independent length-2M dot product: no factorisation, one launch.
//
// What bounds it: FP64 operations, which a quarter of an SM issues one warp instruction of every
// 64 clocks, so the time is the longest chain on one warp as long as the grid does not fill the GPU
// (91 tiles at 50 modes).  Hence
//  * 8 x 8 tiles of the upper triangle, sigma and A on warps of their own, and the unitarity residual
//    |U^dag U - 1| (Hermitian: the real part with the xx tiles, the imaginary part with the xp ones)
//    on four more, in halves;
//  * the 4M weights (an exp each) computed once per cluster of eight CTAs and read through
//    distributed shared memory: computed per entry and per j, as before, the exp and the division
//    were nearly all of the time, 241 us at 50 modes on a GB300 and 446 at 100.
// Now 17 us at 50 modes and 57 at 100 (with the status' memset).  Every entry is still
// the sum over j in order, the product of the two rows' entries rounded first: log P of a pattern
// whose sum cancels by 1e25 and more moves with the last bit of O.  (Splitting the sums over x and p
// quadratures would take 15 and 37 us.)
#include <cooperative_groups.h>

#include "gbs_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kTile = 8, kEnt = kTile * kTile, kCluster = 8, kMaxModes = 128;
constexpr int kParts = 4, kStateThreads = kEnt * kParts;

__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kStateThreads)
    state_kernel(int M, int tiles, const double *__restrict__ U, const double *__restrict__ r, double eta,
                 double *__restrict__ sigma, double *__restrict__ O, double *__restrict__ logdet,
                 int32_t *__restrict__ status) {
    __shared__ double2 w[2 * kMaxModes];  // (s_j, 1 / (s_j + 1/2)), j = x then p quadratures
    __shared__ double rows[2][kTile][2 * kMaxModes + 1];  // the tile's rows i and k of R
    __shared__ double part[kParts][kEnt];
    const cg::cluster_group cl = cg::this_cluster();
    const int t = threadIdx.x, N = 2 * M, rank = (int)cl.block_rank();
    // this CTA's share of the weights: x quadratures get e^{-2r}/2, p quadratures e^{2r}/2
    for (int j = rank + kCluster * t; j < N; j += kCluster * kStateThreads) {
        const double rj = r[j < M ? j : j - M];
        const double s = eta * (0.5 * exp(j < M ? -2.0 * rj : 2.0 * rj)) + 0.5 * (1.0 - eta);
        w[j] = make_double2(s, 1.0 / (s + 0.5));
    }
    cl.sync();
    for (int j = t; j < N; j += kStateThreads)
        if ((j & (kCluster - 1)) != rank) w[j] = cl.map_shared_rank(w, j & (kCluster - 1))[j];
    cl.sync();  // the weights are in, and no CTA still reads another's when that one exits

    // tile (bi, bk), bi <= bk, of the upper triangle, in rows
    int bi = 0, rest = blockIdx.x;
    while (bi < tiles && rest >= tiles - bi) {
        rest -= tiles - bi;
        ++bi;
    }
    const int bk = bi + rest;
    if (bi < tiles) {
        // R = [[Re U, -Im U], [Im U, Re U]] in xp order
        for (int f = t; f < 2 * kTile * M; f += kStateThreads) {
            const int g = f / M, j = f - g * M, side = g >= kTile, l = g & (kTile - 1), row = (side ? bk : bi) * kTile + l;
            if (row >= N) continue;
            const bool ip = row >= M;
            const double *u = U + 2 * ((size_t)(ip ? row - M : row) * M + j);  // 8-byte aligned
            rows[side][l][j] = ip ? u[1] : u[0];
            rows[side][l][M + j] = ip ? u[0] : -u[1];
        }
        __syncthreads();
        const int e = t & (kEnt - 1), pt = t / kEnt, li = e / kTile, lk = e % kTile;
        const int i = bi * kTile + li, k = bk * kTile + lk;
        if (i < N && k < N) {
            double acc = 0.0;
            if (pt < 2) {
                const double *a = rows[0][li], *b = rows[1][lk];
#pragma unroll 4
                for (int j = 0; j < N; ++j) acc = fma(a[j] * b[j], pt ? w[j].y : w[j].x, acc);
            } else if (i < M) {
                // column i of U against column c: the real part (k < M), or the imaginary part
                const bool kp = k >= M, im = pt == 3;
                const int c = kp ? k - M : k;
                const double *a = U + 2 * i + im, *b = U + 2 * c + (im != kp);
                if (i <= c) {
#pragma unroll 4
                    for (int j = 0; j < M; ++j) acc = fma(a[(size_t)2 * j * M], b[(size_t)2 * j * M], acc);
                    if (kp && im) acc = -acc;
                }
            }
            part[pt][e] = acc;
        }
        __syncthreads();
        if (i < N && k < N) {
            if (pt == 0 && sigma && i <= k) {
                sigma[i * N + k] = part[0][e];
                sigma[k * N + i] = part[0][e];
            } else if (pt == 1 && i <= k) {
                const double v = (i == k ? 1.0 : 0.0) - part[1][e];
                O[i * N + k] = v;
                O[k * N + i] = v;
            } else if (pt == 2) {
                const double v = part[2][e] + part[3][e] - (i == k && i < M ? 1.0 : 0.0);
                if (!(fabs(v) <= 1e-10)) atomicExch(status, (int32_t)GBS_E_INVALID);
            }
        }
    }
    // log det by the last CTA of the grid: one term a thread (a sinh and a log1p are a long chain on
    // this pipe), added in the order of a warp that strides the modes
    if (blockIdx.x == gridDim.x - 1) {
        __syncthreads();
        double *term = &rows[0][0][0];
        for (int j = t; j < M; j += kStateThreads) {
            const double rj = r[j];
            if (!(rj >= 0.0) || !isfinite(rj)) atomicExch(status, (int32_t)GBS_E_INVALID);
            const double sh = sinh(rj);
            term[j] = log1p(eta * (2.0 - eta) * sh * sh);
        }
        __syncthreads();
        if (t < 32) {
            double acc = 0.0;
            for (int j = t; j < M; j += 32) acc += term[j];
            for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (t == 0) *logdet = acc;
        }
    }
}

}  // namespace

int launch_build_state(gbs_ctx *ctx, int M, const double *U, const double *r, double eta,
                       double *sigma, double *O, double *logdet, int32_t *status_dev) {
    int32_t *st = status_dev ? status_dev : ctx->dscratch;
    GBS_CUDA(ctx, cudaMemsetAsync(st, 0, sizeof(int32_t), ctx->stream));
    const int tiles = (2 * M + kTile - 1) / kTile, n = tiles * (tiles + 1) / 2;
    const int grid = (n + kCluster - 1) / kCluster * kCluster;
    state_kernel<<<grid, kStateThreads, 0, ctx->stream>>>(M, tiles, U, r, eta, sigma, O, logdet, st);
    GBS_CUDA(ctx, cudaGetLastError());
    if (status_dev) return GBS_OK;
    GBS_CUDA(ctx, cudaMemcpyAsync(ctx->pinned, st, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    GBS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    int32_t h = *(int32_t *)ctx->pinned;
    if (h) return gbs_fail(ctx, h, "gbs_build_state: U not unitary to 1e-10, or r < 0 / not finite");
    return GBS_OK;
}
