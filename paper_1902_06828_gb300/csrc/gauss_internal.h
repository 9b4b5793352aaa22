// Internal interface of the linear-Gaussian CMI kernels (not public).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace teksg {

constexpr int kGaussMaxDims = 40;   // dx + dy + dz
constexpr int kGaussMaxX = 8;       // dx

// Columns are X (dx), then Y (dy), then Z; W = (Y, Z) has dw = dy + dz
// columns.  The value of column c at point t is base[cols[c] + t].
struct GaussArgs {
    const float *base;
    const int *cols;        // [d] device
    int N, S, dx, dy, dw, d;
    const int32_t *perms;   // [S][N] surrogate permutations of the rows of X
    // the same permutations as 16-bit rows of perm_pitch entries (a multiple
    // of 8), or nullptr: read by the tensor-core contraction when set
    const uint16_t *perms16;
    int perm_pitch;
    // batched contraction: the permutations turned, entry s of point t (0: the
    // point itself) at perm_t[t * perm_t_pitch + s], or nullptr
    const uint16_t *perm_t;
    int perm_t_pitch;
    // tensor-core contraction inputs prepared once per call: W's B tiles
    // (split TF32, core-matrix layout, 8 KB per 32-point chunk and pass) and
    // the centred X columns in FP32, xcen[i * xcen_pitch + t] (pitch a
    // multiple of 32); gauss_tc_workspace bytes in all
    float *btile;
    float *xcen;
    int xcen_pitch;
    // cmi_gauss's statistics: all columns centred in FP64, cen[c * xcen_pitch + t],
    // zero past N; partial sums of the columns and of the products of column
    // pairs over kGaussParts ranges of the points; inverse factors [dw][dw] (lower)
    // and {||L_W^-1||_F^2, ||L_Z^-1||_F^2, tr S_WW, tr S_ZZ, tr S_XX}
    double *cen, *sum_part, *cov_part, *inv_w, *inv_z, *traces;
    double *mean;           // [d] (X only where own_w = 0)
    const double *meanw;    // [dw] means of the W columns: mean + dx, or another estimate's
    double *cov;            // [d][d] sample covariance, ddof = 1 (its X-W blocks are not formed:
                            // cross holds them, for every surrogate)
    double *LW, *LZ;        // [dw][dw] lower Cholesky factors of S_WW and S_ZZ
    double *norms;          // ||L_W^-1||_F^2, ||L_Z^-1||_F^2
    double *scratch;        // [kGaussMaxDims]
    int *status;            // [0] 1: a fixed block is not positive definite;
                            // [1] 1: a tensor-core wait timed out
    double *cross;          // [S + 1][dx][dw] cross-covariance of permuted X with W
    double *out, *err;      // [S + 1] estimates and error bounds
    // the W-W block of the covariance and the factors can be another
    // estimate's with the same W (own_w = 0: covw, LW, LZ, norms point there,
    // and this estimate computes only its X rows); own_w = 1: covw = cov
    const double *covw;
    int own_w;
    double *xc;             // [dx][N] X columns centred in FP64, stored as float pairs
                            // (hi, lo) when dw <= kGaussFFMaxW (batched contraction only)
    // the contraction is split along the points: split p sums chunks
    // [p * chunks_per_split, ...) into cross_part[p][S + 1][dx][dw]
    int splits, chunks_per_split;
    int group;              // chunks per FP32 accumulation group of the tensor-core contraction
    double *cross_part;
};
// chunks of 32 points per split of the tensor-core contraction (two CTAs an SM)
// and per FP32 accumulation group
int gauss_tc_split_chunks(int N, int rows, int sms, int *group);
// bytes of the tensor-core contraction's prepared inputs and the statistics
// (btile .. traces), and their pointers in a buffer at base
constexpr int kGaussParts = 8;
size_t gauss_tc_workspace(int N, int dx, int dw);
void gauss_tc_bind(GaussArgs &A, void *base);

// column sums and the contraction's inputs, then covariances and factors
cudaError_t gauss_launch_prepare(const GaussArgs &A, cudaStream_t st);
cudaError_t gauss_launch_factor(const GaussArgs &A, cudaStream_t st);
cudaError_t gauss_launch_cross_tc(const GaussArgs &A, cudaStream_t st);
double gauss_tc_gamma();   // relative error factor of the tensor-core contraction
// relative error factor of the FP64 contraction: a sum of N FP64 products
// errs by at most gamma_N sum |x||w|, gamma_N = N u / (1 - N u), u = 2^-53
// (N + 2 for the centring roundings)
__host__ __device__ inline double gauss_f64_gamma(int N)
{
    const double nu = (double)(N + 2) * 0x1p-53;
    return nu / (1.0 - nu);
}
// estimates with dw <= kGaussFFMaxW take the float-float contraction instead:
// 3 * 2^-48 per product and at most 128^2 * 2^-48 per window of kGaussFFWindow
// 32-point chunks (2^-34 covers both), then the FP64 sums
constexpr int kGaussFFMaxW = 16;
// points whose centred X column (8 bytes each) fits a CTA's shared memory; such
// estimates with dw <= kGaussFFMaxW and perm_t set gather there
constexpr int kGaussFFColMax = 26000;
// perm_t of one set: S permutations of N <= 65535 points as 32-bit rows
struct PermTurnJob {
    const int32_t *src;
    uint16_t *dst;
    int S, N, pitch;
};
cudaError_t gauss_launch_turn(const PermTurnJob *jobs_dev, const PermTurnJob *jobs_host, int n,
                              cudaStream_t st);
constexpr int kGaussFFWindow = 4;
__host__ __device__ inline double gauss_batch_gamma(int N, int dw)
{
    return gauss_f64_gamma(N) + (dw <= kGaussFFMaxW ? 0x1p-34 : 0.0);
}
// the whole FP64 pipeline (means, covariance, factors, centred X columns into
// xc, FP64 contraction and its reduction, Schur complements) for n <= 65535
// estimates in one launch per kernel: estimate i's arguments at args_dev[i]
// (device) and args_host[i]
cudaError_t gauss_launch_batch_f64(const GaussArgs *args_dev, const GaussArgs *args_host, int n,
                                   cudaStream_t st);
cudaError_t gauss_launch_schur(const GaussArgs &A, double gamma, cudaStream_t st);
// keys[2i], keys[2i + 1] = order-preserving int128 (hi, lo) of v[i]; a value
// that is not finite sets *bad
cudaError_t gauss_launch_keys(const double *v, int n, long long *keys, int *bad, cudaStream_t st);

}  // namespace teksg
