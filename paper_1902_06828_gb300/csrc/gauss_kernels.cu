// Linear-Gaussian CMI (cmi_gauss) kernels.
//
// Plug-in estimate from the sample covariance (ddof = 1) of the embedded
// variables (Methods, Vector autoregressive process: the Gaussian estimator;
// transfer entropy equals Granger causality for Gaussian variables):
//   I(X;Y|Z) = 1/2 [ln|S_XZ| + ln|S_YZ| - ln|S_Z| - ln|S_XYZ|]
//            = 1/2 [ln|Schur_X|Z| - ln|Schur_X|W|],   W = (Y, Z),
// with Schur_X|V = S_XX - S_XV S_VV^-1 S_VX.  S_XX, S_ZZ and S_WW do not
// depend on the surrogate (a permutation of the rows of X leaves S_XX
// unchanged), so they are formed and factored once in FP64; each surrogate
// only needs its cross-covariance S_XW, a contraction over the N points.
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "gauss_internal.h"

namespace teksg {

namespace {

__device__ __forceinline__ double block_sum(double v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int a = 0; a < (int)(blockDim.x >> 5); ++a) s += red[a];
    __syncthreads();
    return s;   // valid in thread 0
}

// column means: block d
__device__ __forceinline__ void gauss_mean_body(const GaussArgs &A, int d)
{
    __shared__ double red[32];
    if (!A.own_w && d >= A.dx) return;   // meanw is another estimate's
    const float *col = A.base + A.cols[d];
    double s = 0.0;
    for (int t = threadIdx.x; t < A.N; t += blockDim.x) s += (double)col[t];
    s = block_sum(s, red);
    if (threadIdx.x == 0) A.mean[d] = s / (double)A.N;
}

// covariance of columns (i, j), i <= j: block = pair index p
__device__ __forceinline__ void gauss_cov_body(const GaussArgs &A, int p)
{
    __shared__ double red[32];
    int i = 0;
    while (p >= A.d - i) {
        p -= A.d - i;
        ++i;
    }
    const int j = i + p;
    if (!A.own_w && i >= A.dx) return;   // a W-W entry: taken from covw
    if (i < A.dx && j >= A.dx) return;   // an X-W entry: in cross
    const float *ci = A.base + A.cols[i];
    const float *cj = A.base + A.cols[j];
    const double mi = i < A.dx ? A.mean[i] : A.meanw[i - A.dx];
    const double mj = j < A.dx ? A.mean[j] : A.meanw[j - A.dx];
    double s = 0.0;
    for (int t = threadIdx.x; t < A.N; t += blockDim.x)
        s += ((double)ci[t] - mi) * ((double)cj[t] - mj);
    s = block_sum(s, red);
    if (threadIdx.x == 0) {
        const double c = s / (double)(A.N - 1);
        A.cov[i * A.d + j] = c;
        A.cov[j * A.d + i] = c;
    }
}

// In-place FP64 Cholesky of an n x n SPD matrix (row-major, lower factor);
// returns false if a pivot is not positive.
__device__ bool chol(double *a, int n, int ld)
{
    for (int j = 0; j < n; ++j) {
        double s = a[j * ld + j];
        for (int k = 0; k < j; ++k) s -= a[j * ld + k] * a[j * ld + k];
        if (!(s > 0.0)) return false;
        const double l = sqrt(s);
        a[j * ld + j] = l;
        for (int i = j + 1; i < n; ++i) {
            double t = a[i * ld + j];
            for (int k = 0; k < j; ++k) t -= a[i * ld + k] * a[j * ld + k];
            a[i * ld + j] = t / l;
        }
    }
    return true;
}

// ||L^-1||_F^2 for lower-triangular L (n x n): sum of squares of the inverse
__device__ double inv_frob2(const double *L, int n, int ld, double *col)
{
    double s = 0.0;
    for (int c = 0; c < n; ++c) {
        for (int i = 0; i < n; ++i) {
            double t = (i == c) ? 1.0 : 0.0;
            for (int k = 0; k < i; ++k) t -= L[i * ld + k] * col[k];
            col[i] = i < c ? 0.0 : t / L[i * ld + i];
            s += col[i] * col[i];
        }
    }
    return s;
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// In-place FP64 Cholesky of an n x n SPD matrix (n <= 64, row-major, lower
// factor) by one warp: the pivot's sum is a warp reduction of lane-strided
// partial sums, the column below it one or two rows per lane.  False (in every
// lane) if a pivot is not positive.
__device__ bool chol_warp(double *a, int n, int ld)
{
    const int lane = threadIdx.x & 31;
    for (int j = 0; j < n; ++j) {
        double v = 0.0;
        for (int k = lane; k < j; k += 32) v += a[j * ld + k] * a[j * ld + k];
        const double s = a[j * ld + j] - warp_sum_d(v);
        if (!(s > 0.0)) return false;
        const double l = sqrt(s);
        double t[2] = {0.0, 0.0};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = j + 1 + lane + 32 * h;
            if (i < n) {
                t[h] = a[i * ld + j];
                for (int k = 0; k < j; ++k) t[h] -= a[i * ld + k] * a[j * ld + k];
            }
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = j + 1 + lane + 32 * h;
            if (i < n) a[i * ld + j] = t[h] / l;
        }
        if (lane == 0) a[j * ld + j] = l;
        __syncwarp();
    }
    return true;
}

// Largest blocks the factor kernel holds: W = (Y, Z) has at most
// kGaussMaxDims - 1 columns (X has at least one) and Z at most
// kGaussMaxDims - 2 (Y has at least one).
constexpr int kFacW = kGaussMaxDims - 1;
constexpr int kFacZ = kGaussMaxDims - 2;
constexpr int kFactorThreads = 128;

// Column c's share of ||L^-1||_F^2 for lower-triangular L (n x n, row-major,
// leading dimension ld): forward substitution of L x = e_c, the entries
// x_c .. x_{n-1} kept in xs[0 .. n - c), summed in order of rows.
__device__ double inv_col_sq(const double *L, int n, int ld, int c, double *xs)
{
    double s = 0.0;
    for (int i = c; i < n; ++i) {
        double t = (i == c) ? 1.0 : 0.0;
        for (int k = c; k < i; ++k) t -= L[i * ld + k] * xs[k - c];
        const double x = t / L[i * ld + i];
        xs[i - c] = x;
        s += x * x;
    }
    return s;
}

// Factor S_WW and S_ZZ (one CTA of kFactorThreads threads).  W = the Y then Z
// columns; Z is the trailing block of W.  Warp 0 factors S_WW while warp 1
// factors S_ZZ (GB300's FP64 pipe is narrow, so the two dependent chains run
// on different schedulers); then every column of both inverses is solved by
// a thread of its own (W's columns on threads 0-63, Z's on 64-127).  Writes
// L_W, L_Z (lower, row-major, ld = dw) and ||L^-1||_F^2 of each; status[0] = 1
// if a block is not positive definite (never cleared here, so estimates
// sharing a status word accumulate it).
__device__ __forceinline__ void gauss_factor_body(const GaussArgs &A)
{
    static_assert(kFacW <= 64 && kFacZ <= 64, "one thread per column, 64 per block");
    // the factorisations run in shared memory (a warp's dependent steps would
    // otherwise wait on global memory) and the factors are written back
    __shared__ double sW[kFacW * kFacW], sZ[kFacZ * kFacZ];
    __shared__ double xW[kFacW * (kFacW + 1) / 2], xZ[kFacZ * (kFacZ + 1) / 2];
    __shared__ double s_norm[kFactorThreads / 32];
    __shared__ int s_ok[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int dx = A.dx, dw = A.dw, dy = A.dy, dz = dw - dy, d = A.d;
    for (int e = tid; e < dw * dw; e += blockDim.x) {
        const int r = e / dw, c = e % dw;
        sW[e] = c <= r ? A.cov[(dx + r) * d + dx + c] : 0.0;
    }
    for (int e = tid; e < dz * dz; e += blockDim.x) {
        const int r = e / dz, c = e % dz;
        sZ[e] = c <= r ? A.cov[(dx + dy + r) * d + dx + dy + c] : 0.0;
    }
    __syncthreads();
    if (warp == 0) {
        const bool ok = chol_warp(sW, dw, dw);
        if (lane == 0) s_ok[0] = ok;
    } else if (warp == 1) {
        const bool ok = dz > 0 ? chol_warp(sZ, dz, dz) : true;
        if (lane == 0) s_ok[1] = ok;
    }
    __syncthreads();
    if (!(s_ok[0] && s_ok[1])) {
        if (tid == 0) A.status[0] = 1;
        return;
    }
    for (int e = tid; e < dw * dw; e += blockDim.x) A.LW[e] = sW[e];
    for (int e = tid; e < dz * dz; e += blockDim.x) A.LZ[(e / dz) * dw + e % dz] = sZ[e];
    double s = 0.0;
    if (tid < 64) {
        if (tid < dw) s = inv_col_sq(sW, dw, dw, tid, xW + tid * dw - tid * (tid - 1) / 2);
    } else {
        const int c = tid - 64;
        if (c < dz) s = inv_col_sq(sZ, dz, dz, c, xZ + c * dz - c * (c - 1) / 2);
    }
    s = warp_sum_d(s);
    if (lane == 0) s_norm[warp] = s;
    __syncthreads();
    if (tid == 0) {
        A.norms[0] = s_norm[0] + s_norm[1];
        A.norms[1] = dz > 0 ? s_norm[2] + s_norm[3] : 0.0;
    }
}

// Per surrogate (one thread): Schur complements given Z and given W, their
// log-determinants, the estimate and a first-order bound on its error from
// the cross-covariance error model |dS_XW_ij| <= gamma sqrt(S_ii S_jj), whose
// squared Frobenius norm over (a, r) is gamma^2 tr(S_XX) sum_r S_rr.  One
// thread per surrogate keeps every FP64 lane busy (a warp per surrogate was
// measured slower: GB300's FP64 pipe is narrow, so idle lanes cost more than
// the dependent chain).
// One half of a surrogate's estimate: the Schur complement of X given Z
// (which = 0, the trailing dz entries of W) or given W (which = 1) from the
// factor L (lower, row-major, ld = dw), its log-determinant and the bound
// on its error.
__device__ __forceinline__ void gauss_schur_half(const GaussArgs &A, double gamma, int s,
                                                 int which, const double *L, double &ld_out,
                                                 double &bound_out)
{
    const int dx = A.dx, dw = A.dw, dy = A.dy, dz = dw - dy, d = A.d;
    const double *c = A.cross + (size_t)s * dx * dw;   // [dx][dw]
    double v[kGaussMaxDims], Sm[kGaussMaxX * kGaussMaxX], tmp[kGaussMaxDims];
    double sxx = 0.0;
    for (int a = 0; a < dx; ++a) sxx += A.cov[a * d + a];
    const int n = which == 0 ? dz : dw;
    const int off = which == 0 ? dy : 0;
    // Sm = S_XX - V^T V, V = L^-1 C_V  (column per x dim)
    for (int a = 0; a < dx; ++a)
        for (int b = 0; b < dx; ++b) Sm[a * dx + b] = A.cov[a * d + b];
    double vnorm2 = 0.0, svv = 0.0;
    double vall[kGaussMaxX * kGaussMaxDims];
    for (int r = 0; r < n; ++r) svv += A.covw[(dx + off + r) * d + dx + off + r];
    for (int a = 0; a < dx; ++a) {
        for (int r = 0; r < n; ++r) {
            double t = c[a * dw + off + r];
            for (int k = 0; k < r; ++k) t -= L[r * dw + k] * v[k];
            v[r] = t / L[r * dw + r];
            vnorm2 += v[r] * v[r];
        }
        for (int r = 0; r < n; ++r) vall[a * kGaussMaxDims + r] = v[r];
    }
    const double dcnorm2 = gamma * gamma * sxx * svv;
    for (int a = 0; a < dx; ++a)
        for (int b = 0; b < dx; ++b) {
            double t = 0.0;
            for (int r = 0; r < n; ++r) t += vall[a * kGaussMaxDims + r] * vall[b * kGaussMaxDims + r];
            Sm[a * dx + b] -= t;
        }
    if (!chol(Sm, dx, dx)) {
        ld_out = CUDART_NAN;
        bound_out = CUDART_INF;
        return;
    }
    double l = 0.0;
    for (int a = 0; a < dx; ++a) l += 2.0 * log(Sm[a * dx + a]);
    ld_out = l;
    // d ln|Sm| <= ||Sm^-1||_F ||dSm||_F,  ||dSm||_F <= 2 ||dC||_F ||L^-1||_F ||V||_F
    const double sinv = sqrt(inv_frob2(Sm, dx, dx, tmp));
    const double linv = n > 0 ? sqrt(A.norms[which == 0 ? 1 : 0]) : 0.0;
    bound_out = sinv * 2.0 * sqrt(dcnorm2) * linv * sqrt(vnorm2);
}

__device__ __forceinline__ void gauss_schur_body(const GaussArgs &A, double gamma, int s)
{
    if (s > A.S) return;
    double ld[2], bound[2];
    for (int which = 0; which < 2; ++which)
        gauss_schur_half(A, gamma, s, which, which == 0 ? A.LZ : A.LW, ld[which], bound[which]);
    A.out[s] = 0.5 * (ld[0] - ld[1]);
    // factor 2 for second-order terms
    A.err[s] = 2.0 * 0.5 * (bound[0] + bound[1]);
}

// ---------------- tensor-core cross-covariance (tcgen05, split TF32) ----------------
// cross[s][i][n] = sum_t A[(s, i)][t] B[n][t] with A[(s, i)][t] = x_i(pi_s(t))
// - mean_i (row = (surrogate s, X dim i)) and B[n][t] = w_n(t) - mean_n.  Each
// operand is split in two TF32 parts, a = a_hi + a_lo (a_hi = tf32(a), a_lo =
// tf32(a - a_hi)); the product is a_hi b_hi + a_hi b_lo + a_lo b_hi, three
// tcgen05.mma.kind::tf32 per K step, FP32 accumulation in tensor memory.
//
// What does not depend on the surrogate is prepared once per call
// (gauss_prep_kernel): W centred in FP64 and split, already laid out as the
// MMA's B tiles (one 8 KB hi + lo tile per 32-point chunk and 32 columns),
// and X centred in FP64 and rounded to FP32 (one rounding of 2^-24).  A CTA
// owns 128 rows and a range of chunks: it copies B tiles with cp.async.bulk two
// chunks ahead, keeps the X column in shared memory (one X dimension and
// N <= kGaussColMax) or reads it through L1, gathers a chunk's A operand
// through the 16-bit permutation rows (both a chunk ahead), lets one thread
// issue the MMAs, and after every kGaussGroup chunks reads the FP32 accumulators
// (tcgen05.ld) and adds them to FP64 sums.  Operands use the canonical
// K-major layout without swizzle: 8-row x 16-byte core matrices, K-adjacent
// core matrices 128 bytes apart (leading byte offset), 8-row groups 1024 bytes
// apart (stride byte offset).
constexpr int kGaussTileM = 128;
constexpr int kGaussTileN = 32;
constexpr int kGaussKC = 32;                     // points per chunk (128 bytes of TF32)
constexpr int kGaussGroup = 4;                   // chunks per FP32 accumulation group
constexpr unsigned kGaussSpinLimit = 1u << 26;   // bounded mbarrier waits

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint32_t to_tf32(float f)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(f));
    return r;
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1u << 46;   // descriptor version for this architecture
    // base offset 0, absolute LBO mode 0, layout type 0 = no swizzle
    return d;
}

__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity)
{
    for (unsigned it = 0; it < kGaussSpinLimit; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(addr), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int a = 0; a < 16; ++a) v[a] = __uint_as_float(r[a]);
}

// byte offset of element (row, k) of a K-major no-swizzle tile with 8 core
// matrices (32 TF32 values) per row group
__device__ __forceinline__ uint32_t cm_offset(int row, int k)
{
    return (uint32_t)(((row >> 3) * 8 + (k >> 2)) * 128 + (row & 7) * 16 + (k & 3) * 4);
}

constexpr int kGaussColMax = 16384;   // X column points kept in shared memory

// ---- the statistics of one call (gauss_launch_prepare, gauss_launch_factor) ----
// GB300's FP64 pipe takes two lanes a clock and SM, so the sums are spread
// over the chip (kGaussParts ranges of the points each, added in order) and a
// term costs one FP64 operation: columns are centred once.  N = 9995: sums 24 ->
// 9 us, covariances of 39 columns 109 -> 21 us (one CTA for each before).

// partial sum of column c over range `part`: grid (d, kGaussParts)
__global__ void __launch_bounds__(128) gauss_sum_kernel(GaussArgs A)
{
    __shared__ double red[32];
    const int c = blockIdx.x, part = blockIdx.y;
    const int t0 = (int)((long long)A.N * part / kGaussParts);
    const int t1 = (int)((long long)A.N * (part + 1) / kGaussParts);
    const float *col = A.base + A.cols[c];
    double s = 0.0;
    for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x) s += (double)col[t];
    s = block_sum(s, red);
    if (threadIdx.x == 0) A.sum_part[c * kGaussParts + part] = s;
}

// Chunk blockIdx.x of 32 points: for pass blockIdx.y < passes, W's B tile
// (tile (pass, chunk) at btile + (pass * nchunks + chunk) * 2048 floats, hi
// then lo, each in the core-matrix layout of 32 columns x 32 points) and W's
// centred columns; for blockIdx.y == passes the X columns, centred in FP64
// and rounded once to FP32 for the gathers.
__global__ void __launch_bounds__(256) gauss_prep_kernel(GaussArgs A, int nchunks, int passes)
{
    __shared__ double s_mean[kGaussTileN];
    const int c = blockIdx.x, pass = blockIdx.y;
    const bool is_x = pass == passes;
    const int col0 = is_x ? 0 : A.dx + pass * kGaussTileN;
    const int n_cols = is_x ? A.dx : min(kGaussTileN, A.dw - pass * kGaussTileN);
    if (threadIdx.x < n_cols) {
        double s = 0.0;
        for (int p = 0; p < kGaussParts; ++p)
            s += A.sum_part[(col0 + threadIdx.x) * kGaussParts + p];
        s_mean[threadIdx.x] = s / (double)A.N;
    }
    __syncthreads();
    float *hb = A.btile + ((size_t)pass * nchunks + c) * 2048;
    float *lb = hb + 1024;
    for (int e = threadIdx.x; e < kGaussTileN * kGaussKC; e += blockDim.x) {
        const int n = e / kGaussKC, k = e % kGaussKC;
        const int t = c * kGaussKC + k;
        double v = 0.0;
        if (n < n_cols && t < A.N) v = (double)A.base[A.cols[col0 + n] + t] - s_mean[n];
        if (n < n_cols) A.cen[(size_t)(col0 + n) * A.xcen_pitch + t] = v;
        if (is_x) {
            if (n < n_cols) A.xcen[(size_t)n * A.xcen_pitch + t] = (float)v;
        } else {
            const float hi = __uint_as_float(to_tf32((float)v));
            const uint32_t off = cm_offset(n, k) / 4;
            hb[off] = hi;
            lb[off] = __uint_as_float(to_tf32((float)(v - (double)hi)));
        }
    }
}

// Products of the centred columns summed over range blockIdx.y for a tile of
// 4 x 4 column pairs (W-W tiles first, then X-X; X-W pairs are cross's): 16
// FP64 FMAs for 8 loads a point and thread, then a sum in thread order.
__device__ __forceinline__ void gauss_tile_pair(int t, int &i, int &j)
{
    j = 0;
    while (t > j) {
        t -= j + 1;
        ++j;
    }
    i = t;
}
__global__ void __launch_bounds__(128) gauss_cov_tiles_kernel(GaussArgs A)
{
    __shared__ double s_sum[16][129];
    const int tw = (A.dw + 3) / 4, nw = tw * (tw + 1) / 2;
    int ti, tj;
    const bool is_x = (int)blockIdx.x >= nw;
    gauss_tile_pair(is_x ? (int)blockIdx.x - nw : (int)blockIdx.x, ti, tj);
    const int c0 = is_x ? 0 : A.dx, n = is_x ? A.dx : A.dw;
    const int part = blockIdx.y, tid = threadIdx.x;
    const int t0 = (int)((long long)A.N * part / kGaussParts);
    const int t1 = (int)((long long)A.N * (part + 1) / kGaussParts);
    const double *pa[4], *pb[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {   // past the last column: the last again, not stored
        pa[a] = A.cen + (size_t)(c0 + min(4 * ti + a, n - 1)) * A.xcen_pitch;
        pb[a] = A.cen + (size_t)(c0 + min(4 * tj + a, n - 1)) * A.xcen_pitch;
    }
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
    for (int t = t0 + tid; t < t1; t += 128) {
        double va[4], vb[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            va[a] = __ldg(pa[a] + t);
            vb[a] = __ldg(pb[a] + t);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = fma(va[a], vb[b], acc[a][b]);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) s_sum[4 * a + b][tid] = acc[a][b];
    __syncthreads();
    const int v = tid >> 3, l = tid & 7;
    double s = 0.0;
    for (int e = 0; e < 16; ++e) s += s_sum[v][16 * l + e];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int i = 4 * ti + (v >> 2), j = 4 * tj + (v & 3);
    if (l == 0 && i < n && j < n && i <= j)
        A.cov_part[((size_t)part * A.d + c0 + i) * A.d + c0 + j] = s;
}

// Covariances from their parts, and the inverse of the Cholesky factor of S_WW
// (block 0) and S_ZZ (block 1; Z is the trailing block of W), as the unit
// lower inverse of an L D L^T factorisation scaled by D^-1/2 at the end.
// Right-looking, the inverse's rows updated beside the trailing block, sixteen
// lanes a row: each of the n steps is a chain of one division and one update
// (an FP64 operation's latency is some 60 clocks), where a warp's row-oriented
// factorisation and a thread's column solve were chains of ~800 (39 columns:
// 190 -> 75 us; 5 columns: 13 -> 11).
constexpr int kFactorLanes = 16;
__global__ void __launch_bounds__(kFactorLanes * 40) gauss_factor_inv_kernel(GaussArgs A)
{
    __shared__ double sA[kFacW * kFacW], sX[kFacW * kFacW];
    __shared__ double s_f[kFacW], s_red[kFactorLanes * 40 / 32];
    static_assert(kFacW <= 40, "a row per sixteen threads");
    const int tid = threadIdx.x, d = A.d, dx = A.dx;
    const int off = blockIdx.x == 0 ? 0 : A.dy, n = A.dw - off;
    auto cov = [&](int i, int j) {   // i <= j
        double v[kGaussParts], s = 0.0;
#pragma unroll
        for (int p = 0; p < kGaussParts; ++p)
            v[p] = __ldg(A.cov_part + ((size_t)p * d + i) * d + j);
#pragma unroll
        for (int p = 0; p < kGaussParts; ++p) s += v[p];
        return s / (double)(A.N - 1);
    };
    const int i = tid / kFactorLanes, l = tid % kFactorLanes;   // this thread's row and lane
    if (i < n)
        for (int c = l; c <= i; c += kFactorLanes) {
            const double v = cov(dx + off + c, dx + off + i);
            sA[i * n + c] = v;
            sX[i * n + c] = i == c ? 1.0 : 0.0;
            if (blockIdx.x == 0)
                A.cov[(dx + i) * d + dx + c] = A.cov[(dx + c) * d + dx + i] = v;
        }
    if (blockIdx.x == 0)
        for (int e = tid; e < dx * dx; e += blockDim.x) {
            const int r = e / dx, c = e - r * dx;
            if (c <= r) A.cov[r * d + c] = A.cov[c * d + r] = cov(c, r);
        }
    __syncthreads();
    if (tid < 32) {   // trace of the W (or Z) block
        double s = 0.0;
        for (int r = tid; r < n; r += 32) s += sA[r * n + r];
        s = warp_sum_d(s);
        if (tid == 0) A.traces[2 + blockIdx.x] = s;
    } else if (tid == 32 && blockIdx.x == 0) {   // and of X's
        double s = 0.0;
        for (int a = 0; a < dx; ++a) s += cov(a, a);
        A.traces[4] = s;
    }
    for (int j = 0; j < n; ++j) {
        __syncthreads();
        const double pivot = sA[j * n + j];
        if (!(pivot > 0.0)) {   // the same value for every thread
            if (tid == 0) A.status[0] = 1;
            return;
        }
        if (tid > j && tid < n) s_f[tid] = sA[tid * n + j] / pivot;
        __syncthreads();
        if (i > j && i < n) {
            const double f = s_f[i];
            for (int c = l; c <= i; c += kFactorLanes) {
                if (c <= j) sX[i * n + c] -= f * sX[j * n + c];
                else sA[i * n + c] -= f * sA[c * n + j];
            }
        }
    }
    __syncthreads();
    if (tid < n) s_f[tid] = sqrt(sA[tid * n + tid]);
    __syncthreads();
    double *inv = blockIdx.x == 0 ? A.inv_w : A.inv_z;
    double s = 0.0;
    for (int e = tid; e < n * n; e += blockDim.x) {
        const int r = e / n, c = e - r * n;
        const double v = c <= r ? sX[e] / s_f[r] : 0.0;
        inv[e] = v;
        s += v * v;
    }
    s = warp_sum_d(s);
    if ((tid & 31) == 0) s_red[tid >> 5] = s;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < kFactorLanes * 40 / 32; ++w) t += s_red[w];
        A.traces[blockIdx.x] = t;
    }
}

// 256 threads: thread (half h = tid / 128, row r = tid % 128) stages points
// 16 h .. 16 h + 15 of every chunk of row r.  A CTA works through
// chunks_per_split chunks (the grid is one wave of two CTAs an SM, so that the
// X column and the launch's other fixed work are paid once per ten chunks): the
// accumulators start anew every A.group chunks and are added to FP64 sums
// in registers.  TILES: 32-column tiles of W, all from the one staged A tile.
// Bound by a chunk's chain of gathers, operand stores, MMAs and waits (3.3 us
// with at most two CTAs an SM).  N = 9995, 1001 rows: 5 columns 39.5 us, 39
// columns 66; with a CTA per group of four chunks, a pass per 32 columns,
// per-entry bounds and operand stores of four bytes in four-way conflict: 45, 99.
template <bool COLSMEM, int TILES, bool P16>
__global__ void __launch_bounds__(256, 2) gauss_cross_tc_kernel(GaussArgs A, int nchunks)
{
    extern __shared__ unsigned char gsm_raw[];
    unsigned char *gsm = gsm_raw + ((1024u - (smem_u32(gsm_raw) & 1023u)) & 1023u);
    float *sA_hi = reinterpret_cast<float *>(gsm);
    float *sA_lo = sA_hi + kGaussTileM * kGaussKC;
    float *sB = sA_lo + kGaussTileM * kGaussKC;          // [2][TILES][2][1024]
    float *scol = sB + 2 * TILES * 2048;                 // [xcen_pitch] with COLSMEM
    __shared__ __align__(8) unsigned long long s_mbar_b[2], s_mbar_m;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;

    const int tid = threadIdx.x, warp = tid >> 5;
    const int r = tid & (kGaussTileM - 1), half = tid >> 7;
    const int rows = (A.S + 1) * A.dx;
    const int m = blockIdx.x * kGaussTileM + r;   // this thread's row
    const int split = blockIdx.y;
    const bool mvalid = m < rows;
    const int ms = mvalid ? m / A.dx : 0, mi = mvalid ? m % A.dx : 0;
    const uint16_t *perm16 =
        P16 && ms > 0 ? A.perms16 + (size_t)(ms - 1) * A.perm_pitch : nullptr;
    const int32_t *perm32 = !P16 && ms > 0 ? A.perms + (size_t)(ms - 1) * A.N : nullptr;
    const float *xg = A.xcen + (size_t)mi * A.xcen_pitch;
    const int ch0 = split * A.chunks_per_split;
    const int nch = min(nchunks, ch0 + A.chunks_per_split) - ch0;   // at least 1
    const uint32_t mbar_m = smem_u32(&s_mbar_m);
    const uint32_t mbar_b[2] = {smem_u32(&s_mbar_b[0]), smem_u32(&s_mbar_b[1])};

    // W's B tiles of the CTA's chunk c, into slot c & 1: one bulk copy of 8 KB a tile
    auto load_b = [&](int c) {
        const uint32_t bar = mbar_b[c & 1];
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"((uint32_t)(TILES * 8192))
                     : "memory");
        for (int t = 0; t < TILES; ++t) {
            const float *src = A.btile + ((size_t)t * nchunks + ch0 + c) * 2048;
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], "
                "8192, [%2];" ::"r"(smem_u32(sB + ((c & 1) * TILES + t) * 2048)),
                "l"(reinterpret_cast<uint64_t>(src)), "r"(bar)
                : "memory");
        }
    };
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "r"((uint32_t)(TILES * kGaussTileN)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        s_fail = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar_b[0]));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar_b[1]));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar_m));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        load_b(0);
        if (nch > 1) load_b(1);
    }
    if (COLSMEM) {   // the (single) X column, centred, into shared memory
        const float4 *src = reinterpret_cast<const float4 *>(A.xcen);
        float4 *dst = reinterpret_cast<float4 *>(scol);
#pragma unroll 4
        for (int e = tid; e < A.xcen_pitch / 4; e += 256) dst[e] = __ldg(src + e);
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) |
                           ((uint32_t)(kGaussTileN >> 3) << 17) |
                           ((uint32_t)(kGaussTileM >> 4) << 24);
    const uint32_t aHi = smem_u32(sA_hi), aLo = smem_u32(sA_lo);

    // Permutation entries of this thread's half chunk, two a word.  Past N any
    // index of the column will do (W's tile is zero there), and a row past the
    // last repeats row 0.
    uint32_t pv[8] = {};
    auto load_perm = [&](int ch) {
        const int k0 = ch * kGaussKC + 16 * half;
        if (!P16) return;
        if (perm16) {   // a row has perm_pitch entries, a multiple of 8, zeros past N
#pragma unroll
            for (int a = 0; a < 2; ++a)
                if (k0 + 8 * a < A.perm_pitch) {
                    const uint4 q = __ldg(reinterpret_cast<const uint4 *>(perm16 + k0) + a);
                    pv[4 * a] = q.x;
                    pv[4 * a + 1] = q.y;
                    pv[4 * a + 2] = q.z;
                    pv[4 * a + 3] = q.w;
                }
        } else {
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const uint32_t t = min(k0 + 2 * a, A.N - 1), t1 = min(k0 + 2 * a + 1, A.N - 1);
                pv[a] = t | t1 << 16;
            }
        }
    };
    float xv[16];
    auto gather = [&](int ch) {   // this thread's half of its row's chunk
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            int idx;
            if (P16) {
                idx = (int)(k & 1 ? pv[k >> 1] >> 16 : pv[k >> 1] & 0xffffu);
            } else {
                const int t = min(ch * kGaussKC + 16 * half + k, A.N - 1);
                idx = perm32 ? __ldg(perm32 + t) : t;
            }
            xv[k] = COLSMEM ? scol[idx] : __ldg(xg + idx);
        }
    };
    double sum[TILES][16];
#pragma unroll
    for (int t = 0; t < TILES; ++t)
#pragma unroll
        for (int n = 0; n < 16; ++n) sum[t][n] = 0.0;
    load_perm(ch0);
    gather(ch0);
    if (nch > 1) load_perm(ch0 + 1);
    bool failed = false;
    int c = 0;
    for (; c < nch && !failed; ++c) {
        // stage A, a core matrix row (four values) a store
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
            float hi[4], lo[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                hi[q] = __uint_as_float(to_tf32(xv[k + q]));
                lo[q] = __uint_as_float(to_tf32(__fsub_rn(xv[k + q], hi[q])));
            }
            const uint32_t off = cm_offset(r, 16 * half + k);
            *reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(sA_hi) + off) =
                make_float4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(sA_lo) + off) =
                make_float4(lo[0], lo[1], lo[2], lo[3]);
        }
        // generic-proxy smem writes -> visible to the tensor core (async proxy)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // without its B tiles the chunk's commit stays out and every wait below ends
            if (!mbar_wait(mbar_b[c & 1], (uint32_t)(c >> 1) & 1u)) {
                atomicExch(&s_fail, 1);
            } else {
#pragma unroll
                for (int t = 0; t < TILES; ++t) {
                    const uint32_t bHi = smem_u32(sB + ((c & 1) * TILES + t) * 2048);
                    const uint32_t bLo = bHi + 4096, acc = tmem + (uint32_t)(t * kGaussTileN);
#pragma unroll
                    for (int q = 0; q < kGaussKC / 8; ++q) {   // K = 8 TF32 per MMA
                        const uint32_t ko = q * 256;            // two core matrices along K
                        const uint64_t dAh = smem_desc(aHi + ko, 128, 1024);
                        const uint64_t dAl = smem_desc(aLo + ko, 128, 1024);
                        const uint64_t dBh = smem_desc(bHi + ko, 128, 1024);
                        const uint64_t dBl = smem_desc(bLo + ko, 128, 1024);
                        mma_tf32(acc, dAh, dBh, idesc,
                                 (c % A.group == 0 && q == 0) ? 0u : 1u);
                        mma_tf32(acc, dAh, dBl, idesc, 1u);
                        mma_tf32(acc, dAl, dBh, idesc, 1u);
                    }
                }
                asm volatile(
                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                    ::"r"(mbar_m)
                    : "memory");
            }
        }
        if (c + 1 < nch) {   // the next chunk's values while the MMAs run
            gather(ch0 + c + 1);
            if (c + 2 < nch) load_perm(ch0 + c + 2);
        }
        // every thread waits: the MMAs have read the A and B tiles before they
        // are written again, and have written the accumulators
        if (!mbar_wait(mbar_m, (uint32_t)c & 1u)) atomicExch(&s_fail, 1);
        __syncthreads();
        failed = s_fail != 0;
        if (failed) break;
        if (tid == 0 && c + 2 < nch) load_b(c + 2);
        if ((c + 1) % A.group == 0 || c + 1 == nch) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int t = 0; t < TILES; ++t) {
                // warps w and w + 4 share TMEM lanes 32 (w % 4) ..; each reads 16 columns
                float v[16];
                tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) +
                              (uint32_t)(t * kGaussTileN) + 16u * half,
                          v);
#pragma unroll
                for (int n = 0; n < 16; ++n) sum[t][n] += (double)v[n];
            }
        }
    }
    if (failed) {
        // bounded waits for the copies and the MMAs in flight before anything is freed
        if (tid == 0) {
            atomicExch(A.status + 1, 1);
            mbar_wait(mbar_b[c & 1], (uint32_t)(c >> 1) & 1u);
            if (c + 1 < nch) mbar_wait(mbar_b[(c + 1) & 1], (uint32_t)((c + 1) >> 1) & 1u);
        }
        mbar_wait(mbar_m, (uint32_t)c & 1u);
    } else if (mvalid) {
        double *part = A.cross_part + ((size_t)split * rows + m) * A.dw + 16 * half;
#pragma unroll
        for (int t = 0; t < TILES; ++t)
#pragma unroll
            for (int n = 0; n < 16; ++n)
                if (t * kGaussTileN + 16 * half + n < A.dw) part[t * kGaussTileN + n] = sum[t][n];
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"((uint32_t)(TILES * kGaussTileN)));
}

// cross = (sum of the splits' partial sums, in split order) / (N - 1)
__device__ __forceinline__ void gauss_cross_reduce_body(const GaussArgs &A, long long e)
{
    const long long total = (long long)(A.S + 1) * A.dx * A.dw;
    if (e >= total) return;
    double s = 0.0;
    int p = 0;
    for (; p + 16 <= A.splits; p += 16) {   // the loads of 16 splits together, added in order
        double v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = __ldg(A.cross_part + (size_t)(p + u) * total + e);
#pragma unroll
        for (int u = 0; u < 16; ++u) s += v[u];
    }
    for (; p < A.splits; ++p) s += A.cross_part[(size_t)p * total + e];
    A.cross[e] = s * (1.0 / (double)(A.N - 1));
}

// FP64 cross-covariance on the CUDA cores, for estimates whose decisions must
// agree with an FP64 evaluation down to near-ties (network inference): the same
// sums as the tensor-core kernel, every product and addition in FP64.  One
// thread per row (surrogate s, X dim a) holds its dw sums in registers; the
// block stages the centred W values of each 32-point chunk in shared memory
// (read as broadcasts) and each thread gathers its permuted X values.  The
// points are split into A.splits ranges of chunks_per_split chunks (grid y),
// and the tensor-core kernel's reduction adds the splits in order.
constexpr int kF64Rows = 128;
// DW4 = dw rounded up to a multiple of 2: the W values past dw are staged as
// zeros, so the inner loop has no per-column guard (a guarded loop unrolled to
// the 32-column maximum would issue 32 FP64 FMAs per point whatever dw is).
// The X values are gathered already centred (gauss_centre_batch), so a point
// costs one FP64 FMA per column and nothing else on the FP64 pipe.
template <int DW4>
__device__ __forceinline__ void gauss_cross_f64_body(const GaussArgs &A, int bx, int by,
                                                     double (*sW)[kGaussMaxDims])
{
    const int rows = (A.S + 1) * A.dx, dw = A.dw;
    const int row = bx * kF64Rows + threadIdx.x;
    const bool live = row < rows;
    const int s = live ? row / A.dx : 0, a = live ? row % A.dx : 0;
    const int32_t *pi = s > 0 ? A.perms + (size_t)(s - 1) * A.N : nullptr;
    const double *xcol = A.xc + (size_t)a * A.N;
    double acc[DW4];
#pragma unroll
    for (int w = 0; w < DW4; ++w) acc[w] = 0.0;
    const int nchunks = (A.N + kGaussKC - 1) / kGaussKC;
    const int c0 = by * A.chunks_per_split;
    const int c1 = min(nchunks, c0 + A.chunks_per_split);
    for (int c = c0; c < c1; ++c) {
        const int t0 = c * kGaussKC, n = min(kGaussKC, A.N - t0);
        __syncthreads();
        for (int e = threadIdx.x; e < kGaussKC * DW4; e += kF64Rows) {
            const int t = e / DW4, w = e - t * DW4;
            sW[t][w] = (t < n && w < dw)
                           ? (double)A.base[A.cols[A.dx + w] + t0 + t] - A.meanw[w]
                           : 0.0;
        }
        __syncthreads();
        if (!live) continue;
#pragma unroll 4
        for (int t = 0; t < n; ++t) {
            const int src = pi ? pi[t0 + t] : t0 + t;
            const double xv = xcol[src];
#pragma unroll
            for (int w = 0; w < DW4; ++w) acc[w] = fma(xv, sW[t][w], acc[w]);
        }
    }
    if (!live) return;
    double *dst = A.cross_part + ((size_t)by * rows + row) * dw;
#pragma unroll
    for (int w = 0; w < DW4; ++w)
        if (w < dw) dst[w] = acc[w];
}

// The same sums in float-float arithmetic on the FP32 pipe, for dw <= 16
// (GB300's FP32 pipe is far wider than its FP64 one).  X and W are centred in
// FP64 and split into two floats, v = hi + lo; a product is hi*hi exactly (the
// rounded product and its FMA residual) plus the cross terms hi*lo + lo*hi by
// FMA (lo*lo, about 2^-48 relative, is dropped); the chunk's products are
// added into a float pair by error-free two-sums, and every 32-point chunk the
// pair is flushed into an FP64 sum.  About 3 * 2^-48 relative error per
// product and n^2 * 2^-48 per 32-term window at worst.
template <int DW>
__device__ __forceinline__ void gauss_cross_ff_body(const GaussArgs &A, int bx, int by,
                                                    float2 (*sW)[kGaussMaxDims])
{
    const int rows = (A.S + 1) * A.dx, dw = A.dw;
    const int row = bx * kF64Rows + threadIdx.x;
    const bool live = row < rows;
    const int s = live ? row / A.dx : 0, a = live ? row % A.dx : 0;
    const int32_t *pi = s > 0 ? A.perms + (size_t)(s - 1) * A.N : nullptr;
    const float2 *xcol = reinterpret_cast<const float2 *>(A.xc) + (size_t)a * A.N;
    double acc[DW];
#pragma unroll
    for (int w = 0; w < DW; ++w) acc[w] = 0.0;
    const int nchunks = (A.N + kGaussKC - 1) / kGaussKC;
    const int c0 = by * A.chunks_per_split;
    const int c1 = min(nchunks, c0 + A.chunks_per_split);
    // the float pair sums kGaussFFWindow chunks (128 points) before each FP64
    // flush: the flushes run on GB300's narrow FP64 pipe
    float sh[DW], sl[DW];
#pragma unroll
    for (int w = 0; w < DW; ++w) sh[w] = sl[w] = 0.f;
    for (int c = c0; c < c1; ++c) {
        const int t0 = c * kGaussKC, n = min(kGaussKC, A.N - t0);
        __syncthreads();
        for (int e = threadIdx.x; e < kGaussKC * DW; e += kF64Rows) {
            const int t = e / DW, w = e - t * DW;
            float2 v = make_float2(0.f, 0.f);
            if (t < n && w < dw) {
                const double d = (double)A.base[A.cols[A.dx + w] + t0 + t] - A.meanw[w];
                v.x = (float)d;
                v.y = (float)(d - (double)v.x);
            }
            sW[t][w] = v;
        }
        __syncthreads();
        if (!live) continue;
        for (int t8 = 0; t8 < n; t8 += 8) {
            // eight permutation entries, then eight X values, before any is used
            int src[8];
            float2 xs[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = min(t8 + u, n - 1);   // past n: W is zero there
                src[u] = pi ? pi[t0 + t] : t0 + t;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) xs[u] = xcol[src[u]];
#pragma unroll
            for (int u = 0; u < 8; ++u) {   // t <= 31: t8 <= 24
                const int t = t8 + u;
                const float2 x = xs[u];
#pragma unroll
                for (int w = 0; w < DW; ++w) {
                    const float2 y = sW[t][w];
                    const float p = __fmul_rn(x.x, y.x);
                    float e = __fmaf_rn(x.x, y.x, -p);
                    e = __fmaf_rn(x.x, y.y, e);
                    e = __fmaf_rn(x.y, y.x, e);
                    const float sn = __fadd_rn(sh[w], p);
                    const float bp = __fsub_rn(sn, sh[w]);
                    const float er =
                        __fadd_rn(__fsub_rn(sh[w], __fsub_rn(sn, bp)), __fsub_rn(p, bp));
                    sl[w] = __fadd_rn(sl[w], __fadd_rn(er, e));
                    sh[w] = sn;
                }
            }
        }
        if ((c - c0) % kGaussFFWindow == kGaussFFWindow - 1 || c == c1 - 1) {
#pragma unroll
            for (int w = 0; w < DW; ++w) {
                acc[w] += (double)sh[w] + (double)sl[w];
                sh[w] = sl[w] = 0.f;
            }
        }
    }
    if (!live) return;
    double *dst = A.cross_part + ((size_t)by * rows + row) * dw;
#pragma unroll
    for (int w = 0; w < DW; ++w)
        if (w < dw) dst[w] = acc[w];
}

// The permutations of a set, turned: [S][N] 32-bit rows -> [N][pitch] 16-bit
// entries, column 0 the identity, so that the rows a warp serves (consecutive
// surrogates) read one point's indices as one line.
__global__ void __launch_bounds__(256) gauss_turn_kernel(const PermTurnJob *jobs)
{
    __shared__ uint16_t tile[64][66];
    const PermTurnJob J = jobs[blockIdx.z];
    const int t0 = blockIdx.x * 64, s0 = blockIdx.y * 64;
    if (t0 >= J.N || s0 >= J.pitch) return;
    for (int e = threadIdx.x; e < 64 * 64; e += 256) {
        const int s = e >> 6, t = e & 63;
        int v = 0;
        if (t0 + t < J.N) {
            if (s0 + s == 0) v = t0 + t;
            else if (s0 + s <= J.S) v = J.src[(size_t)(s0 + s - 1) * J.N + t0 + t];
        }
        tile[t][s] = (uint16_t)v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 64 * 32; e += 256) {
        const int t = e >> 5, s = 2 * (e & 31);
        if (t0 + t < J.N && s0 + s < J.pitch)
            *reinterpret_cast<uint32_t *>(J.dst + (size_t)(t0 + t) * J.pitch + s0 + s) =
                *reinterpret_cast<const uint32_t *>(&tile[t][s]);
    }
}

// The float-float contraction of gauss_cross_ff_body with its gathers in
// shared memory.  One thread per surrogate and X dimension; the CTA keeps the
// centred X column there (80 KB at N = 10^4, two CTAs an SM) and reads the
// turned permutations, so that a warp's 32 gathers cost their bank conflicts
// (about 7 cycles of 8-byte loads) and its 32 indices one line, where gathers
// through L1 took a cycle per row each for the indices and the values (64
// cycles a point, against 12 of arithmetic at dw = 4).  All launches of a
// 10-node network (N = 9995, 201 rows an estimate): 22.1 -> 9.5 ms; issue 56 to 69%
// and the shared-memory pipe 59 to 74% busy.
// smem: N float2
//
// The CTA's H parts of `rows` threads take consecutive splits of the points
// with one copy of the column: seven warps (201 surrogates) an SM's half would
// not cover the latency of the index loads, which also run eight points ahead.
constexpr int kFFTile = 64;   // points of W staged at a time
template <int DW, int H>
__device__ __forceinline__ void gauss_cross_col_body(const GaussArgs &A, int bx, int by, int rows_t,
                                                     const float2 *col, float2 (*sWh)[DW])
{
    const int part = H == 1 ? 0 : (int)threadIdx.x / rows_t;
    const int tid = (int)threadIdx.x - part * rows_t;
    const int split = by * H + part;
    const int nb = (A.S + rows_t) / rows_t;   // blocks of surrogates per X dimension
    const int a = bx / nb, s = (bx - a * nb) * rows_t + tid, dw = A.dw;
    const bool live = s <= A.S && split < A.splits;
    const uint16_t *pt = A.perm_t + min(s, A.S);
    const size_t pitch = (size_t)A.perm_t_pitch;
    float2 (*sW)[DW] = sWh + part * kFFTile;
    double acc[DW];
    float sh[DW], sl[DW];
#pragma unroll
    for (int w = 0; w < DW; ++w) {
        acc[w] = 0.0;
        sh[w] = sl[w] = 0.f;
    }
    const int span = A.chunks_per_split * kGaussKC;
    const int t_begin = split * span;
    const int t_end = min(A.N, t_begin + span);   // may lie below t_begin in the last CTA
    int src[8];
    auto load_src = [&](int t) {
#pragma unroll
        for (int u = 0; u < 8; ++u) src[u] = pt[(size_t)min(t + u, A.N - 1) * pitch];
    };
    load_src(t_begin);
    int window = 0;   // points in the float pairs since their last flush
    for (int dt = 0; dt < span; dt += kFFTile) {   // the same steps in every part
        const int t0 = t_begin + dt, n = min(kFFTile, t_end - t0);
        __syncthreads();
        for (int e = tid; e < kFFTile * DW; e += rows_t) {
            const int t = e / DW, w = e - t * DW;
            float2 v = make_float2(0.f, 0.f);
            if (t < n && w < dw) {
                const double d = (double)A.base[A.cols[A.dx + w] + t0 + t] - A.meanw[w];
                v.x = (float)d;
                v.y = (float)(d - (double)v.x);
            }
            sW[t][w] = v;
        }
        __syncthreads();
        for (int t8 = 0; t8 < n; t8 += 8) {   // past n: W is zero
            float2 xs[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) xs[u] = col[src[u]];
            load_src(t0 + t8 + 8);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float2 x = xs[u];
#pragma unroll
                for (int w = 0; w < DW; ++w) {
                    const float2 y = sW[t8 + u][w];
                    const float p = __fmul_rn(x.x, y.x);
                    float e = __fmaf_rn(x.x, y.x, -p);
                    e = __fmaf_rn(x.x, y.y, e);
                    e = __fmaf_rn(x.y, y.x, e);
                    const float sn = __fadd_rn(sh[w], p);
                    const float bp = __fsub_rn(sn, sh[w]);
                    const float er =
                        __fadd_rn(__fsub_rn(sh[w], __fsub_rn(sn, bp)), __fsub_rn(p, bp));
                    sl[w] = __fadd_rn(sl[w], __fadd_rn(er, e));
                    sh[w] = sn;
                }
            }
        }
        window += kFFTile;
        if (window >= kGaussFFWindow * kGaussKC || dt + kFFTile >= span) {
            window = 0;
#pragma unroll
            for (int w = 0; w < DW; ++w) {
                acc[w] += (double)sh[w] + (double)sl[w];
                sh[w] = sl[w] = 0.f;
            }
        }
    }
    if (!live) return;
    const int rows = (A.S + 1) * A.dx;
    double *dst = A.cross_part + ((size_t)split * rows + (size_t)s * A.dx + a) * dw;
#pragma unroll
    for (int w = 0; w < DW; ++w)
        if (w < dw) dst[w] = acc[w];
}

// Estimates whose contraction runs there, in two kernels by register use
constexpr int kFFSmallW = 8;
__device__ __forceinline__ bool gauss_takes_col(const GaussArgs &A)
{
    return A.perm_t != nullptr && A.dw <= kGaussFFMaxW && A.N <= kGaussFFColMax;
}

template <int H>
__global__ void __launch_bounds__(256 * H, 2) gauss_cross_col_batch(const GaussArgs *args,
                                                                    int rows_t)
{
    constexpr bool kSmall = H > 1;
    constexpr int WMAX = kSmall ? kFFSmallW : kGaussFFMaxW;
    extern __shared__ __align__(16) float2 ccol[];
    __shared__ __align__(16) float2 sW[H * kFFTile * WMAX];
    const GaussArgs A = args[blockIdx.z];
    const int nb = (A.S + rows_t) / rows_t;
    if (!gauss_takes_col(A) || (A.dw <= kFFSmallW) != kSmall || (int)blockIdx.x >= nb * A.dx ||
        (int)blockIdx.y * H >= A.splits)
        return;
    const int a = (int)blockIdx.x / nb;
    const float2 *src = reinterpret_cast<const float2 *>(A.xc) + (size_t)a * A.N;
    for (int t = threadIdx.x; t < A.N; t += blockDim.x) ccol[t] = __ldg(src + t);
#define TE_COL_CASE(DW)                                                                          \
    gauss_cross_col_body<DW, H>(A, blockIdx.x, blockIdx.y, rows_t, ccol,                         \
                                reinterpret_cast<float2 (*)[DW]>(sW))
    if constexpr (kSmall) {
        switch (A.dw) {
        case 1: TE_COL_CASE(1); break;
        case 2: TE_COL_CASE(2); break;
        case 3: TE_COL_CASE(3); break;
        case 4: TE_COL_CASE(4); break;
        case 5: TE_COL_CASE(5); break;
        case 6: TE_COL_CASE(6); break;
        case 7: TE_COL_CASE(7); break;
        default: TE_COL_CASE(8); break;
        }
    } else {
        switch ((A.dw + 1) >> 1) {
        case 5: TE_COL_CASE(10); break;
        case 6: TE_COL_CASE(12); break;
        case 7: TE_COL_CASE(14); break;
        default: TE_COL_CASE(16); break;
        }
    }
#undef TE_COL_CASE
}

__device__ __forceinline__ void gauss_cross_f64_any(const GaussArgs &A, int bx, int by)
{
    __shared__ double sW[kGaussKC][kGaussMaxDims];
    float2 (*sF)[kGaussMaxDims] = reinterpret_cast<float2 (*)[kGaussMaxDims]>(sW);
    switch ((A.dw + 1) >> 1) {
    case 0:
    case 1: gauss_cross_ff_body<2>(A, bx, by, sF); return;
    case 2: gauss_cross_ff_body<4>(A, bx, by, sF); return;
    case 3: gauss_cross_ff_body<6>(A, bx, by, sF); return;
    case 4: gauss_cross_ff_body<8>(A, bx, by, sF); return;
    case 5: gauss_cross_ff_body<10>(A, bx, by, sF); return;
    case 6: gauss_cross_ff_body<12>(A, bx, by, sF); return;
    case 7: gauss_cross_ff_body<14>(A, bx, by, sF); return;
    case 8: gauss_cross_ff_body<16>(A, bx, by, sF); return;
    default: break;
    }
    switch ((A.dw + 1) >> 1) {
    case 9: gauss_cross_f64_body<18>(A, bx, by, sW); break;
    case 10: gauss_cross_f64_body<20>(A, bx, by, sW); break;
    case 11: gauss_cross_f64_body<22>(A, bx, by, sW); break;
    case 12: gauss_cross_f64_body<24>(A, bx, by, sW); break;
    case 13: gauss_cross_f64_body<26>(A, bx, by, sW); break;
    case 14: gauss_cross_f64_body<28>(A, bx, by, sW); break;
    case 15: gauss_cross_f64_body<30>(A, bx, by, sW); break;
    case 16: gauss_cross_f64_body<32>(A, bx, by, sW); break;
    case 17: gauss_cross_f64_body<34>(A, bx, by, sW); break;
    case 18: gauss_cross_f64_body<36>(A, bx, by, sW); break;
    case 19: gauss_cross_f64_body<38>(A, bx, by, sW); break;
    default: gauss_cross_f64_body<40>(A, bx, by, sW); break;
    }
}

// Order-preserving integer image of the estimates, in the (hi, lo) int128 form
// the test-statistics kernel compares: key(a) < key(b) exactly when a < b
// (sign-magnitude bits turned into two's complement order; -0 taken as +0).
// A value that is not finite (a singular Schur complement) sets *bad.
__global__ void gauss_keys_kernel(const double *v, int n, long long *keys, int *bad)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = v[i] + 0.0;
    if (!isfinite(x)) *bad = 1;
    const long long b = __double_as_longlong(x);
    const long long k = b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
    keys[2 * (size_t)i] = k < 0 ? -1 : 0;
    keys[2 * (size_t)i + 1] = k;
}

// Single-call Schur step.  V = L^-1 C_V by the inverse factor, eight lanes
// per surrogate and block (Z, W) taking every eighth row, so that no lane waits
// on another's rows; S_XX - V^T V, its log-determinant and the bound are then
// done for all of the CTA's surrogates by one warp (FP64 instructions cost 16
// clocks a warp however many lanes take part).  1001 rows of 39 columns: 123 ->
// 19 us, of 5 columns: 15 -> 8 (a thread per row and block, solving by rows).  DX: X dimensions, 1 or up to 8.
constexpr int kSchurS = 8;        // surrogates per CTA
constexpr int kSchurThreads = kSchurS * 16;
template <int DX>
__global__ void __launch_bounds__(kSchurThreads) gauss_schur_kernel(GaussArgs A, double gamma)
{
    constexpr int NP = DX * (DX + 1) / 2;
    __shared__ double s_inv[2][kFacW * kFacW];
    __shared__ double s_c[kSchurS][DX * (kGaussMaxDims - DX)];
    __shared__ double s_dot[kSchurS * 2][NP];
    const int tid = threadIdx.x, dx = DX == 1 ? 1 : A.dx, dw = A.dw, dy = A.dy, dz = dw - dy;
    const int d = A.d, s0 = blockIdx.x * kSchurS;
    for (int e = tid; e < dw * dw; e += kSchurThreads) s_inv[1][e] = A.inv_w[e];
    for (int e = tid; e < dz * dz; e += kSchurThreads) s_inv[0][e] = A.inv_z[e];
    const int per = dx * dw;
    for (int e = tid; e < kSchurS * per; e += kSchurThreads) {
        const int s = e / per;
        s_c[s][e - s * per] = s0 + s <= A.S ? A.cross[(size_t)(s0 + s) * per + e - s * per] : 0.0;
    }
    __syncthreads();
    const int s = tid >> 4, which = (tid >> 3) & 1, l = tid & 7;
    const int n = which == 0 ? dz : dw, off = which == 0 ? dy : 0;
    double dot[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) dot[p] = 0.0;
    for (int r = l; r < n; r += 8) {
        double v[DX];
#pragma unroll
        for (int a = 0; a < DX; ++a) {
            v[a] = 0.0;
            if (a < dx) {
                double t0 = 0.0, t1 = 0.0;
                int k = 0;
                for (; k + 1 <= r; k += 2) {
                    t0 = fma(s_inv[which][r * n + k], s_c[s][a * dw + off + k], t0);
                    t1 = fma(s_inv[which][r * n + k + 1], s_c[s][a * dw + off + k + 1], t1);
                }
                if (k <= r) t0 = fma(s_inv[which][r * n + k], s_c[s][a * dw + off + k], t0);
                v[a] = t0 + t1;
            }
        }
#pragma unroll
        for (int a = 0, p = 0; a < DX; ++a)
#pragma unroll
            for (int b = 0; b <= a; ++b, ++p) dot[p] = fma(v[a], v[b], dot[p]);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) dot[p] += __shfl_xor_sync(0xffffffffu, dot[p], o);
        if (l == 0) s_dot[2 * s + which][p] = dot[p];
    }
    __syncthreads();
    if (tid >= 32) return;
    // lane 2 s + which
    double ld = 0.0, bound = 0.0;
    const int sl = tid >> 1, w = tid & 1;
    if (tid < 2 * kSchurS) {
        double Sm[DX * DX], tmp[DX], vnorm2 = 0.0;
#pragma unroll
        for (int a = 0, p = 0; a < DX; ++a)
#pragma unroll
            for (int b = 0; b <= a; ++b, ++p)
                if (a < dx) {
                    const double t = s_dot[tid][p];
                    if (a == b) vnorm2 += t;
                    Sm[a * dx + b] = Sm[b * dx + a] = A.cov[a * d + b] - t;
                }
        if (!chol(Sm, dx, dx)) {
            ld = CUDART_NAN;
            bound = CUDART_INF;
        } else {
            for (int a = 0; a < dx; ++a) ld += 2.0 * log(Sm[a * dx + a]);
            // d ln|Sm| <= ||Sm^-1||_F ||dSm||_F,  ||dSm||_F <= 2 ||dC||_F ||L^-1||_F ||V||_F
            const double sinv = sqrt(inv_frob2(Sm, dx, dx, tmp));
            const double linv = (w == 0 ? dz : dw) > 0 ? sqrt(A.traces[1 - w]) : 0.0;
            const double svv = (w == 0 ? dz : dw) > 0 ? A.traces[3 - w] : 0.0;
            const double dcnorm2 = gamma * gamma * A.traces[4] * svv;
            bound = sinv * 2.0 * sqrt(dcnorm2) * linv * sqrt(vnorm2);
        }
    }
    const double ld_o = __shfl_xor_sync(0xffffffffu, ld, 1);
    const double bound_o = __shfl_xor_sync(0xffffffffu, bound, 1);
    if (tid < 2 * kSchurS && w == 0 && s0 + sl <= A.S) {
        A.out[s0 + sl] = 0.5 * (ld - ld_o);
        // factor 2 for second-order terms
        A.err[s0 + sl] = 2.0 * 0.5 * (bound + bound_o);
    }
}
__global__ void gauss_cross_reduce_kernel(GaussArgs A)
{
    gauss_cross_reduce_body(A, blockIdx.x * (long long)blockDim.x + threadIdx.x);
}

// The same kernels over a batch of estimates: estimate blockIdx.z, its
// arguments read from args; blocks beyond the estimate's own grid return.
__global__ void gauss_mean_batch(const GaussArgs *args)
{
    const GaussArgs A = args[blockIdx.z];
    if ((int)blockIdx.x < A.d) gauss_mean_body(A, blockIdx.x);
}
// xc[a][t] = x_a(t) - mean_a in FP64 (as a float pair hi + lo when the
// float-float contraction takes the estimate), grid y = X dim a
__global__ void gauss_centre_batch(const GaussArgs *args)
{
    const GaussArgs A = args[blockIdx.z];
    const int a = blockIdx.y;
    if (a >= A.dx) return;
    const float *col = A.base + A.cols[a];
    const double m = A.mean[a];
    const bool ff = A.dw <= kGaussFFMaxW;   // float pairs for the float-float contraction
    double *dst = A.xc + (size_t)a * A.N;
    float2 *dst2 = reinterpret_cast<float2 *>(A.xc) + (size_t)a * A.N;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < A.N; t += gridDim.x * blockDim.x) {
        const double d = (double)col[t] - m;
        if (ff) {
            const float hi = (float)d;
            dst2[t] = make_float2(hi, (float)(d - (double)hi));
        } else {
            dst[t] = d;
        }
    }
}
__global__ void gauss_cov_batch(const GaussArgs *args)
{
    const GaussArgs A = args[blockIdx.z];
    if ((int)blockIdx.x < A.d * (A.d + 1) / 2) gauss_cov_body(A, blockIdx.x);
}
__global__ void gauss_factor_batch(const GaussArgs *args)
{
    const GaussArgs A = args[blockIdx.z];
    if (A.own_w) gauss_factor_body(A);
}
__global__ void __launch_bounds__(kF64Rows) gauss_cross_f64_batch(const GaussArgs *args)
{
    const GaussArgs A = args[blockIdx.z];
    if (gauss_takes_col(A)) return;
    if ((int)blockIdx.x * kF64Rows < (A.S + 1) * A.dx && (int)blockIdx.y < A.splits)
        gauss_cross_f64_any(A, blockIdx.x, blockIdx.y);
}
__global__ void gauss_cross_reduce_batch(const GaussArgs *args)
{
    const GaussArgs A = args[blockIdx.z];
    gauss_cross_reduce_body(A, blockIdx.x * (long long)blockDim.x + threadIdx.x);
}
__global__ void gauss_schur_f64_batch(const GaussArgs *args)
{
    const GaussArgs A = args[blockIdx.z];
    gauss_schur_body(A, gauss_batch_gamma(A.N, A.dw), blockIdx.x * blockDim.x + threadIdx.x);
}

}  // namespace

cudaError_t gauss_launch_batch_f64(const GaussArgs *args_dev, const GaussArgs *args_host, int n,
                                   cudaStream_t st)
{
    if (n < 1) return cudaSuccess;
    if (n > 65535) return cudaErrorInvalidValue;
    int md = 1, mrb = 1, msp = 1, ms = 1, mdx = 1;
    // the shared-memory contraction's share: [0] dw <= kFFSmallW, [1] wider
    int col_n[2] = {0, 0}, col_rows = 32, col_blocks = 1;
    bool others = false;
    long long mtot = 1;
    for (int i = 0; i < n; ++i) {
        const GaussArgs &A = args_host[i];
        const int rows = (A.S + 1) * A.dx;
        if (A.splits < 1 || A.splits > 65535) return cudaErrorInvalidValue;
        md = std::max(md, A.d);
        mdx = std::max(mdx, A.dx);
        mrb = std::max(mrb, (rows + kF64Rows - 1) / kF64Rows);
        msp = std::max(msp, A.splits);
        ms = std::max(ms, A.S + 1);
        mtot = std::max(mtot, (long long)rows * A.dw);
        if (A.perm_t && A.dw <= kGaussFFMaxW && A.N <= kGaussFFColMax) {
            int &cn = col_n[A.dw <= kFFSmallW ? 0 : 1];
            cn = std::max(cn, A.N);
            col_rows = std::max(col_rows, std::min(256, (A.S + 32) & ~31));
        } else {
            others = true;
        }
    }
    for (int i = 0; i < n; ++i)
        col_blocks =
            std::max(col_blocks, (args_host[i].S + col_rows) / col_rows * args_host[i].dx);
    gauss_mean_batch<<<dim3(md, 1, n), 256, 0, st>>>(args_dev);
    gauss_cov_batch<<<dim3(md * (md + 1) / 2, 1, n), 256, 0, st>>>(args_dev);
    gauss_factor_batch<<<dim3(1, 1, n), kFactorThreads, 0, st>>>(args_dev);
    gauss_centre_batch<<<dim3(8, mdx, n), 256, 0, st>>>(args_dev);
    const void *cf[2] = {reinterpret_cast<const void *>(&gauss_cross_col_batch<2>),
                         reinterpret_cast<const void *>(&gauss_cross_col_batch<1>)};
    for (int c = 0; c < 2; ++c) {
        if (!col_n[c]) continue;
        static bool attr_done[2][64] = {};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess && !(dev >= 0 && dev < 64 && attr_done[c][dev])) {
            e = cudaFuncSetAttribute(cf[c], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kGaussFFColMax * 8);
            if (e == cudaSuccess && dev >= 0 && dev < 64) attr_done[c][dev] = true;
        }
        const int parts = c == 0 ? 2 : 1;
        void *ka[] = {&args_dev, &col_rows};
        if (e == cudaSuccess)
            e = cudaLaunchKernel(cf[c], dim3(col_blocks, (msp + parts - 1) / parts, n),
                                 dim3(col_rows * parts), ka, (size_t)col_n[c] * 8, st);
        if (e != cudaSuccess) return e;
    }
    if (others)
        gauss_cross_f64_batch<<<dim3(mrb, msp, n), kF64Rows, 0, st>>>(args_dev);
    gauss_cross_reduce_batch<<<dim3((unsigned)((mtot + 255) / 256), 1, n), 256, 0, st>>>(args_dev);
    gauss_schur_f64_batch<<<dim3((ms + 63) / 64, 1, n), 64, 0, st>>>(args_dev);
    return cudaGetLastError();
}

cudaError_t gauss_launch_turn(const PermTurnJob *jobs_dev, const PermTurnJob *jobs_host, int n,
                              cudaStream_t st)
{
    if (n < 1) return cudaSuccess;
    if (n > 65535) return cudaErrorInvalidValue;
    int mt = 1, ms = 1;
    for (int i = 0; i < n; ++i) {
        if (jobs_host[i].N > 65535 || (jobs_host[i].pitch & 1)) return cudaErrorInvalidValue;
        mt = std::max(mt, (jobs_host[i].N + 63) / 64);
        ms = std::max(ms, (jobs_host[i].pitch + 63) / 64);
    }
    gauss_turn_kernel<<<dim3(mt, ms, n), 256, 0, st>>>(jobs_dev);
    return cudaGetLastError();
}

cudaError_t gauss_launch_keys(const double *v, int n, long long *keys, int *bad, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    gauss_keys_kernel<<<(n + 255) / 256, 256, 0, st>>>(v, n, keys, bad);
    return cudaGetLastError();
}

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// byte offsets of the parts of the buffer (btile first), and their end
struct GaussTcLayout {
    size_t xcen, cen, sum_part, cov_part, inv_w, inv_z, traces, end;
};
static GaussTcLayout gauss_tc_layout(int N, int dx, int dw)
{
    const size_t nchunks = (size_t)(N + kGaussKC - 1) / kGaussKC;
    const size_t passes = (size_t)(dw + kGaussTileN - 1) / kGaussTileN;
    const size_t pitch = ((size_t)N + 31) & ~(size_t)31, d = (size_t)(dx + dw);
    GaussTcLayout o;
    o.xcen = align256(passes * nchunks * 2048 * 4);
    o.cen = align256(o.xcen + (size_t)dx * pitch * 4);
    o.sum_part = align256(o.cen + d * pitch * 8);
    o.cov_part = align256(o.sum_part + d * kGaussParts * 8);
    o.inv_w = align256(o.cov_part + (size_t)kGaussParts * d * d * 8);
    o.inv_z = align256(o.inv_w + (size_t)dw * dw * 8);
    o.traces = align256(o.inv_z + (size_t)dw * dw * 8);
    o.end = align256(o.traces + 8 * 8);
    return o;
}

size_t gauss_tc_workspace(int N, int dx, int dw) { return gauss_tc_layout(N, dx, dw).end; }

void gauss_tc_bind(GaussArgs &A, void *base)
{
    const GaussTcLayout o = gauss_tc_layout(A.N, A.dx, A.dw);
    char *b = (char *)base;
    A.btile = (float *)b;
    A.xcen = (float *)(b + o.xcen);
    A.xcen_pitch = (A.N + 31) & ~31;
    A.cen = (double *)(b + o.cen);
    A.sum_part = (double *)(b + o.sum_part);
    A.cov_part = (double *)(b + o.cov_part);
    A.inv_w = (double *)(b + o.inv_w);
    A.inv_z = (double *)(b + o.inv_z);
    A.traces = (double *)(b + o.traces);
}

cudaError_t gauss_launch_prepare(const GaussArgs &A, cudaStream_t st)
{
    gauss_sum_kernel<<<dim3(A.d, kGaussParts), 128, 0, st>>>(A);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int nchunks = (A.N + kGaussKC - 1) / kGaussKC;
    const int passes = (A.dw + kGaussTileN - 1) / kGaussTileN;
    gauss_prep_kernel<<<dim3(nchunks, passes + 1), 256, 0, st>>>(A, nchunks, passes);
    return cudaGetLastError();
}

cudaError_t gauss_launch_factor(const GaussArgs &A, cudaStream_t st)
{
    const int tw = (A.dw + 3) / 4, tx = (A.dx + 3) / 4;
    gauss_cov_tiles_kernel<<<dim3(tw * (tw + 1) / 2 + tx * (tx + 1) / 2, kGaussParts), 128, 0,
                             st>>>(A);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    gauss_factor_inv_kernel<<<2, kFactorLanes * 40, 0, st>>>(A);
    return cudaGetLastError();
}

int gauss_tc_split_chunks(int N, int rows, int sms, int *group)
{
    const int nchunks = (N + kGaussKC - 1) / kGaussKC;
    const int groups = (nchunks + kGaussGroup - 1) / kGaussGroup;
    *group = (nchunks + groups - 1) / groups;
    // whole accumulation groups, so that no sum depends on the split
    const int tiles = (rows + kGaussTileM - 1) / kGaussTileM;
    const int ctas = std::max(1, 2 * sms / tiles);
    return *group * ((groups + ctas - 1) / ctas);
}

template <bool COLSMEM, int TILES, bool P16>
static cudaError_t gauss_cross_tc(const GaussArgs &A, int rows, int nchunks, cudaStream_t st)
{
    const size_t smem = 1024 + (size_t)4 * (2 * kGaussTileM * kGaussKC + 2 * TILES * 2048 +
                                            (COLSMEM ? A.xcen_pitch : 0));
    const auto f = &gauss_cross_tc_kernel<COLSMEM, TILES, P16>;
    static bool attr_done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && !attr_done[dev]) {
        if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      200 * 1024)) != cudaSuccess)
            return e;
        attr_done[dev] = true;
    }
    f<<<dim3((rows + kGaussTileM - 1) / kGaussTileM, A.splits), 256, smem, st>>>(A, nchunks);
    return cudaGetLastError();
}

cudaError_t gauss_launch_cross_tc(const GaussArgs &A, cudaStream_t st)
{
    const int rows = (A.S + 1) * A.dx;
    const int nchunks = (A.N + kGaussKC - 1) / kGaussKC;
    if (A.splits < 1 || A.splits > 65535 || A.group < 1 || A.group > kGaussGroup ||
        A.chunks_per_split < 1 || A.chunks_per_split % A.group ||
        (long long)(A.splits - 1) * A.chunks_per_split >= nchunks || A.dw > 2 * kGaussTileN ||
        !A.btile || !A.xcen || (A.xcen_pitch & 31) || A.xcen_pitch < A.N ||
        (reinterpret_cast<uintptr_t>(A.btile) & 15) || (reinterpret_cast<uintptr_t>(A.xcen) & 15))
        return cudaErrorInvalidValue;
    if (A.perms16 && (A.perm_pitch < A.N || (A.perm_pitch & 7) ||
                      (reinterpret_cast<uintptr_t>(A.perms16) & 15)))
        return cudaErrorInvalidValue;
    const bool colsmem = A.dx == 1 && A.xcen_pitch <= kGaussColMax, wide = A.dw > kGaussTileN;
    const cudaError_t e =
        !A.perms16 ? (wide ? gauss_cross_tc<false, 2, false>(A, rows, nchunks, st)
                           : gauss_cross_tc<false, 1, false>(A, rows, nchunks, st))
        : colsmem  ? (wide ? gauss_cross_tc<true, 2, true>(A, rows, nchunks, st)
                           : gauss_cross_tc<true, 1, true>(A, rows, nchunks, st))
                   : (wide ? gauss_cross_tc<false, 2, true>(A, rows, nchunks, st)
                           : gauss_cross_tc<false, 1, true>(A, rows, nchunks, st));
    if (e != cudaSuccess) return e;
    const long long total = (long long)rows * A.dw;
    gauss_cross_reduce_kernel<<<(unsigned)((total + 63) / 64), 64, 0, st>>>(A);
    return cudaGetLastError();
}

double gauss_tc_gamma()
{
    // split products: 3 * 2^-22 relative; FP32 rounding of the centred X (one,
    // counted twice);
    // FP32 accumulation of at most 3 * kGaussKC * kGaussGroup products per
    // group, 2^-23 per addition
    return 3.0 * std::ldexp(1.0, -22) + 2.0 * std::ldexp(1.0, -24) +
           3.0 * kGaussKC * kGaussGroup * std::ldexp(1.0, -23);
}

cudaError_t gauss_launch_schur(const GaussArgs &A, double gamma, cudaStream_t st)
{
    const int grid = (A.S + kSchurS) / kSchurS;
    if (A.dx == 1) gauss_schur_kernel<1><<<grid, kSchurThreads, 0, st>>>(A, gamma);
    else gauss_schur_kernel<kGaussMaxX><<<grid, kSchurThreads, 0, st>>>(A, gamma);
    return cudaGetLastError();
}

}  // namespace teksg
