// Dense FP64 kernels of the ChFSI closure (Algorithm 1 steps 2-5, Sec. 3.4):
// Gram / projection products A^T B with a deterministic split-K reduction over
// the long dimension N, the product with an n x n matrix (X_F = Y R^-1,
// Psi = X_F Q), a blocked right-looking Cholesky S = R^T R, the inverse of the
// upper-triangular factor, and small element-wise helpers.
//
// FP64 on this part runs on the DFMA pipe (about 1.2 TFLOP/s for the whole GPU, two
// multiply-adds a cycle and SM), so the tiles are sized for DFMA issue, not for bandwidth:
// 64 x 64 output tiles, 256 threads, 4 x 4 outputs per thread with stride-16 row/column
// ownership so that shared-memory reads are conflict-free and global stores coalesce --
// or 16 x 16 tiles, one output per thread, where 64 x 64 tiles leave SMs idle.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace chfsi {

namespace {

constexpr int BK = 16;   // reduction chunk

struct GemmArgs {
    const double* A; int64_t lda; bool a_t;   // a_t: A stored K x M, element (i,k) = A[k*lda+i]
    const double* B; int64_t ldb;             // B stored K x Nc, element (k,j) = B[k*ldb+j]
    double* C; int64_t ldc;
    int64_t M, Nc, K;
    double alpha;
    bool accumulate;                          // C = C + alpha*AB (else C = alpha*AB)
    bool upper_tiles;                         // only tiles with tile_row <= tile_col
    bool b_upper;                             // B upper triangular: k <= j
    int splits;
    double* part;                             // splits x M x Nc partials, or nullptr
    bool a_upper = false;                     // A upper triangular: k >= i
    // nbatch > 1: independent products (splits = 1), operands `stride` elements apart; batch b
    // has min(Nc, Ntot - b Nstep) columns, and as many k where k_is_nc
    int nbatch = 1;
    int64_t strideA = 0, strideB = 0, strideC = 0, Ntot = 0, Nstep = 0;
    bool k_is_nc = false;
    // merge products of the eigensolver: K = Nc = lda = ldb = ldc = the count at kn[b kn_stride],
    // min(M, Ntot - b M) rows
    const double* kn = nullptr;
    int kn_stride = 0;
};

// TB x TB output tile, TB / 16 squared outputs per thread.
template <int TB>
__global__ void __launch_bounds__(256) gemm_kernel(GemmArgs g) {
    constexpr int T = TB / 16;
    __shared__ double As[BK][TB + 1];
    __shared__ double Bs[BK][TB];
    const int bi = blockIdx.y, bj = blockIdx.x, z = g.nbatch > 1 ? 0 : blockIdx.z;
    if (g.nbatch > 1 || g.kn) {
        const int64_t b = blockIdx.z, cols = g.Ntot - b * g.Nstep;
        g.A += b * g.strideA;
        g.B += b * g.strideB;
        g.C += b * g.strideC;
        if (g.kn) {
            if (g.Ntot - b * g.M < g.M) g.M = g.Ntot - b * g.M;
            g.K = g.Nc = g.lda = g.ldb = g.ldc = (int64_t)g.kn[b * g.kn_stride];
            if ((int64_t)bj * TB >= g.Nc || (int64_t)bi * TB >= g.M) return;
        } else {
            if (cols < g.Nc) g.Nc = cols;
            if (g.k_is_nc) g.K = g.Nc;
        }
    }
    if (g.upper_tiles && bi > bj) return;
    const int64_t i0 = (int64_t)bi * TB, j0 = (int64_t)bj * TB;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;

    int64_t kc = (g.K + g.splits - 1) / g.splits;
    kc = (kc + BK - 1) / BK * BK;
    int64_t k_begin = (int64_t)z * kc;
    int64_t k_end = k_begin + kc < g.K ? k_begin + kc : g.K;
    if (g.b_upper) {
        int64_t lim = j0 + TB;
        if (k_end > lim) k_end = lim;
    }
    if (g.a_upper && k_begin < i0) k_begin = i0;

    double acc[T][T];
#pragma unroll
    for (int a = 0; a < T; a++)
#pragma unroll
        for (int b = 0; b < T; b++) acc[a][b] = 0.0;

    for (int64_t k0 = k_begin; k0 < k_end; k0 += BK) {
        // stage A chunk as As[k][i] and B chunk as Bs[k][j]
        for (int e = threadIdx.x; e < BK * TB; e += 256) {
            int kk, ii;
            double va = 0.0;
            if (g.a_t) {
                kk = e / TB; ii = e % TB;                     // coalesced along i
                int64_t k = k0 + kk, i = i0 + ii;
                if (k < k_end && i < g.M) va = g.A[k * g.lda + i];
            } else {
                ii = e / BK; kk = e % BK;                     // coalesced along k
                int64_t k = k0 + kk, i = i0 + ii;
                if (k < k_end && i < g.M) va = g.A[i * g.lda + k];
            }
            As[kk][ii] = va;
            int kb = e / TB, jb = e % TB;
            int64_t k = k0 + kb, j = j0 + jb;
            Bs[kb][jb] = (k < k_end && j < g.Nc) ? g.B[k * g.ldb + j] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; kk++) {
            double av[T], bv[T];
#pragma unroll
            for (int a = 0; a < T; a++) av[a] = As[kk][ty + 16 * a];
#pragma unroll
            for (int b = 0; b < T; b++) bv[b] = Bs[kk][tx + 16 * b];
#pragma unroll
            for (int a = 0; a < T; a++)
#pragma unroll
                for (int b = 0; b < T; b++) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
        }
        __syncthreads();
    }

#pragma unroll
    for (int a = 0; a < T; a++) {
        int64_t i = i0 + ty + 16 * a;
        if (i >= g.M) continue;
#pragma unroll
        for (int b = 0; b < T; b++) {
            int64_t j = j0 + tx + 16 * b;
            if (j >= g.Nc) continue;
            if (g.part) {
                g.part[((int64_t)z * g.M + i) * g.Nc + j] = g.alpha * acc[a][b];
            } else {
                double v = g.alpha * acc[a][b];
                if (g.accumulate) v += g.C[i * g.ldc + j];
                g.C[i * g.ldc + j] = v;
            }
        }
    }
}

// C[i][j] = sum_z part[z][i][j] in split order; with `mirror`, tb x tb tiles below the
// diagonal take the transposed upper-tile sum.
__global__ void reduce_parts_kernel(const double* __restrict__ part, int splits, int64_t M, int64_t Nc,
                                    double* C, int64_t ldc, bool mirror, int tb) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= M * Nc) return;
    int64_t i = idx / Nc, j = idx % Nc;
    int64_t si = i, sj = j;
    if (mirror && (i / tb) > (j / tb)) { si = j; sj = i; }
    double s = 0.0;
    for (int z = 0; z < splits; z++) s += part[((int64_t)z * M + si) * Nc + sj];
    C[i * ldc + j] = s;
}

// Tile edge: 64, or 16 where fewer than four 64 x 64 tiles per SM would run.  A tile's time is
// its multiply-adds at two a cycle (a 64 x 64 x 64 product takes one SM 68 us), so small
// products need many small tiles; at two multiply-adds a cycle the 16 x 16 tile's
// operands are no load on shared memory or L2.  Measured: the products of a 96-state
// closure over 8000 rows 8.48 -> 0.71 ms together; with four and more tiles per SM the
// 64 x 64 tiles, at 97% of the DFMA pipe, stay.
int gemm_tile(int64_t M, int64_t Nc, int64_t batches, bool upper) {
    int64_t tm = (M + 63) / 64, tn = (Nc + 63) / 64, tiles = tm * tn;
    if (upper) tiles = tm * (tm + 1) / 2;
    return tiles * batches < 4 * sm_count_or_default() ? 16 : 64;
}

int run_gemm(const GemmArgs& g, cudaStream_t s) {
    if (g.M <= 0 || g.Nc <= 0) return CHFSI_OK;
    const int64_t z = g.nbatch > 1 ? g.nbatch : g.splits;
    const int tb = gemm_tile(g.M, g.Nc, z, g.upper_tiles);
    dim3 grid((unsigned)((g.Nc + tb - 1) / tb), (unsigned)((g.M + tb - 1) / tb), (unsigned)z);
    if (tb == 64) gemm_kernel<64><<<grid, 256, 0, s>>>(g);
    else gemm_kernel<16><<<grid, 256, 0, s>>>(g);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

// ---------------------------------------------------------------- Cholesky

constexpr int NB = 64;    // columns between trailing updates
constexpr int ND = 32;    // diagonal block

// q = v / d from the reciprocal r of d, with one correction (Markstein): three FP64
// operations in place of the division's dozen on a pipe that takes 64 cycles a warp.
__device__ __forceinline__ double div_by(double v, double d, double r) {
    const double q = v * r;
    return fma(fma(-q, d, v), r, q);
}

// Upper Cholesky of the nb x nb diagonal block at S[k0][k0] (nb <= 32, in place): four warps,
// lane = column, warp w the rows i = w mod 4 in registers (one warp per FP64 unit of the
// SM).  A step's chain is the root and reciprocal of the pivot, the scaled row and one
// update; 64 columns in one block of 256 threads with three barriers a step took 105 us,
// two 32-column blocks take 28 us each.
__global__ void __launch_bounds__(128) chol_diag_kernel(double* S, int64_t lds, int64_t k0, int nb,
                                                        unsigned* status) {
    __shared__ double row[2][ND];
    const int w = threadIdx.x >> 5, j = threadIdx.x & 31;
    double a[ND / 4];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < ND / 4; q++) {
        const int i = 4 * q + w;
        a[q] = (i < nb && j < nb && i <= j) ? S[(k0 + i) * lds + k0 + j] : (i == j ? 1.0 : 0.0);
    }
#pragma unroll
    for (int k = 0; k < ND; k++) {
        if (w == (k & 3)) row[k & 1][j] = a[k / 4];
        __syncthreads();
        double p = row[k & 1][k];
        if (!(p > 0.0) || !isfinite(p)) { bad = true; p = 1.0; }
        // root and reciprocal from one reciprocal square root and a correction each: a shorter
        // chain than sqrt and a division (a block 37 -> 28 us)
        const double r = rsqrt(p), d0 = p * r, d = fma(fma(-d0, d0, p), 0.5 * r, d0);
        const double x = j == k ? d : div_by(row[k & 1][j], d, r);   // R[k][j], j >= k
        if (w == (k & 3)) a[k / 4] = j >= k ? x : 0.0;
#pragma unroll
        for (int q = 0; q < ND / 4; q++) {
            if (4 * q + 3 <= k) continue;
            const int i = 4 * q + w;
            const double xi = __shfl_sync(0xffffffffu, x, i);
            if (i > k && j >= i) a[q] = fma(-xi, x, a[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < ND / 4; q++) {
        const int i = 4 * q + w;
        if (i < nb && j < nb) S[(k0 + i) * lds + k0 + j] = j >= i ? a[q] : 0.0;
    }
    if (threadIdx.x == 0 && bad) raise_status(status, DEV_CHOL);
}

// Panel: R[k0:k0+nb, j] = R_kk^-T S[k0:k0+nb, j] for j >= k0+nb (forward substitution), 16
// columns per block so that the multiply-adds spread over the SMs; row i of the solution,
// then its update of the rows below, one barrier a step.  (A thread per column with its 64
// entries in local memory took 182 us a panel; two 32-row panels take 13 us each.)
constexpr int kPanelCols = 16;

__global__ void __launch_bounds__(256) chol_panel_kernel(double* S, int64_t lds, int64_t n, int64_t k0, int nb) {
    __shared__ double R[ND][ND + 1];
    __shared__ double z[ND][kPanelCols];
    __shared__ double rinv[ND];
    for (int e = threadIdx.x; e < nb * nb; e += 256) R[e / nb][e % nb] = S[(k0 + e / nb) * lds + k0 + e % nb];
    const int c = threadIdx.x % kPanelCols, r = threadIdx.x / kPanelCols;
    const int64_t j = k0 + nb + (int64_t)blockIdx.x * kPanelCols + c;
    double v[2];
#pragma unroll
    for (int h = 0; h < 2; h++) v[h] = (j < n && r + 16 * h < nb) ? S[(k0 + r + 16 * h) * lds + j] : 0.0;
    __syncthreads();
    if (threadIdx.x < nb) rinv[threadIdx.x] = 1.0 / R[threadIdx.x][threadIdx.x];
    __syncthreads();
    for (int i = 0; i < nb; i++) {
        if (r == (i & 15)) z[i][c] = div_by(i < 16 ? v[0] : v[1], R[i][i], rinv[i]);
        __syncthreads();
        const double zi = z[i][c];
#pragma unroll
        for (int h = 0; h < 2; h++)
            if (r + 16 * h > i && r + 16 * h < nb) v[h] = fma(-R[i][r + 16 * h], zi, v[h]);
    }
    if (j < n) {
#pragma unroll
        for (int h = 0; h < 2; h++)
            if (r + 16 * h < nb) S[(k0 + r + 16 * h) * lds + j] = z[r + 16 * h][c];
    }
}

__global__ void zero_lower_kernel(double* S, int64_t lds, int64_t n) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * n) return;
    int64_t i = idx / n, j = idx % n;
    if (j < i) S[i * lds + j] = 0.0;
}

// ---------------------------------------------------------------- triangular inverse

constexpr int kTriLeaf = 64;

// Inverse of the 64 x 64 diagonal blocks of an upper-triangular R (block b at row and column
// 64 b), one block per CTA: from the last row up, row i of X is the scaled row of the
// identity minus the updates received from the rows below, then row i updates the rows
// above; one barrier a row.  A thread holds one column's rows r = 4 q + w (w = threadIdx.x /
// 64).  Entries below the diagonal are written as zeros.
__global__ void __launch_bounds__(256) tri_inv_leaf_kernel(const double* __restrict__ R, int64_t ldr, double* X,
                                                           int64_t ldx, int64_t n) {
    __shared__ double Rs[kTriLeaf][kTriLeaf + 1];
    __shared__ double xi[2][kTriLeaf];
    const int64_t b0 = (int64_t)blockIdx.x * kTriLeaf;
    const int nb = (int)(n - b0 < kTriLeaf ? n - b0 : kTriLeaf);
    for (int e = threadIdx.x; e < kTriLeaf * kTriLeaf; e += 256) {
        const int i = e / kTriLeaf, j = e % kTriLeaf;
        Rs[i][j] = (i < nb && j < nb && j >= i) ? R[(b0 + i) * ldr + b0 + j] : (i == j ? 1.0 : 0.0);
    }
    __syncthreads();
    const int j = threadIdx.x & 63, w = threadIdx.x >> 6;
    double x[kTriLeaf / 4];
#pragma unroll
    for (int q = 0; q < kTriLeaf / 4; q++) x[q] = 4 * q + w == j ? 1.0 : 0.0;
    if (threadIdx.x < kTriLeaf) Rs[threadIdx.x][kTriLeaf] = 1.0 / Rs[threadIdx.x][threadIdx.x];
    __syncthreads();
#pragma unroll
    for (int i = kTriLeaf - 1; i >= 0; i--) {
        if (w == (i & 3)) {
            x[i / 4] = div_by(x[i / 4], Rs[i][i], Rs[i][kTriLeaf]);
            xi[i & 1][j] = x[i / 4];
        }
        __syncthreads();
        const double v = xi[i & 1][j];
#pragma unroll
        for (int q = 0; q < kTriLeaf / 4; q++) {
            if (4 * q >= i) continue;
            const int l = 4 * q + w;
            if (l < i && j >= i) x[q] = fma(-Rs[l][i], v, x[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < kTriLeaf / 4; q++) {
        const int i = 4 * q + w;
        if (i < nb && j < nb) X[(b0 + i) * ldx + b0 + j] = j >= i ? x[q] : 0.0;
    }
}

__global__ void transpose_kernel(const double* __restrict__ A, int64_t lda, double* B, int64_t ldb, int64_t n) {
    __shared__ double t[32][33];
    int64_t bx = (int64_t)blockIdx.x * 32, by = (int64_t)blockIdx.y * 32;
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        int64_t i = by + k, j = bx + threadIdx.x;
        if (i < n && j < n) t[k][threadIdx.x] = A[i * lda + j];
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        int64_t i = bx + k, j = by + threadIdx.x;
        if (i < n && j < n) B[i * ldb + j] = t[threadIdx.x][k];
    }
}

__global__ void symmetrize_kernel(double* S, int64_t lds, int64_t n) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * n) return;
    int64_t i = idx / n, j = idx % n;
    if (j <= i) return;
    double v = 0.5 * (S[i * lds + j] + S[j * lds + i]);
    S[i * lds + j] = v;
    S[j * lds + i] = v;
}

// ---------------------------------------------------------------- conversions

template <typename TS, typename TD>
__global__ void convert_kernel(const TS* __restrict__ src, int64_t lds, TD* dst, int64_t ldd, int64_t rows,
                               int64_t n, int64_t width) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * width) return;
    const int64_t i = idx / width, j = idx % width;
    float fv;
    double dv;
    if (j < n) {
        if constexpr (std::is_same<TS, __nv_bfloat16>::value) { fv = __bfloat162float(src[i * lds + j]); dv = fv; }
        else { dv = (double)src[i * lds + j]; fv = (float)src[i * lds + j]; }
    } else {
        dv = 0.0; fv = 0.0f;
    }
    if constexpr (std::is_same<TD, double>::value) dst[i * ldd + j] = dv;
    else if constexpr (std::is_same<TD, float>::value) dst[i * ldd + j] = fv;
    else dst[i * ldd + j] = __float2bfloat16_rn(fv);
}

template <typename TS, typename TD>
int launch_convert(const void* src, int64_t lds, void* dst, int64_t ldd, int64_t rows, int64_t n, int64_t width,
                   cudaStream_t s) {
    int64_t total = rows * width;
    if (total <= 0) return CHFSI_OK;
    convert_kernel<TS, TD><<<(unsigned)((total + 255) / 256), 256, 0, s>>>(
        static_cast<const TS*>(src), lds, static_cast<TD*>(dst), ldd, rows, n, width);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

__global__ void convert_values_kernel(const double* __restrict__ src, float* dst, int64_t count, bool bf) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    float f = (float)src[i];
    if (bf) f = __bfloat162float(__float2bfloat16_rn(f));
    dst[i] = f;
}

}  // namespace

int gemm_tn_splits(int64_t K, int64_t n) {
    const int64_t sms = sm_count_or_default();
    int64_t tiles = ((n + 63) / 64);
    tiles = tiles * (tiles + 1) / 2;
    int64_t want = (4 * sms + tiles - 1) / tiles;        // about four 64 x 64 tiles per SM
    int64_t maxs = (K + 2047) / 2048;                    // keep >= 2048 rows per split
    int64_t s = want < maxs ? want : maxs;
    // fewer tiles than that: 16 x 16 tiles (run_gemm), enough splits for a dozen of them per
    // SM while each keeps 256 rows
    if (tiles * s < 4 * sms) {
        const int64_t t = (n + 15) / 16, more = (12 * sms + t * (t + 1) / 2 - 1) / (t * (t + 1) / 2);
        const int64_t most = (K + 255) / 256, want16 = more < most ? more : most;
        if (want16 > s) s = want16;
        if (tiles * s >= 4 * sms) s = (4 * sms - 1) / tiles;
    }
    if (s < 1) s = 1;
    if (s > 64) s = 64;
    return (int)s;
}

int gemm_tn(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t K, int64_t n, double* S,
            int64_t lds, bool symmetric, double* part, int splits, cudaStream_t s) {
    if (n <= 0) return CHFSI_OK;
    GemmArgs g{A, lda, true, B, ldb, S, lds, n, n, K, 1.0, false, symmetric, false, splits, part};
    int rc = run_gemm(g, s);
    if (rc) return rc;
    int64_t total = n * n;
    reduce_parts_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(part, splits, n, n, S, lds, symmetric,
                                                                        gemm_tile(n, n, splits, symmetric));
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

int gemm_nn(const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc, int64_t M,
            int64_t n, bool b_upper, cudaStream_t s) {
    GemmArgs g{A, lda, false, B, ldb, C, ldc, M, n, n, 1.0, false, false, b_upper, 1, nullptr};
    return run_gemm(g, s);
}

int gemm_merges(const double* G, const double* U, double* Gn, int64_t k, int64_t n, int nm, const double* kn,
                int kn_stride, cudaStream_t s) {
    GemmArgs g{G, k, false, U, k, Gn, k, k < n ? k : n, k < n ? k : n, k, 1.0, false, false, false, 1, nullptr};
    g.M = k;
    g.nbatch = nm;
    g.Ntot = n;
    g.strideA = g.strideB = g.strideC = k * k;
    g.kn = kn;
    g.kn_stride = kn_stride;
    const int tb = gemm_tile(g.Nc, g.Nc, nm, false);
    const dim3 grid((unsigned)((g.Nc + tb - 1) / tb), (unsigned)((g.Nc + tb - 1) / tb), (unsigned)nm);
    if (tb == 64) gemm_kernel<64><<<grid, 256, 0, s>>>(g);
    else gemm_kernel<16><<<grid, 256, 0, s>>>(g);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

int gemm_general(const double* A, int64_t lda, bool a_t, const double* B, int64_t ldb, double* C, int64_t ldc,
                 int64_t M, int64_t Nc, int64_t K, double alpha, bool accumulate, cudaStream_t s) {
    if (M <= 0 || Nc <= 0) return CHFSI_OK;
    GemmArgs g{A, lda, a_t, B, ldb, C, ldc, M, Nc, K, alpha, accumulate, false, false, 1, nullptr};
    return run_gemm(g, s);
}

namespace {

constexpr int64_t kCholOzakiMin = 256;   // trailing blocks from this size on as Ozaki products

}  // namespace

int cholesky_upper(double* S, int64_t n, int64_t lds, unsigned* status, cudaStream_t s, void* oz_ws,
                   size_t oz_bytes) {
    int rc;
    for (int64_t k0 = 0; k0 < n; k0 += NB) {
        const int nb = (int)((n - k0) < NB ? (n - k0) : NB);
        // the nb rows in blocks of 32: diagonal block, its panel, and the update of the second
        // block's rows
        for (int64_t k = k0; k < k0 + nb; k += ND) {
            const int nd = (int)(k0 + nb - k < ND ? k0 + nb - k : ND);
            chol_diag_kernel<<<1, 128, 0, s>>>(S, lds, k, nd, status);
            CHFSI_LAUNCH_CHECK();
            const int64_t right = n - k - nd;
            if (right <= 0) break;
            chol_panel_kernel<<<(unsigned)((right + kPanelCols - 1) / kPanelCols), 256, 0, s>>>(S, lds, n, k, nd);
            CHFSI_LAUNCH_CHECK();
            if (k + nd < k0 + nb) {
                const double* Rk = S + k * lds + (k + nd);
                const int64_t below = k0 + nb - k - nd;
                GemmArgs g{Rk, lds, true, Rk, lds, S + (k + nd) * lds + (k + nd), lds, below, right, nd, -1.0, true,
                           false, false, 1, nullptr};
                if ((rc = run_gemm(g, s))) return rc;
            }
        }
        int64_t rest = n - k0 - nb;
        if (rest <= 0) break;
        // trailing update S22 -= R12^T R12: an Ozaki product on the tensor cores when its
        // workspace is given, else FP64 on the DFMA pipe (upper tiles)
        const double* R12 = S + k0 * lds + (k0 + nb);
        double* S22 = S + (k0 + nb) * lds + (k0 + nb);
        if (oz_ws && rest >= kCholOzakiMin &&
            oz_bytes >= ozaki_workspace_bytes(true, rest, rest, nb, true)) {
            if ((rc = ozaki_gemm_tn(R12, lds, R12, lds, nb, rest, rest, S22, lds, true, oz_ws, oz_bytes, status, s,
                                    true)))
                return rc;
            continue;
        }
        GemmArgs g{R12, lds, true, R12, lds, S22, lds, rest, rest, nb, -1.0, true, true, false, 1, nullptr};
        if ((rc = run_gemm(g, s))) return rc;
    }
    int64_t total = n * n;
    zero_lower_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(S, lds, n);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

namespace {

__global__ void negate_block_kernel(double* X, int64_t ldx, int64_t rows, int64_t cols) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * cols) return;
    X[(idx / cols) * ldx + idx % cols] = -X[(idx / cols) * ldx + idx % cols];
}

constexpr int64_t kTriInvOzaki = 256;   // halves of this size and more as Ozaki products

}  // namespace

// R^-1 of an upper-triangular R: the 64 x 64 diagonal blocks in one launch, then pairs of
// blocks of h = 64, 128, ... rows: with [R11 R12; 0 R22] the off-diagonal block of the inverse
// is -X11 R12 X22 (T = R12 X22 into `tmp`, then X11 T) -- all pairs of a size in one
// FP64 launch a product, or from 256 rows on as Ozaki products on the tensor cores when
// oz_ws is given and the depth fits (<= 8192).  (Column by column, a warp each, blocks of up
// to 1024 columns took 1.4 ms; the diagonal blocks now take 56 us and an FP64 product 8 - 20.)
int tri_inverse_upper_blocked(const double* R, int64_t ldr, double* X, int64_t ldx, int64_t n, double* tmp,
                              int64_t ldt, void* oz_ws, size_t oz_bytes, unsigned* status, cudaStream_t s) {
    if (n <= 0) return CHFSI_OK;
    int rc;
    CHFSI_CUDA_TRY(cudaMemset2DAsync(X, sizeof(double) * (size_t)ldx, 0, sizeof(double) * (size_t)n, (size_t)n, s));
    tri_inv_leaf_kernel<<<(unsigned)((n + kTriLeaf - 1) / kTriLeaf), 256, 0, s>>>(R, ldr, X, ldx, n);
    CHFSI_LAUNCH_CHECK();
    for (int64_t h = kTriLeaf; h < n; h *= 2) {
        const int64_t pairs = (n - h + 2 * h - 1) / (2 * h);     // blocks at 2 h b with rows right of the first h
        if (oz_ws && h >= kTriInvOzaki && h <= 8192 && oz_bytes >= ozaki_workspace_bytes(false, h, h, h, false)) {
            for (int64_t b = 0; b < pairs; b++) {
                const int64_t o = 2 * h * b, r = std::min(h, n - o - h);
                const double* R12 = R + o * ldr + o + h;
                const double* X22 = X + (o + h) * ldx + o + h;
                double* X12 = X + o * ldx + o + h;
                if ((rc = ozaki_gemm_nn(R12, ldr, X22, ldx, h, r, r, tmp, ldt, true, oz_ws, oz_bytes, status, s)))
                    return rc;
                if ((rc = ozaki_gemm_nn(X + o * ldx + o, ldx, tmp, ldt, h, h, r, X12, ldx, false, oz_ws, oz_bytes,
                                        status, s)))
                    return rc;
                negate_block_kernel<<<(unsigned)((h * r + 255) / 256), 256, 0, s>>>(X12, ldx, h, r);
                CHFSI_LAUNCH_CHECK();
            }
            continue;
        }
        GemmArgs g{R + h, ldr, false, X + h * ldx + h, ldx, tmp, ldt, h, h, h, 1.0, false, false, true, 1, nullptr};
        g.nbatch = (int)pairs;
        g.Ntot = n - h;
        g.Nstep = 2 * h;
        g.k_is_nc = true;
        g.strideA = 2 * h * (ldr + 1);
        g.strideB = 2 * h * (ldx + 1);
        g.strideC = 2 * h * ldt;
        if (pairs == 1) { g.Nc = g.K = std::min(h, n - h); }
        if ((rc = run_gemm(g, s))) return rc;
        GemmArgs f{X, ldx, false, tmp, ldt, X + h, ldx, h, h, h, -1.0, false, false, false, 1, nullptr};
        f.a_upper = true;
        f.nbatch = (int)pairs;
        f.Ntot = n - h;
        f.Nstep = 2 * h;
        f.strideA = 2 * h * (ldx + 1);
        f.strideB = 2 * h * ldt;
        f.strideC = 2 * h * (ldx + 1);
        if (pairs == 1) f.Nc = std::min(h, n - h);
        if ((rc = run_gemm(f, s))) return rc;
    }
    return CHFSI_OK;
}

int transpose(const double* A, int64_t lda, double* B, int64_t ldb, int64_t n, cudaStream_t s) {
    if (n <= 0) return CHFSI_OK;
    dim3 grid((unsigned)((n + 31) / 32), (unsigned)((n + 31) / 32));
    transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(A, lda, B, ldb, n);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

int symmetrize(double* S, int64_t n, int64_t lds, cudaStream_t s) {
    int64_t total = n * n;
    if (total <= 0) return CHFSI_OK;
    symmetrize_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(S, lds, n);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

int convert_block(const void* src, Buf st, int64_t lds, void* dst, Buf dt, int64_t ldd, int64_t rows, int64_t n,
                  int64_t width, cudaStream_t s) {
    if (width < n || width > ldd) return CHFSI_ERR_ARG;
    if (st == Buf::F64 && dt == Buf::F32) return launch_convert<double, float>(src, lds, dst, ldd, rows, n, width, s);
    if (st == Buf::F64 && dt == Buf::BF16)
        return launch_convert<double, __nv_bfloat16>(src, lds, dst, ldd, rows, n, width, s);
    if (st == Buf::F32 && dt == Buf::F64) return launch_convert<float, double>(src, lds, dst, ldd, rows, n, width, s);
    if (st == Buf::F32 && dt == Buf::BF16)
        return launch_convert<float, __nv_bfloat16>(src, lds, dst, ldd, rows, n, width, s);
    if (st == Buf::F64 && dt == Buf::F64) return launch_convert<double, double>(src, lds, dst, ldd, rows, n, width, s);
    if (st == Buf::F32 && dt == Buf::F32) return launch_convert<float, float>(src, lds, dst, ldd, rows, n, width, s);
    return CHFSI_ERR_UNSUPPORTED;
}

int convert_values(const double* src, void* dst, Buf dt, int64_t count, bool round_bf16, cudaStream_t s) {
    if (dt != Buf::F32) return CHFSI_ERR_UNSUPPORTED;
    if (count <= 0) return CHFSI_OK;
    convert_values_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(src, static_cast<float*>(dst), count,
                                                                          round_bf16);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

int fill_zero(void* p, size_t bytes, cudaStream_t s) {
    if (!bytes) return CHFSI_OK;
    CHFSI_CUDA_TRY(cudaMemsetAsync(p, 0, bytes, s));
    return CHFSI_OK;
}

}  // namespace chfsi
