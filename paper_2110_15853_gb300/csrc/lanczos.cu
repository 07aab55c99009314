// Spectral bounds for Algorithm 1 (Sec. 3.4 takes eps_0, eps_ub^w, eps_ub^uw as
// inputs without saying how they are found): k-step Lanczos with full
// re-orthogonalisation on the GPU, then the extreme eigenvalues of the k x k
// tridiagonal T_k by Sturm counts, a warp for each end and 32 points a round.
//
// Every scalar (alpha_j, beta_j, the re-orthogonalisation coefficients, the stop
// flag) stays in device memory, so the k steps queue without host round trips.
// Every reduction uses a fixed partition and a fixed combination order, so the
// result is bitwise reproducible run to run.
#include "common.cuh"
#include "kernels.cuh"

namespace chfsi {

namespace {

// SpMV: rows whose sums a warp adds up together, 4, or 1 where rows have kLongRow entries and
// more on average (a sum's six additions a lane are then few beside its entries, and few
// long rows need all the warps).  20 steps with four rows and with one: 5000 rows of 5000
// entries 4.73 and 2.17 ms, 8000 of 1500 2.09 and 1.69, 64000 of 1500 5.52 and 5.28; but 64000 of
// 600 3.05 and 3.21, 262144 of 655 10.4 and 11.3, 64000 of 300 2.32 and 2.60.
constexpr int kRowsPerWarp = 4;
constexpr int64_t kLongRow = 1024;
inline int rows_per_warp(int64_t N, int64_t nnz) { return nnz >= kLongRow * N ? 1 : kRowsPerWarp; }
inline int64_t spmv_block_count(int64_t N, int rows) { return (N + 8 * rows - 1) / (8 * rows); }
constexpr int kChunk = 512;          // vector kernels: rows per block, two a thread (2048 left 120 SMs
                                     // of 152 idle at N = 64000)
constexpr int kUnroll = 4;           // SpMV: entries in flight per lane
constexpr int kMaxSteps = 64;
constexpr int kGroups = 256;                        // groups of parts
constexpr int64_t kMaxPartReads = (int64_t)1 << 22; // by all blocks of a kernel: 32 MB from L2, about the
                                                    // 5 us of a launch that groups them

// scal layout
enum {
    S_ALPHA = 0,                 // [kMaxSteps]
    S_BETA = kMaxSteps,          // [kMaxSteps]
    S_K = 2 * kMaxSteps,         // number of completed steps (as double)
    S_STOP = S_K + 1,            // 1.0 after breakdown
    S_SCALE = S_STOP + 1,        // running max |alpha_i| + beta_{i-1}
    S_TOTAL = S_SCALE + 1,
};

__device__ __forceinline__ double block_sum(double v, double* red) {
    // fixed-shape tree over the block (blockDim.x = 256)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += red[w];
    return t;   // valid on thread 0
}

// w = H v ; part[b] = sum over the block's rows of v[r] w[r].  A warp takes kRows rows, their
// entries strided over the lanes with kUnroll in flight a lane (the column index, then the
// gather, are dependent reads), and adds up four rows' lane sums together: six
// FP64 additions a lane where row by row took twenty, half of the FP64 pipe's time on rows of
// 300 entries (83 -> 64 us at 19.2 M entries; reading them takes 34).
template <int kRows>
__global__ void __launch_bounds__(256) spmv_dot_kernel(int64_t N, const int64_t* __restrict__ row_ptr,
                                                       const int32_t* __restrict__ col,
                                                       const double* __restrict__ val, int64_t nnz,
                                                       const double* __restrict__ v, double* w, double* part,
                                                       const double* scal, unsigned* status) {
    if (scal[S_STOP] != 0.0) return;
    static_assert(kRows == 4 || kRows == 1, "lane sums of four rows, or of one");
    __shared__ double rowdot[8 * kRows];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r0 = (int64_t)blockIdx.x * (8 * kRows) + warp * kRows;
    int64_t ptr = lane <= kRows && r0 + lane <= N ? row_ptr[r0 + lane] : 0;
    double s[kRows];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < kRows; q++) {
        s[q] = 0.0;
        if (r0 + q >= N) continue;
        int64_t b = __shfl_sync(0xffffffffu, ptr, q), e = __shfl_sync(0xffffffffu, ptr, q + 1);
        if (b < 0) b = 0;
        if (e > nnz) e = nnz;
        for (int64_t p = b + lane; p < e; p += 32 * kUnroll) {
            int32_t c[kUnroll];
            double h[kUnroll], x[kUnroll];
#pragma unroll
            for (int u = 0; u < kUnroll; u++) {
                const bool in = p + 32 * u < e;
                c[u] = in ? col[p + 32 * u] : 0;
                h[u] = in ? val[p + 32 * u] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kUnroll; u++) {
                const bool out = c[u] < 0 || (int64_t)c[u] >= N;
                bad |= out;
                x[u] = out ? 0.0 : v[c[u]];
                if (out) h[u] = 0.0;
            }
#pragma unroll
            for (int u = 0; u < kUnroll; u++)
                if (p + 32 * u < e) s[q] = fma(h[u], x[u], s[q]);
        }
    }
    // lanes 8 q .. 8 q + 7 end with the sum of row q (kRows = 1: all lanes with the row's)
    constexpr int kLanes = 32 / kRows;
    double t;
    if constexpr (kRows == 4) {
        const bool up16 = lane & 16, up8 = lane & 8;
        double t0 = up16 ? s[2] : s[0], t1 = up16 ? s[3] : s[1];
        t0 += __shfl_xor_sync(0xffffffffu, up16 ? s[0] : s[2], 16);
        t1 += __shfl_xor_sync(0xffffffffu, up16 ? s[1] : s[3], 16);
        t = up8 ? t1 : t0;
        t += __shfl_xor_sync(0xffffffffu, up8 ? t0 : t1, 8);
    } else {
        t = s[0];
    }
#pragma unroll
    for (int o = kRows == 4 ? 4 : 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (__any_sync(0xffffffffu, bad) && lane == 0) raise_status(status, DEV_PATTERN);
    const int64_t r = r0 + lane / kLanes;
    if (lane % kLanes == 0) {
        double d = 0.0;
        if (r < N) {
            w[r] = t;
            d = v[r] * t;
        }
        rowdot[warp * kRows + lane / kLanes] = d;
    }
    __syncthreads();
    if (warp == 0) {
        double d = lane < 8 * kRows ? rowdot[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) part[blockIdx.x] = d;
    }
}

// The sum of nparts partial sums, on every thread: each block of the kernels below adds up
// the parts that it needs itself, in the same order as every other (a launch of one block
// for each of the three sums of a step took 6.5 us).  The reads of all blocks grow with N^2,
// so where there are more than kMaxPartReads of them group_parts_kernel adds up kGroups
// groups of parts first: 20 steps at 4.2 M rows of 27 entries took 125 ms without it.
__device__ __forceinline__ double sum_parts(const double* part, int64_t nparts, double* red) {
    __shared__ double total;
    double s = 0.0;
    for (int64_t b = threadIdx.x; b < nparts; b += blockDim.x) s += part[b];
    const double t = block_sum(s, red);
    if (threadIdx.x == 0) total = t;
    __syncthreads();
    return total;
}

// out[g][i] = sum over the parts b of group g of part[b][i], i < ncol (cols: ncol rounded up to
// a power of two), a block per group of consecutive parts, in a fixed order.
__global__ void __launch_bounds__(256) group_parts_kernel(const double* __restrict__ part, int64_t nparts, int ncol,
                                                          int cols, double* __restrict__ out, const double* scal) {
    if (scal && scal[S_STOP] != 0.0) return;
    __shared__ double red[256];
    const int i = threadIdx.x & (cols - 1), sub = threadIdx.x / cols, subs = 256 / cols;
    const int64_t per = (nparts + gridDim.x - 1) / gridDim.x, lo = per * blockIdx.x;
    const int64_t hi = lo + per < nparts ? lo + per : nparts;
    double s = 0.0;
    if (i < ncol)
#pragma unroll 4
        for (int64_t b = lo + sub; b < hi; b += subs) s += part[b * ncol + i];
    red[threadIdx.x] = s;
    for (int o = 128; o >= cols; o >>= 1) {
        __syncthreads();
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    }
    if ((int)threadIdx.x < ncol) out[(int64_t)blockIdx.x * ncol + threadIdx.x] = red[threadIdx.x];
}

// alpha_j from the SpMV's parts; w -= alpha_j v_j + beta_{j-1} v_{j-1}; part[b*(j+1) + i] =
// <V_i, w> over the block's rows
__global__ void __launch_bounds__(256) three_term_dots_kernel(int64_t N, double* w, const double* V, int j,
                                                              const double* aparts, int64_t naparts, double* part,
                                                              double* scal) {
    if (scal[S_STOP] != 0.0) return;
    __shared__ double red[8][kMaxSteps];
    const int64_t r0 = (int64_t)blockIdx.x * kChunk;
    const int64_t r1 = r0 + kChunk < N ? r0 + kChunk : N;
    const double al = sum_parts(aparts, naparts, &red[0][0]);
    if (blockIdx.x == 0 && threadIdx.x == 0) scal[S_ALPHA + j] = al;
    const double bp = j > 0 ? scal[S_BETA + j - 1] : 0.0;
    const double* vj = V + (int64_t)j * N;
    const double* vjm = j > 0 ? V + (int64_t)(j - 1) * N : nullptr;
    constexpr int kRows = kChunk / 256;
    double x[kRows];
#pragma unroll
    for (int u = 0; u < kRows; u++) {
        const int64_t r = r0 + threadIdx.x + 256 * u;
        x[u] = 0.0;
        if (r < r1) {
            x[u] = w[r] - al * vj[r];
            if (vjm) x[u] -= bp * vjm[r];
            w[r] = x[u];
        }
    }
    __syncthreads();   // red is free again
    // four dots at a time; the warps' sums wait in shared memory for one barrier at the end (a
    // block-wide sum per dot took 1.5 us each)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i0 = 0; i0 <= j; i0 += 4) {
        double d[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            d[q] = 0.0;
            if (i0 + q > j) continue;
            const double* vi = V + (int64_t)(i0 + q) * N;
#pragma unroll
            for (int u = 0; u < kRows; u++) {
                const int64_t r = r0 + threadIdx.x + 256 * u;
                if (r < r1) d[q] = fma(vi[r], x[u], d[q]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < 4; q++) d[q] += __shfl_xor_sync(0xffffffffu, d[q], o);
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (lane == 0 && i0 + q <= j) red[warp][i0 + q] = d[q];
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
        double t = 0.0;
        for (int q = 0; q < 8; q++) t += red[q][i];
        part[(int64_t)blockIdx.x * (j + 1) + i] = t;
    }
}

// h_i from the dots' parts (four threads a coefficient); w -= sum_i h_i V_i ; part[b] = |w|^2
// over the block's rows
__global__ void __launch_bounds__(256) reorth_norm_kernel(int64_t N, double* w, const double* V, int j,
                                                          const double* hparts, int64_t nparts, double* part,
                                                          const double* scal) {
    if (scal[S_STOP] != 0.0) return;
    __shared__ double red[8], hs[kMaxSteps];
    static_assert(4 * kMaxSteps <= 256, "four threads a coefficient");
    {
        const int i = threadIdx.x >> 2;
        double h[4] = {0.0, 0.0, 0.0, 0.0};
        if (i <= j) {
            int64_t b = threadIdx.x & 3;
            for (; b + 12 < nparts; b += 16)
#pragma unroll
                for (int q = 0; q < 4; q++) h[q] += hparts[(b + 4 * q) * (j + 1) + i];
            for (; b < nparts; b += 4) h[0] += hparts[b * (j + 1) + i];
        }
        double t = (h[0] + h[1]) + (h[2] + h[3]);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        if ((threadIdx.x & 3) == 0 && i <= j) hs[i] = t;
    }
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * kChunk;
    const int64_t r1 = r0 + kChunk < N ? r0 + kChunk : N;
    double s = 0.0;
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
        double x = w[r];
        int i = 0;
        for (; i + 4 <= j + 1; i += 4) {       // four reads in flight
            double v[4];
#pragma unroll
            for (int q = 0; q < 4; q++) v[q] = V[(int64_t)(i + q) * N + r];
#pragma unroll
            for (int q = 0; q < 4; q++) x -= hs[i + q] * v[q];
        }
        for (; i <= j; i++) x -= hs[i] * V[(int64_t)i * N + r];
        w[r] = x;
        s = fma(x, x, s);
    }
    double t = block_sum(s, red);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// beta_j = |w| from the parts, breakdown test; v_{j+1} = w / beta_j
__global__ void __launch_bounds__(256) scale_next_kernel(int64_t N, const double* w, double* V, int j,
                                                         const double* part, int64_t nparts, double* scal) {
    if (scal[S_STOP] != 0.0) return;
    __shared__ double red[8];
    const double beta = sqrt(sum_parts(part, nparts, red));
    // every block comes to the same scale, whether block 0 has stored it yet or not
    const double cand = fabs(scal[S_ALPHA + j]) + (j > 0 ? scal[S_BETA + j - 1] : 0.0);
    const double scale = fmax(*(const volatile double*)&scal[S_SCALE], cand);
    const bool stop = beta <= 1e-12 * scale;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        scal[S_SCALE] = scale;
        scal[S_K] = (double)(j + 1);
        scal[S_BETA + j] = stop ? 0.0 : beta;
        if (stop) scal[S_STOP] = 1.0;
    }
    if (stop) return;
    const int64_t r0 = (int64_t)blockIdx.x * kChunk;
    const int64_t r1 = r0 + kChunk < N ? r0 + kChunk : N;
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) V[(int64_t)(j + 1) * N + r] = w[r] / beta;
}

// v_0 = v0 / |v0| (norm from part sums, fixed order)
__global__ void __launch_bounds__(256) sq_part_kernel(int64_t N, const double* v, double* part) {
    __shared__ double red[8];
    const int64_t r0 = (int64_t)blockIdx.x * kChunk;
    const int64_t r1 = r0 + kChunk < N ? r0 + kChunk : N;
    double s = 0.0;
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) s = fma(v[r], v[r], s);
    double t = block_sum(s, red);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// A chunk of rows per block; every block sums the parts in the same order.
__global__ void __launch_bounds__(256) norm0_kernel(int64_t N, const double* v0, double* V, const double* part,
                                                    int64_t nparts, double* scal) {
    __shared__ double red[8];
    __shared__ double nrm;
    double s = 0.0;
    for (int64_t b = threadIdx.x; b < nparts; b += blockDim.x) s += part[b];
    double t = block_sum(s, red);
    if (threadIdx.x == 0) {
        nrm = sqrt(t);
        if (blockIdx.x == 0) {
            for (int i = 0; i < S_TOTAL; i++) scal[i] = 0.0;
            if (!(nrm > 0.0) || !isfinite(nrm)) scal[S_STOP] = 2.0;   // unusable start vector
        }
    }
    __syncthreads();
    if (!(nrm > 0.0) || !isfinite(nrm)) return;
    const int64_t r0 = (int64_t)blockIdx.x * kChunk;
    const int64_t r1 = r0 + kChunk < N ? r0 + kChunk : N;
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) V[r] = v0[r] / nrm;
}

// Number of eigenvalues of the symmetric tridiagonal (d, e) that are < x.
__device__ int sturm_count(const double* d, const double* e, int k, double x) {
    int cnt = 0;
    double q = d[0] - x;
    const double tiny = 1e-300;
    if (q == 0.0) q = -tiny;
    if (q < 0.0) cnt++;
    for (int i = 1; i < k; i++) {
        q = (d[i] - x) - e[i - 1] * e[i - 1] / q;
        if (q == 0.0) q = -tiny;
        if (q < 0.0) cnt++;
    }
    return cnt;
}

// The point of (a, b) where the Sturm count reaches `target` (the target-th smallest
// eigenvalue of T_k), by multisection on one warp: each lane counts at one of 32
// equally spaced interior points, and the bracket shrinks to the interval between the
// last point below the target and the first at or above it (a factor 33 per round, where
// bisection gives 2).  Every lane ends with the same bracket.
__device__ double sturm_edge(const double* d, const double* e, int k, double a, double b, int target) {
    const int lane = threadIdx.x & 31;
    for (int it = 0; it < 64; it++) {
        const double h = (b - a) / 33.0;
        const double x = a + h * (double)(lane + 1);
        const bool ge = !(x < b) || sturm_count(d, e, k, x) >= target;
        const unsigned mask = __ballot_sync(0xffffffffu, ge);
        double na, nb;
        if (mask == 0) {
            na = __shfl_sync(0xffffffffu, x, 31);
            nb = b;
        } else {
            const int f = __ffs(mask) - 1;
            nb = __shfl_sync(0xffffffffu, x, f);
            const double xl = __shfl_sync(0xffffffffu, x, f > 0 ? f - 1 : 0);
            na = f > 0 ? xl : a;
        }
        if (!(na > a) && !(nb < b)) break;   // the bracket is at rounding resolution
        a = na > a ? na : a;
        b = nb < b ? nb : b;
    }
    return 0.5 * (a + b);
}

// Smallest and largest eigenvalue of T_k by multisection (one warp each), then the bounds.
__global__ void bounds_kernel(const double* scal, int64_t N, int64_t n_wanted, double* out) {
    __shared__ double theta[2];
    if (scal[S_STOP] == 2.0) {
        if (threadIdx.x == 0) out[0] = out[1] = out[2] = nan("");
        return;
    }
    int k = (int)scal[S_K];
    const double* d = scal + S_ALPHA;
    const double* e = scal + S_BETA;
    double lo = d[0], hi = d[0];
    for (int i = 0; i < k; i++) {
        double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < k ? fabs(e[i]) : 0.0);
        lo = fmin(lo, d[i] - r);
        hi = fmax(hi, d[i] + r);
    }
    double span = hi - lo;
    lo -= 1e-12 * (span + 1.0);
    hi += 1e-12 * (span + 1.0);
    const int end = threadIdx.x >> 5;
    const double edge = sturm_edge(d, e, k, lo, hi, end == 0 ? 1 : k);
    if ((threadIdx.x & 31) == 0) theta[end] = edge;
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double theta_min = theta[0], theta_max = theta[1];
    const double resid = fabs(e[k - 1]);
    const double a0 = theta_min;
    const double bb = theta_max + resid;
    const double aa = a0 + (bb - a0) * pow((double)n_wanted / (double)N, 2.0 / 3.0);
    out[0] = aa;
    out[1] = bb;
    out[2] = a0;
}

}  // namespace

// Two sets of parts, the SpMV's (or the norms') and the dots', and one of groups.
static size_t lanczos_first_parts(int64_t N) {
    const int64_t spmv_blocks = spmv_block_count(N, 1), chunks = (N + kChunk - 1) / kChunk;
    return (size_t)((spmv_blocks > chunks ? spmv_blocks : chunks) + 1);
}

size_t lanczos_part_count(int64_t N, int steps) {
    const int64_t chunks = (N + kChunk - 1) / kChunk;
    return lanczos_first_parts(N) + (size_t)(chunks * (steps + 1)) + (size_t)kGroups * kMaxSteps;
}

// Partial sums for a kernel of `blocks` blocks that each read all of them: `count` x ncol
// at p, added up in groups first where those reads are too many.
struct Parts {
    const double* p;
    int64_t count;
};
static int group_parts(Parts& q, int ncol, int64_t blocks, double* groups, const double* scal, cudaStream_t s) {
    if (blocks * q.count * ncol <= kMaxPartReads) return CHFSI_OK;
    int cols = 1;
    while (cols < ncol) cols *= 2;
    group_parts_kernel<<<kGroups, 256, 0, s>>>(q.p, q.count, ncol, cols, groups, scal);
    CHFSI_LAUNCH_CHECK();
    q = Parts{groups, kGroups};
    return CHFSI_OK;
}

int lanczos_run(const CsrDev& h, int steps, const double* v0, int64_t n_wanted, double* V, double* w,
                double* part, double* scal, double* dev_out, unsigned* status, cudaStream_t s) {
    const int64_t N = h.N;
    int k = steps < N ? steps : (int)N;
    if (k < 1 || k > kMaxSteps) return CHFSI_ERR_ARG;
    const double* val = static_cast<const double*>(h.val);
    const int64_t chunks = (N + kChunk - 1) / kChunk;
    const int rows = rows_per_warp(N, h.nnz);
    const int64_t spmv_blocks = spmv_block_count(N, rows);
    auto spmv = rows == 1 ? spmv_dot_kernel<1> : spmv_dot_kernel<kRowsPerWarp>;

    double* part2 = part + lanczos_first_parts(N);
    double* groups = part2 + chunks * (steps + 1);

    sq_part_kernel<<<(unsigned)chunks, 256, 0, s>>>(N, v0, part);
    CHFSI_LAUNCH_CHECK();
    int rc;
    Parts q{part, chunks};
    if ((rc = group_parts(q, 1, chunks, groups, nullptr, s))) return rc;
    norm0_kernel<<<(unsigned)chunks, 256, 0, s>>>(N, v0, V, q.p, q.count, scal);
    CHFSI_LAUNCH_CHECK();
    for (int j = 0; j < k; j++) {
        const double* vj = V + (int64_t)j * N;
        spmv<<<(unsigned)spmv_blocks, 256, 0, s>>>(N, h.row_ptr, h.col, val, h.nnz, vj, w, part, scal, status);
        CHFSI_LAUNCH_CHECK();
        q = Parts{part, spmv_blocks};
        if ((rc = group_parts(q, 1, chunks, groups, scal, s))) return rc;
        three_term_dots_kernel<<<(unsigned)chunks, 256, 0, s>>>(N, w, V, j, q.p, q.count, part2, scal);
        CHFSI_LAUNCH_CHECK();
        q = Parts{part2, chunks};
        if ((rc = group_parts(q, j + 1, chunks, groups, scal, s))) return rc;
        reorth_norm_kernel<<<(unsigned)chunks, 256, 0, s>>>(N, w, V, j, q.p, q.count, part, scal);
        CHFSI_LAUNCH_CHECK();
        q = Parts{part, chunks};
        if ((rc = group_parts(q, 1, chunks, groups, scal, s))) return rc;
        scale_next_kernel<<<(unsigned)chunks, 256, 0, s>>>(N, w, V, j, q.p, q.count, scal);
        CHFSI_LAUNCH_CHECK();
    }
    bounds_kernel<<<1, 64, 0, s>>>(scal, N, n_wanted, dev_out);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

}  // namespace chfsi
