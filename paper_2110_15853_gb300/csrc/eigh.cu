// Dense symmetric eigensolver of the Rayleigh-Ritz step (Algorithm 1 step 4, Sec. 3.4:
// H_F Q = Q Lambda), FP64, written for the GPU:
//   1. Householder tridiagonalisation  A = Q_H T Q_H^T, one reflector per column
//      (reflector of row j, symmetric matrix-vector product with the trailing block,
//      symmetric rank-2 update);
//   2. divide and conquer on T (Cuppen's splitting T = diag(T1, T2) + rho u u^T), the merges
//      of a level together: leaves of 32 rows by parallel-ordered Jacobi in shared memory; each merge
//      deflates (small components of z, nearly equal poles rotated together), finds
//      the roots of the secular equation 1 + rho sum z_j^2 / (d_j - lambda) (one warp
//      per root, bracketed steps of a two-pole rational model from the nearer pole), recomputes z
//      from the roots (the
//      Gu-Eisenstat formula, so that the eigenvectors come out orthogonal), and
//      multiplies the subproblem vectors by the eigenvectors of D + rho z z^T;
//   3. back-transformation Q = Q_H Q_T in panels of 64 reflectors (compact WY form
//      I - V T V^T, three matrix products per panel).
// Everything runs in this library's kernels, FP64 on the DFMA pipe or, for the products from
// 256 rows on, FP64-accurate Ozaki products on the tensor cores; the host orders the
// launches and reads the merges' sizes.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"

namespace chfsi {

namespace {

constexpr double kEps = 2.220446049250313e-16;
constexpr int kLeaf = 32;
constexpr int kPanel = 64;
constexpr int kSecularSmem = 6144;   // poles and weights staged in shared memory up to this size

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the block (blockDim.x a multiple of 32, at most 1024); every thread gets it.
__device__ double block_sum(double v) {
    __shared__ double part[32];
    __shared__ double total;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) part[w] = v;
    __syncthreads();
    if (w == 0) {
        double t = lane < (int)(blockDim.x >> 5) ? part[lane] : 0.0;
        t = warp_sum(t);
        if (lane == 0) total = t;
    }
    __syncthreads();
    return total;
}

// ------------------------------------------------------------------ 0. scale

// The largest exponent field of A's entries (zeroed before) and, where the largest entry is not
// within 2^-64 .. 2^64, the power of two that takes it into [1/2, 1).  Products and squares
// of the rows of the matrix that the solver works on then neither overflow nor vanish for
// any finite A, and kNegligible below is a fixed number.  An entry that is not finite is
// reported here.
__global__ void __launch_bounds__(256) matrix_exponent_kernel(const double* __restrict__ A, int64_t lda, int64_t n,
                                                              int* emax, unsigned* status) {
    int m = 0;
    for (int64_t r = blockIdx.x; r < n; r += gridDim.x)
        for (int64_t c = threadIdx.x; c < n; c += blockDim.x) {
            const int e = (__double2hiint(A[r * lda + c]) >> 20) & 0x7ff;
            m = e > m ? e : m;
        }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) {
        if (m) atomicMax(emax, m);
        if (m == 0x7ff) raise_status(status, DEV_NONFINITE);
    }
}

// e of the scale 2^-e (0 also where A is zero, subnormal throughout or not finite).
__device__ __forceinline__ int scale_exponent(const int* emax) {
    const int m = *emax, e = m - 1022;
    return m == 0 || m == 0x7ff || (e >= -64 && e <= 64) ? 0 : e;
}

// A *= 2^-e (exact unless the result is subnormal).
__global__ void __launch_bounds__(256) scale_matrix_kernel(double* A, int64_t lda, int64_t n, const int* emax) {
    const int e = scale_exponent(emax);
    if (e == 0) return;
    const double f = scalbn(1.0, -e);      // 2^-1024 (subnormal) .. 2^1021
    for (int64_t r = blockIdx.x; r < n; r += gridDim.x)
        for (int64_t c = threadIdx.x; c < n; c += blockDim.x) A[r * lda + c] *= f;
}

// w *= 2^e.
__global__ void unscale_kernel(double* w, int64_t n, const int* emax) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int e = scale_exponent(emax);
    if (i < n && e != 0) w[i] = scalbn(w[i], e);
}

// ------------------------------------------------------------------ 1. tridiagonalisation

// A panel reduces kPanel32 columns j0 .. j0 + 31 against the trailing matrix as it stood at
// the panel's start (A0); the reflectors v_t and the vectors w_t of the panel's columns
// are kept as rows of PV = [V; W; V] (length n each), so that the matrix current at column
// j is A0 - sum_t (v_t w_t^T + w_t v_t^T).  One cooperative launch does a whole panel; after
// it the trailing matrix takes A -= V^T W + W^T V in one product of depth 2 * 32.
//
// With x = A[j][j+1:] (row j up to date), H = I - tau v v^T maps x to beta e_1, v = scale (x -
// beta e_1) (v_0 = 1).  A column takes two passes with a grid barrier after each:
//   1. every block reads x into shared memory; a warp per row forms A0 x (one FMA an entry;
//      A0 v = scale (A0 x - beta A0 e_1)) and, as further rows, the dots V_t . x and
//      W_t . x; the blocks' shares of x . A0 x go to part.  beta, tau and scale come
//      from x itself, in every block alike.
//   2. with those sums p . v = tau (v . A0 v - 2 sum_t (V_t . v)(W_t . v)) is known before p is, so
//      each block forms p, w = p - (tau / 2)(p . v) v and row j + 1 of the current matrix for
//      its own columns at once.
// A row, a product and a p kernel per column with a reduction at the end of each took 31 us a
// column at n = 2400 (27 of them latency: launch, dependent L2 reads, the last block's sum),
// and an unblocked pair of kernels 23 us at n = 640; this takes 18 and 12 us.
constexpr int kPanel32 = 32;   // columns per panel of the tridiagonalisation
constexpr int kTriThreads = 256, kTriWarps = kTriThreads / 32;
constexpr int kTriCols = 16;   // columns of pass 2 per block and turn
constexpr int kTriUnroll = 8;  // loads in flight per lane in pass 1
constexpr int64_t kTriStaged = 20000;   // x in shared memory up to this n

// Barrier counter of the panel kernels (it counts on from launch to launch) and the flag of
// a barrier that gave up, after which later panels do nothing.
struct TriScalars {
    unsigned count, gave_up;
    int emax;                    // largest exponent field of A
};

// A rest of x below 1e-140 (A's largest entry is 2^-64 and more) is left out: with the squares of
// scale = 1 / (x_0 - beta) below, a smaller one would overflow.
constexpr double kNegligible = 1e-280;

__device__ __forceinline__ void reflector(double x0, double sumsq, double& beta, double& t, double& scale) {
    if (sumsq <= kNegligible) {
        beta = x0;
        t = 0.0;
        scale = 0.0;
    } else {
        const double nrm = sqrt(x0 * x0 + sumsq);
        beta = x0 >= 0.0 ? -nrm : nrm;
        t = (beta - x0) / beta;
        scale = 1.0 / (x0 - beta);
    }
}

struct TriPanel {
    double* A;
    int64_t lda, n, j0;
    int nc;                      // columns of the panel
    bool staged;                 // x fits shared memory
    double *PV, *part, *ybuf, *dots, *d, *e, *tau;
    TriScalars* tri;
    int* vwmax;                  // largest exponent fields of the panel's V and of its W (zeroed before)
    unsigned base;               // count at the start of this launch
    uint64_t wait_ns;            // limit of a barrier's wait
    unsigned* status;
};

// Arrive at grid barrier number `b` of this launch; wait for it (bounded: the launch is
// cooperative, so every block is resident, but a wait that gives up is flagged, not endless).
// After it the panels to come do nothing, d, e and tau keep the zeros that they start with
// where no panel got to, and the call ends with the status.  The clock is read every 1024
// polls, or at each one for limits below a millisecond.
__device__ __forceinline__ void grid_arrive(const TriPanel& a) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&a.tri->count, 1u);
    }
}
__device__ __forceinline__ bool grid_wait(const TriPanel& a, unsigned b) {
    __shared__ int ok;
    if (threadIdx.x == 0) {
        const unsigned target = a.base + (b + 1) * gridDim.x;
        const volatile unsigned* c = &a.tri->count;
        const unsigned mask = a.wait_ns < 1000000ull ? 0u : 1023u;
        uint64_t t0 = 0;
        ok = 1;
        for (unsigned polls = 1; (int)(*c - target) < 0; polls++) {
            if ((polls & mask) == 0) {
                uint64_t t;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t0 == 0) t0 = t;
                else if (t - t0 > a.wait_ns) {
                    a.tri->gave_up = 1;
                    raise_status(a.status, DEV_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

__global__ void __launch_bounds__(kTriThreads) tri_panel_kernel(const __grid_constant__ TriPanel a) {
    extern __shared__ __align__(16) double xs_raw[];
    __shared__ double c1s[kPanel32], c2s[kPanel32], vj[kPanel32], wj[kPanel32];
    __shared__ double red[2][kTriWarps][kTriCols];
    __shared__ double wpart[kTriWarps], tot[3];
    if (*(const volatile unsigned*)&a.tri->gave_up) return;
    const int64_t n = a.n, lda = a.lda;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)blockIdx.x * kTriWarps + warp, nw = (int64_t)gridDim.x * kTriWarps;
    const bool pair_ok = a.staged && (lda % 2) == 0 && (reinterpret_cast<uintptr_t>(a.A) & 15u) == 0;
    unsigned bar = 0;
    int vmax = 0, wmax = 0;      // of this thread's entries beyond the panel and its first column
    for (int i = 0; i < a.nc; i++) {
        const int64_t j = a.j0 + i, m = n - j - 1;
        double* xg = a.A + j * lda + j + 1;
        const int head = (reinterpret_cast<uintptr_t>(xg) & 15u) ? 1 : 0;   // entries before a 16-byte boundary
        double* xs = xs_raw + head;                                          // aligned like xg
        auto x_at = [&](int64_t q) { return a.staged ? xs[q] : __ldcg(xg + q); };
        if (a.staged)
            for (int64_t q = threadIdx.x; q < m; q += kTriThreads) xs[q] = __ldcg(xg + q);
        const double* next = a.A + (j + 1) * lda;            // row j + 1 of A0
        const double a00 = next[j + 1];
        if ((int)threadIdx.x < i) {
            vj[threadIdx.x] = __ldcg(a.PV + (int64_t)threadIdx.x * n + j + 1);
            wj[threadIdx.x] = __ldcg(a.PV + (int64_t)(kPanel32 + threadIdx.x) * n + j + 1);
        }
        __syncthreads();
        // ---- pass 1: the dots of W_t (t < i) and V_t with x, then the rows of A0
        double xy = 0.0;
        for (int64_t r = gw; r < m + 2 * i; r += nw) {
            const int64_t row = r - 2 * i;
            double acc[kTriUnroll];
#pragma unroll
            for (int q = 0; q < kTriUnroll; q++) acc[q] = 0.0;
            if (row < 0) {
                const double* pv = a.PV + (r < i ? kPanel32 + r : r - i) * n + j + 1;
                int64_t q = lane;
                for (; q + 32 * 3 < m; q += 32 * 4) {
                    double v[4];
#pragma unroll
                    for (int k = 0; k < 4; k++) v[k] = __ldcg(pv + q + 32 * k);
#pragma unroll
                    for (int k = 0; k < 4; k++) acc[k] = fma(v[k], x_at(q + 32 * k), acc[k]);
                }
                for (; q < m; q += 32) acc[0] = fma(__ldcg(pv + q), x_at(q), acc[0]);
            } else {
                const double* ar = a.A + (j + 1 + row) * lda + j + 1;
                if (pair_ok) {
                    const int64_t m2 = (m - head) / 2;
                    const double2* a2 = reinterpret_cast<const double2*>(ar + head);
                    const double2* x2 = reinterpret_cast<const double2*>(xs + head);
                    if (head && lane == 0) acc[0] = ar[0] * xs[0];
                    int64_t q = lane;
                    for (; q + 32 * (kTriUnroll - 1) < m2; q += 32 * kTriUnroll) {
                        double2 v[kTriUnroll];
#pragma unroll
                        for (int k = 0; k < kTriUnroll; k++) v[k] = a2[q + 32 * k];
#pragma unroll
                        for (int k = 0; k < kTriUnroll; k++) {
                            const double2 xv = x2[q + 32 * k];
                            acc[k] = fma(v[k].x, xv.x, acc[k]);
                            acc[k] = fma(v[k].y, xv.y, acc[k]);
                        }
                    }
                    double2 v[kTriUnroll];
#pragma unroll
                    for (int k = 0; k < kTriUnroll; k++)
                        v[k] = q + 32 * k < m2 ? a2[q + 32 * k] : make_double2(0.0, 0.0);
#pragma unroll
                    for (int k = 0; k < kTriUnroll; k++)
                        if (q + 32 * k < m2) {
                            const double2 xv = x2[q + 32 * k];
                            acc[k] = fma(v[k].x, xv.x, acc[k]);
                            acc[k] = fma(v[k].y, xv.y, acc[k]);
                        }
                    if (((m - head) & 1) && lane == 0) acc[1] = fma(ar[m - 1], xs[m - 1], acc[1]);
                } else {
                    int64_t q = lane;
                    for (; q + 32 * 3 < m; q += 32 * 4)
#pragma unroll
                        for (int k = 0; k < 4; k++) acc[k] = fma(ar[q + 32 * k], x_at(q + 32 * k), acc[k]);
                    for (; q < m; q += 32) acc[0] = fma(ar[q], x_at(q), acc[0]);
                }
            }
#pragma unroll
            for (int w = kTriUnroll / 2; w > 0; w /= 2)
#pragma unroll
                for (int q = 0; q < w; q++) acc[q] += acc[q + w];
            const double sum = warp_sum(acc[0]);
            if (lane == 0) {
                if (row < 0) {
                    a.dots[r] = sum;
                } else {
                    a.ybuf[row] = sum;
                    xy = fma(x_at(row), sum, xy);
                }
            }
        }
        if (lane == 0) wpart[warp] = xy;
        __syncthreads();
        if (warp == 0) {
            double v = lane < kTriWarps ? wpart[lane] : 0.0;
#pragma unroll
            for (int o = kTriWarps / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) a.part[blockIdx.x] = v;
        }
        // the reflector, in every block alike: while the others finish when x is staged (in A's
        // row j it is overwritten once all have arrived)
        if (a.staged) grid_arrive(a);
        double sq = 0.0;
        for (int64_t q = 1 + threadIdx.x; q < m; q += kTriThreads) sq = fma(x_at(q), x_at(q), sq);
        sq = block_sum(sq);
        double beta, t, scale;
        reflector(x_at(0), sq, beta, t, scale);
        if (!a.staged) grid_arrive(a);
        // this thread's entries of V, W and row j + 1 for pass 2, ready since the last column
        const int cl = threadIdx.x % kTriCols, g = threadIdx.x / kTriCols;
        const int64_t cfirst = j + 1 + (int64_t)blockIdx.x * kTriCols + cl;
        double vt[2], wt[2], an = 0.0;
        auto load_vw = [&](int64_t c) {
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int q = g + 16 * u;
                vt[u] = c < n && q < i ? __ldcg(a.PV + (int64_t)q * n + c) : 0.0;
                wt[u] = c < n && q < i ? __ldcg(a.PV + (int64_t)(kPanel32 + q) * n + c) : 0.0;
            }
            if (threadIdx.x < kTriCols && c < n) an = next[c];
        };
        load_vw(cfirst);
        if (!grid_wait(a, bar++)) return;
        // ---- pass 2
        const double yx0 = __ldcg(a.ybuf);
        double yc = threadIdx.x < kTriCols && cfirst < n ? __ldcg(a.ybuf + (cfirst - j - 1)) : 0.0;
        if (warp == 0) {
            double v = 0.0;
            for (unsigned b = lane; b < gridDim.x; b += 32) v += __ldcg(a.part + b);
            v = warp_sum(v);
            if (lane == 0) tot[0] = v;
        } else if (warp <= 2) {
            double c1 = 0.0, c2 = 0.0, v0 = 0.0, w0 = 0.0;
            if (lane < i) {
                v0 = vj[lane];
                w0 = wj[lane];
                c1 = scale == 0.0 ? w0 : scale * fma(-beta, w0, __ldcg(a.dots + lane));        // W_t . v
                c2 = scale == 0.0 ? v0 : scale * fma(-beta, v0, __ldcg(a.dots + i + lane));    // V_t . v
            }
            if (warp == 1) {
                c1s[lane] = c1;
                c2s[lane] = c2;
            }
            const double sum = warp_sum(warp == 1 ? c1 * c2 : fma(v0, c1, w0 * c2));
            if (lane == 0) tot[warp] = sum;
        }
        __syncthreads();
        const double y0 = scale == 0.0 ? a00 : scale * fma(-beta, a00, yx0);                   // (A0 v)_0
        const double vav = scale == 0.0 ? a00
                                        : scale * scale * fma(beta, fma(beta, a00, -2.0 * yx0), tot[0]);
        const double kw = 0.5 * t * t * (vav - 2.0 * tot[1]);                                  // (tau / 2) p . v
        const double wnext = t * (y0 - tot[2]) - kw;                                           // w at index j + 1
        double* Vi = a.PV + (int64_t)i * n;
        double* Wi = a.PV + (int64_t)(kPanel32 + i) * n;
        double* Vc = a.PV + (int64_t)(2 * kPanel32 + i) * n;
        for (int64_t c0 = j + 1 + (int64_t)blockIdx.x * kTriCols; c0 < n; c0 += (int64_t)gridDim.x * kTriCols) {
            const int64_t c = c0 + cl;
            double s1 = 0.0, s2 = 0.0;
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int q = g + 16 * u;
                if (q < i) {
                    s1 = fma(vt[u], c1s[q], fma(wt[u], c2s[q], s1));
                    s2 = fma(vj[q], wt[u], fma(wj[q], vt[u], s2));
                }
            }
            s1 += __shfl_xor_sync(0xffffffffu, s1, 16);
            s2 += __shfl_xor_sync(0xffffffffu, s2, 16);
            if (lane < kTriCols) {
                red[0][warp][cl] = s1;
                red[1][warp][cl] = s2;
            }
            __syncthreads();
            if (threadIdx.x < 32) {       // lanes 0-15 sum the first kind, 16-31 the second
                const double* rp = &red[lane >> 4][0][cl];
                double u[4];
#pragma unroll
                for (int k = 0; k < 4; k++) u[k] = rp[k * kTriCols] + rp[(k + 4) * kTriCols];
                const double sum = (u[0] + u[2]) + (u[1] + u[3]);
                const double sum2 = __shfl_xor_sync(0xffffffffu, sum, 16);
                if (lane < kTriCols && c < n) {
                    const double y = scale == 0.0 ? an : scale * fma(-beta, an, yc);
                    const double v = c == j + 1 ? 1.0 : x_at(c - j - 1) * scale;
                    const double w = fma(-kw, v, t * (y - sum));
                    Vi[c] = v;
                    Wi[c] = w;
                    Vc[c] = v;
                    if (i + 1 < a.nc) a.A[(j + 1) * lda + c] = an - sum2 - fma(wnext, v, w);
                    a.A[j * lda + c] = v;    // kept for the back-transformation
                    if (c > a.j0 + a.nc) {
                        vmax = max(vmax, (__double2hiint(v) >> 20) & 0x7ff);
                        wmax = max(wmax, (__double2hiint(w) >> 20) & 0x7ff);
                    }
                }
            }
            __syncthreads();
            const int64_t cn = c + (int64_t)gridDim.x * kTriCols;      // a further turn
            if (cn - cl < n) {
                load_vw(cn);
                if (threadIdx.x < kTriCols && cn < n) yc = __ldcg(a.ybuf + (cn - j - 1));
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.d[j] = __ldcg(a.A + j * lda + j);
            a.e[j] = beta;
            a.tau[j] = t;
        }
        if (i + 1 < a.nc) {
            grid_arrive(a);
            if (!grid_wait(a, bar++)) return;
        }
    }
    if (warp == 0) {
        vmax = __reduce_max_sync(0xffffffffu, vmax);
        wmax = __reduce_max_sync(0xffffffffu, wmax);
        if (lane == 0 && vmax) atomicMax(a.vwmax, vmax);
        if (lane == 0 && wmax) atomicMax(a.vwmax + 1, wmax);
    }
}

// V *= 2^h, W *= 2^-h in the columns of the trailing matrix, before an Ozaki product, where their
// largest magnitudes are 2^4 and more apart: V W stays as it is, and both come to the same
// size.  A row of the product's operands holds entries of V and of W under one
// power-of-two scale, so that the smaller kind loses as many of the 56 bits as W (of
// A's spread) and V (of 1's) differ by.  Three of them leave it at the accuracy of FP64 updates;
// 1500 x 1500 ones with a random part of 1e-3 left residuals of 9e-14 |A| (FP64 1e-14, with
// this pass 7e-15).  2 - 3 us a panel.
constexpr int kBalanceRows = 8;
__global__ void __launch_bounds__(256) panel_balance_kernel(double* PV, int64_t n, int64_t jn, const int* vwmax) {
    const int apart = vwmax[0] && vwmax[1] ? vwmax[1] - vwmax[0] : 0, h = apart / 2;
    const int64_t c = jn + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (abs(apart) < 4 || c >= n) return;
    const int t0 = blockIdx.y * kBalanceRows;           // rows V, W, V
    const double f = scalbn(1.0, t0 / kPanel32 == 1 ? -h : h);
    double x[kBalanceRows];
#pragma unroll
    for (int t = 0; t < kBalanceRows; t++) x[t] = PV[(t0 + t) * n + c];
#pragma unroll
    for (int t = 0; t < kBalanceRows; t++) PV[(t0 + t) * n + c] = x[t] * f;
}

// The last 2 x 2 (or 1 x 1) block of T.
__global__ void tridiag_tail_kernel(const double* A, int64_t lda, int64_t n, double* d, double* e, double* tau) {
    if (threadIdx.x != 0) return;
    if (n >= 2) {
        d[n - 2] = A[(n - 2) * lda + n - 2];
        e[n - 2] = A[(n - 2) * lda + n - 1];
        tau[n - 2] = 0.0;
    }
    d[n - 1] = A[(n - 1) * lda + n - 1];
}

// ------------------------------------------------------------------ 2. divide and conquer

// Cuppen's splitting at every leaf boundary m: d[m-1] and d[m] lose rho = e[m-1];
// the original off-diagonal is kept in ebak.
__global__ void dc_split_kernel(int64_t n, double* d, const double* e, double* ebak) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n - 1) ebak[i] = e[i];
    const int64_t m = (i + 1) * kLeaf;   // boundary number i
    if (m < n) {
        const double rho = e[m - 1];
        d[m - 1] -= rho;
        d[m] -= rho;
    }
}

// Key of the order in which eigenvalues are ranked: that of the reals, -0 with 0, and every
// NaN last, so that the ranks (ties by index) are a permutation whatever the values.
// Integer instructions, off the FP64 pipe.
__device__ __forceinline__ long long order_key(double x) {
    const long long b = __double_as_longlong(x), mag = b & 0x7fffffffffffffffll;
    if (mag > 0x7ff0000000000000ll) return 0x7fffffffffffffffll;
    return b < 0 ? -mag : mag;
}

// Leaf eigenproblems by parallel (round-robin ordered) Jacobi; one block per leaf.
// Writes ascending eigenvalues to w[l ..] and the eigenvectors into the diagonal block
// Q[l.., l..] (the rest of Q is zero).
__global__ void __launch_bounds__(256) dc_leaf_kernel(int64_t n, const double* d, const double* e, double* w,
                                                      double* Q, int64_t ldq) {
    __shared__ double A[kLeaf][kLeaf + 1];
    __shared__ double V[kLeaf][kLeaf + 1];
    __shared__ double rc[kLeaf / 2], rs[kLeaf / 2];
    __shared__ int rp[kLeaf / 2], rq[kLeaf / 2];
    __shared__ int rank[kLeaf];
    const int64_t l = (int64_t)blockIdx.x * kLeaf;
    const int s = (int)((n - l) < kLeaf ? (n - l) : kLeaf);
    for (int idx = threadIdx.x; idx < kLeaf * kLeaf; idx += blockDim.x) {
        const int i = idx / kLeaf, j = idx % kLeaf;
        double v = 0.0;
        if (i < s && j < s) {
            if (i == j) v = d[l + i];
            else if (j == i + 1) v = e[l + i];
            else if (i == j + 1) v = e[l + j];
        }
        A[i][j] = v;
        V[i][j] = i == j ? 1.0 : 0.0;
    }
    __syncthreads();
    for (int sweep = 0; sweep < 20; sweep++) {
        double o = 0.0, t2 = 0.0;
        for (int idx = threadIdx.x; idx < kLeaf * kLeaf; idx += blockDim.x) {
            const int i = idx / kLeaf, j = idx % kLeaf;
            const double a2 = A[i][j] * A[i][j];
            t2 += a2;
            if (i != j) o += a2;
        }
        o = block_sum(o);
        t2 = block_sum(t2);
        if (o <= 1e-30 * t2 || o == 0.0) break;   // off-diagonal below about 1e-15 |A|
        for (int round = 0; round < kLeaf - 1; round++) {
            // pairs of this round: players 0 .. kLeaf-1, player 0 fixed, the others rotating
            if (threadIdx.x < kLeaf / 2) {
                const int k = threadIdx.x;
                auto player = [&](int pos) { return pos == 0 ? 0 : ((pos - 1 + round) % (kLeaf - 1)) + 1; };
                int p = player(k), q = player(kLeaf - 1 - k);
                if (p > q) { const int t = p; p = q; q = t; }
                const double apq = A[p][q];
                double c = 1.0, sn = 0.0;
                // an entry below 1e-19 |A| is left (the sweeps end at 1e-15 |A| over all of them)
                if (apq != 0.0 && fabs(apq) > 1e-300 && apq * apq > 1e-38 * t2) {
                    const double theta = (A[q][q] - A[p][p]) / (2.0 * apq);
                    const double t = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                    c = rsqrt(t * t + 1.0);
                    sn = t * c;
                }
                rp[k] = p; rq[k] = q; rc[k] = c; rs[k] = sn;
            }
            __syncthreads();
            // rows p, q of A (rotations of one round touch disjoint rows)
            for (int idx = threadIdx.x; idx < (kLeaf / 2) * kLeaf; idx += blockDim.x) {
                const int k = idx / kLeaf, col = idx % kLeaf;
                const int p = rp[k], q = rq[k];
                const double c = rc[k], sn = rs[k];
                if (sn == 0.0) continue;                 // uniform in the warp
                const double ap = A[p][col], aq = A[q][col];
                A[p][col] = c * ap - sn * aq;
                A[q][col] = sn * ap + c * aq;
            }
            __syncthreads();
            // columns p, q of A and of V
            for (int idx = threadIdx.x; idx < (kLeaf / 2) * kLeaf; idx += blockDim.x) {
                const int k = idx / kLeaf, row = idx % kLeaf;
                const int p = rp[k], q = rq[k];
                const double c = rc[k], sn = rs[k];
                if (sn == 0.0) continue;
                const double ap = A[row][p], aq = A[row][q];
                A[row][p] = c * ap - sn * aq;
                A[row][q] = sn * ap + c * aq;
                const double vp = V[row][p], vq = V[row][q];
                V[row][p] = c * vp - sn * vq;
                V[row][q] = sn * vp + c * vq;
            }
            __syncthreads();
        }
    }
    // ascending order of the s real eigenvalues (the padding rows never mix with them)
    if (threadIdx.x < s) {
        const int i = threadIdx.x;
        const long long li = order_key(A[i][i]);
        int r = 0;
        for (int j = 0; j < s; j++) {
            const long long lj = order_key(A[j][j]);
            r += (lj < li) || (lj == li && j < i);
        }
        rank[i] = r;
    }
    __syncthreads();
    if (threadIdx.x < s) w[l + rank[threadIdx.x]] = A[threadIdx.x][threadIdx.x];
    for (int idx = threadIdx.x; idx < s * s; idx += blockDim.x) {
        const int r = idx / s, i = idx % s;
        Q[(l + r) * ldq + l + rank[i]] = V[r][i];
    }
}

// Per-merge scratch (device arrays of n, or of n x n for the matrices).
struct MergeBufs {
    double *D, *z, *Dnd, *znd, *tau_r, *zhat, *norm, *val, *rot_c, *rot_s, *par;
    int *perm, *defl, *ndidx, *pos, *org, *rot_a, *rot_b, *rank;
    double *G, *U, *Gn;
};

// The merges of a level run together: merge b = blockIdx.z joins the blocks [l, m) and [m, r) of
// half = kLeaf 2^level rows (the last block may be shorter), l = 2 half b.  Every launch of a
// level takes all of them; one merge at a time, the launches of 74 merges at n = 2400
// mostly waited for one block or one warp per root.
struct Merge {
    int64_t l, m, r, k;
};
__device__ __forceinline__ Merge merge_at(int64_t half, int64_t n, MergeBufs& b) {
    const int64_t i = blockIdx.z;
    Merge g;
    g.l = 2 * half * i;
    g.m = g.l + half;
    g.r = g.l + 2 * half < n ? g.l + 2 * half : n;
    g.k = g.r - g.l;
    b.D += g.l; b.z += g.l; b.Dnd += g.l; b.znd += g.l; b.tau_r += g.l; b.zhat += g.l; b.norm += g.l; b.val += g.l;
    b.rot_c += g.l; b.rot_s += g.l;
    b.perm += g.l; b.defl += g.l; b.ndidx += g.l; b.pos += g.l; b.org += g.l; b.rot_a += g.l; b.rot_b += g.l;
    b.rank += g.l;
    b.par += 8 * i;
    const int64_t mat = i * (2 * half) * (2 * half);   // at most n^2 - k^2: 2 half <= l for i > 0
    b.G += mat; b.U += mat; b.Gn += mat;
    return g;
}

// par[] = {rho_hat, sign, k_nd, nrot}.
// Merge preparation: z from the boundary rows, signs, the sorted poles, deflation with
// the Givens rotations of nearly equal poles.  One block per merge.  Each pole finds its
// place in the merged order by a binary search in the other half; the poles that stay are
// numbered by a block-wide count.  Only when two neighbouring ones are close enough for a
// rotation does one thread walk through them (the walk alone took 115 us a merge).
// The places are a permutation, and perm a list of valid columns, only because both halves
// are sorted numbers.  Where a pole, a weight or rho is not finite, or a half is not sorted
// (after input that was not finite or a panel that gave up), the poles keep their
// own order, all deflated, and the status word says so: nothing indexes with what
// the workspace happened to hold.
__global__ void __launch_bounds__(1024) dc_merge_prep_kernel(int64_t half, int64_t n, const double* w,
                                                             const double* Q, int64_t ldq, const double* ebak,
                                                             MergeBufs b, unsigned* status) {
    __shared__ int wcount[32], total;
    __shared__ double wmax[32];
    const Merge g = merge_at(half, n, b);
    const int64_t l = g.l, m = g.m;
    const int n1 = (int)(m - l), k = (int)g.k, n2 = k - n1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double rho0 = ebak[m - 1];
    const double sg = rho0 >= 0.0 ? 1.0 : -1.0;
    double zz = 0.0, dmax = 0.0;
    bool bad = !isfinite(rho0);
    for (int p = threadIdx.x; p < k; p += blockDim.x) {
        const double zp = p < n1 ? Q[(m - 1) * ldq + l + p] : Q[m * ldq + m + (p - n1)];
        const double d = sg * w[l + p];
        bad |= !isfinite(zp) || !isfinite(d) || (p != 0 && p != n1 && !(w[l + p - 1] <= w[l + p]));
        b.z[p] = zp;
        b.D[p] = d;
        dmax = fmax(dmax, fabs(d));
        zz += zp * zp;
    }
    zz = block_sum(zz);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (lane == 0) wmax[warp] = dmax;
    __syncthreads();
    dmax = wmax[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    const double rho_hat = fabs(rho0) * zz;
    if (__syncthreads_or(bad)) {
        for (int p = threadIdx.x; p < k; p += blockDim.x) {
            b.perm[p] = p;
            b.val[p] = b.D[p];
            b.defl[p] = 1;
            b.pos[p] = -1;
        }
        if (threadIdx.x == 0) {
            b.par[0] = rho_hat;
            b.par[1] = sg;
            b.par[2] = 0.0;
            b.par[3] = 0.0;
            raise_status(status, DEV_NONFINITE);
        }
        return;
    }
    const double zs = 1.0 / sqrt(zz > 0.0 ? zz : 1.0);
    // merged order of the two sorted halves (ascending when sg > 0, descending otherwise):
    // entry t of a half goes behind the entries of the other half that come before it (those
    // of the first half also when equal)
    auto at1 = [&](int t) { return sg > 0.0 ? t : n1 - 1 - t; };
    auto at2 = [&](int t) { return sg > 0.0 ? n1 + t : k - 1 - t; };
    for (int p = threadIdx.x; p < k; p += blockDim.x) {
        const bool first = p < n1;
        const int t = first ? p : p - n1, q = first ? at1(t) : at2(t);
        const double d = b.D[q];
        int lo = 0, hi = first ? n2 : n1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const double o = first ? b.D[at2(mid)] : b.D[at1(mid)];
            if (first ? o < d : o <= d) lo = mid + 1;
            else hi = mid;
        }
        b.perm[t + lo] = q;
        b.val[t + lo] = d;                 // sorted poles (modified by the rotations below)
        b.tau_r[t + lo] = b.z[q] * zs;     // sorted, normalised z (temporarily)
    }
    __syncthreads();
    const double tol = 8.0 * kEps * fmax(dmax, rho_hat);
    // small components of z, and the numbers of the others
    auto number = [&](bool small) {
        int kn = 0;
        for (int p0 = 0; p0 < k; p0 += blockDim.x) {
            const int p = p0 + threadIdx.x;
            bool stay = false;
            if (p < k) {
                if (small) b.defl[p] = fabs(rho_hat * b.tau_r[p]) <= tol;
                stay = !b.defl[p];
            }
            const unsigned bits = __ballot_sync(0xffffffffu, stay);
            if (lane == 0) wcount[warp] = __popc(bits);
            __syncthreads();
            int before = 0, sum = 0;
            for (int q = 0; q < (int)(blockDim.x >> 5); q++) {
                before += q < warp ? wcount[q] : 0;
                sum += wcount[q];
            }
            const int c = kn + before + __popc(bits & ((1u << lane) - 1));
            if (p < k) b.pos[p] = stay ? c : -1;
            if (stay) b.ndidx[c] = p;
            kn += sum;
            __syncthreads();
        }
        return kn;
    };
    int kn = number(true);
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    for (int c = threadIdx.x; c + 1 < kn; c += blockDim.x)
        if (fabs(b.val[b.ndidx[c + 1]] - b.val[b.ndidx[c]]) <= tol) total = 1;
    __syncthreads();
    int nrot = 0;
    if (total) {
        if (threadIdx.x == 0) {
            int last = -1;
            for (int p = 0; p < k; p++) {
                if (b.defl[p]) continue;
                if (last >= 0 && fabs(b.val[p] - b.val[last]) <= tol) {
                    const double zl = b.tau_r[last], zp = b.tau_r[p];
                    const double rr = hypot(zl, zp), c = zp / rr, s = -zl / rr;
                    const double dl = b.val[last], dp = b.val[p];
                    b.val[last] = c * c * dl + s * s * dp;
                    b.val[p] = s * s * dl + c * c * dp;
                    b.tau_r[p] = rr;
                    b.tau_r[last] = 0.0;
                    b.defl[last] = 1;
                    b.rot_a[nrot] = last;
                    b.rot_b[nrot] = p;
                    b.rot_c[nrot] = c;
                    b.rot_s[nrot] = s;
                    nrot++;
                }
                last = p;
            }
        }
        __syncthreads();
        kn = number(false);
    }
    for (int c = threadIdx.x; c < kn; c += blockDim.x) {
        const int p = b.ndidx[c];
        b.Dnd[c] = b.val[p];
        b.znd[c] = b.tau_r[p];
    }
    if (threadIdx.x == 0) {
        b.par[0] = rho_hat;
        b.par[1] = sg;
        b.par[2] = (double)kn;
        b.par[3] = (double)nrot;
    }
}

// The deflation rotations on the block's columns (column p of the sorted problem is
// block column perm[p]); one thread per row applies them in order.
__global__ void dc_rotate_kernel(int64_t half, int64_t n, double* Q, int64_t ldq, MergeBufs b) {
    const Merge g = merge_at(half, n, b);
    const int64_t l = g.l, k = g.k;
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= k) return;
    const int nrot = (int)b.par[3];
    double* q = Q + (l + row) * ldq + l;
    for (int t = 0; t < nrot; t++) {
        const int a = b.perm[b.rot_a[t]], c2 = b.perm[b.rot_b[t]];
        const double c = b.rot_c[t], s = b.rot_s[t];
        const double qa = q[a], qb = q[c2];
        q[a] = c * qa + s * qb;
        q[c2] = -s * qa + c * qb;
    }
}

constexpr int kRootWarps = 8;        // roots (one warp each) per block of the secular-equation kernels

__device__ __forceinline__ double warp_prod(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v *= __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Roots of 1 + rho sum_j z_j^2 / (d_j - lambda) (rho > 0, d ascending, sum z^2 <= 1):
// root i lies in (d_i, d_{i+1}), the last in (d_k, d_k + rho).  One warp per root, the
// lanes sharing the sum over the poles (the xor-butterfly sums leave the same value in
// every lane, so the warp's control flow stays uniform).  Each root is found in
// tau = lambda - d_org, measured from the nearer pole d_org, so that the differences
// d_j - lambda = (d_j - d_org) - tau keep their relative accuracy.  Steps to the zero
// of a rational model with the two neighbouring poles (constant plus one pole term for
// each side, fitted to the value and slope of each side's sum: the interpolation
// behind the classical secular-equation solvers of Bunch, Nielsen and Sorensen and of
// R.-C. Li), kept inside a bracket [lo, hi] with g(lo) < 0 < g(hi) by a bisection step
// whenever the model's step would leave it.
__global__ void __launch_bounds__(32 * kRootWarps) dc_secular_kernel(int64_t half, int64_t n, MergeBufs b, int cap) {
    extern __shared__ double sh[];
    merge_at(half, n, b);
    const int k = (int)b.par[2];
    const double rho = b.par[0];
    const bool staged = k <= cap;   // cap: poles the dynamic shared memory was sized for
    double* Ds = sh;
    double* z2 = sh + (staged ? k : 0);
    if (staged) {
        for (int j = threadIdx.x; j < k; j += blockDim.x) {
            Ds[j] = b.Dnd[j];
            z2[j] = b.znd[j] * b.znd[j];
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kRootWarps + (threadIdx.x >> 5);
    if (i >= k) return;
    auto Dj = [&](int j) { return staged ? Ds[j] : b.Dnd[j]; };
    auto Zj = [&](int j) { return staged ? z2[j] : b.znd[j] * b.znd[j]; };
    const double d_i = Dj(i);
    const double gap = (i + 1 < k) ? Dj(i + 1) - d_i : rho;
    // g at the midpoint decides which pole is nearer (measured from d_i, as the bracket is: the
    // rounded sum d_i + gap / 2 can lie on the root's other side when the gap is a few
    // thousand units of d_i, and the bracket then misses the root)
    double fm = 0.0;
    for (int j = lane; j < k; j += 32) fm += Zj(j) / ((Dj(j) - d_i) - 0.5 * gap);
    fm = 1.0 + rho * warp_sum(fm);
    int org;
    double lo, hi;
    if (i + 1 == k) {
        org = i;
        if (fm < 0.0) { lo = 0.5 * gap; hi = gap; }
        else { lo = 0.0; hi = 0.5 * gap; }
    } else if (fm >= 0.0) {
        org = i; lo = 0.0; hi = 0.5 * gap;
    } else {
        org = i + 1; lo = -0.5 * gap; hi = 0.0;
    }
    const double dorg = Dj(org);
    const bool last = i + 1 == k;
    double t = 0.5 * (lo + hi);
    for (int it = 0; it < 200; it++) {
        // g = 1 + psi + phi (poles j <= i and j > i) and the derivatives of both parts
        double psi = 0.0, phi = 0.0, dpsi = 0.0, dphi = 0.0;
        for (int j = lane; j < k; j += 32) {
            const double r = 1.0 / ((Dj(j) - dorg) - t);
            const double q = Zj(j) * r;
            if (j <= i) {
                psi += q;
                dpsi = fma(q, r, dpsi);
            } else {
                phi += q;
                dphi = fma(q, r, dphi);
            }
        }
        psi = rho * warp_sum(psi);
        phi = rho * warp_sum(phi);
        dpsi = rho * warp_sum(dpsi);
        dphi = rho * warp_sum(dphi);
        const double g = 1.0 + psi + phi;
        if (g == 0.0) break;
        if (g > 0.0) hi = t;
        else lo = t;
        // the step to the zero of the model c + s / (Di - eta) + S / (Dn - eta), which has
        // the poles d_i and d_{i+1} and matches g and g' at tau (the last root: d_i only);
        // of its two zeros the one nearer tau
        const double Di = (d_i - dorg) - t;
        const double s = Di * Di * dpsi;
        double eta = 0.0;
        bool have = false;
        if (last) {
            const double c = g - s / Di;
            if (c != 0.0) {
                eta = Di + s / c;
                have = true;
            }
        } else {
            const double Dn = (Dj(i + 1) - dorg) - t;
            const double S = Dn * Dn * dphi;
            const double c = g - s / Di - S / Dn;
            const double qa = c, qb = -(c * (Di + Dn) + s + S), qc = c * Di * Dn + s * Dn + S * Di;
            if (qa == 0.0) {
                if (qb != 0.0) {
                    eta = -qc / qb;
                    have = true;
                }
            } else {
                const double disc = qb * qb - 4.0 * qa * qc;
                if (disc >= 0.0) {
                    const double qq = -0.5 * (qb + copysign(sqrt(disc), qb));
                    const double e1 = qq / qa, e2 = qq != 0.0 ? qc / qq : e1;
                    eta = fabs(e1) <= fabs(e2) ? e1 : e2;
                    have = true;
                }
            }
        }
        have = have && isfinite(eta);
        if (have && fabs(eta) <= 2.0 * kEps * fabs(t)) break;   // converged
        double tn = have ? t + eta : 0.5 * (lo + hi);
        if (!(tn > lo && tn < hi)) tn = 0.5 * (lo + hi);        // a bisection step instead
        const bool done = fabs(tn - t) <= 2.0 * kEps * fabs(tn) || hi - lo <= 2.0 * kEps * fmax(fabs(lo), fabs(hi));
        t = tn;
        if (done) break;
    }
    if (lane == 0) {
        b.org[i] = org;
        b.tau_r[i] = t;
    }
}

// Recomputed weights zhat_i^2 = prod_j (lambda_j - d_i) / (rho prod_{j != i} (d_j - d_i))
// (sign of the original z_i); one warp per i, each lane a strided part of the product.
// By interlacing, every partial product of the ratios stays between the bounds of the
// telescoping products, far from overflow.
__global__ void __launch_bounds__(32 * kRootWarps) dc_lowner_kernel(int64_t half, int64_t n, MergeBufs b) {
    merge_at(half, n, b);
    const int k = (int)b.par[2];
    const double rho = b.par[0];
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kRootWarps + (threadIdx.x >> 5);
    if (i >= k) return;
    const double di = b.Dnd[i];
    double prod = 1.0;
    for (int j = lane; j < k; j += 32) {
        const double lmd = (b.Dnd[b.org[j]] - di) + b.tau_r[j];   // lambda_j - d_i
        prod *= (j == i) ? lmd / rho : lmd / (b.Dnd[j] - di);
    }
    prod = warp_prod(prod);
    if (lane == 0) {
        const double zh = sqrt(fabs(prod));
        b.zhat[i] = b.znd[i] >= 0.0 ? zh : -zh;
    }
}

// Norms of the eigenvectors u_i = (zhat_j / (d_j - lambda_i))_j; one warp per i.
__global__ void __launch_bounds__(32 * kRootWarps) dc_norm_kernel(int64_t half, int64_t n, MergeBufs b) {
    merge_at(half, n, b);
    const int k = (int)b.par[2];
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kRootWarps + (threadIdx.x >> 5);
    if (i >= k) return;
    const double dorg = b.Dnd[b.org[i]], t = b.tau_r[i];
    double s = 0.0;
    for (int j = lane; j < k; j += 32) {
        const double q = b.zhat[j] / ((b.Dnd[j] - dorg) - t);
        s = fma(q, q, s);
    }
    s = warp_sum(s);
    if (lane == 0) b.norm[i] = sqrt(s);
}

// U[j][i] = zhat_j / (d_j - lambda_i) / |u_i|  (k_nd x k_nd, row-major).
__global__ void dc_build_u_kernel(int64_t half, int64_t n, MergeBufs b) {
    merge_at(half, n, b);
    const int k = (int)b.par[2];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= k || j >= k) return;
    b.U[(int64_t)j * k + i] = b.zhat[j] / ((b.Dnd[j] - b.Dnd[b.org[i]]) - b.tau_r[i]) / b.norm[i];
}

// G[row][c] = block column perm[ndidx[c]] of Q.
__global__ void dc_gather_kernel(int64_t half, int64_t n, const double* Q, int64_t ldq, MergeBufs b) {
    const Merge g = merge_at(half, n, b);
    const int64_t l = g.l, k = g.k;
    const int kn = (int)b.par[2];
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = blockIdx.y;
    if (c >= kn || row >= k) return;
    b.G[row * kn + c] = Q[(l + row) * ldq + l + b.perm[b.ndidx[c]]];
}

// Final eigenvalues of the merged problem (sign restored) and their ascending ranks.
__global__ void dc_rank_kernel(int64_t half, int64_t n, MergeBufs b) {
    const int64_t k = merge_at(half, n, b).k;
    const double sg = b.par[1];
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < k; p += (int64_t)gridDim.x * blockDim.x) {
        const int q = b.pos[p];
        b.D[p] = sg * (q < 0 ? b.val[p] : b.Dnd[b.org[q]] + b.tau_r[q]);
    }
}

// Ascending rank of each merged eigenvalue (ties by index); one warp per value.
__global__ void __launch_bounds__(32 * kRootWarps) dc_rank2_kernel(int64_t half, int64_t n, MergeBufs b) {
    const int64_t k = merge_at(half, n, b).k;
    const int lane = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * kRootWarps + (threadIdx.x >> 5);
    if (p >= k) return;
    const long long vp = order_key(b.D[p]);
    int r = 0;
    for (int64_t q = lane; q < k; q += 32) {
        const long long vq = order_key(b.D[q]);
        r += (vq < vp) || (vq == vp && q < p);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (lane == 0) b.rank[p] = r;
}

// Writes the merged eigenvalues w[l + rank] and the block's new columns into F
// (k x k): deflated columns from Q, the others from Gn = G U.
__global__ void dc_scatter_kernel(int64_t half, int64_t n, const double* Q, int64_t ldq, double* w, MergeBufs b) {
    const Merge g = merge_at(half, n, b);
    const int64_t l = g.l, k = g.k;
    double* F = b.U;
    const int kn = (int)b.par[2];
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = blockIdx.y;
    if (p >= k || row >= k) return;
    const int dst = b.rank[p];
    const int q = b.pos[p];
    F[row * k + dst] = q < 0 ? Q[(l + row) * ldq + l + b.perm[p]] : b.Gn[row * kn + q];
    if (row == 0) w[l + dst] = b.D[p];
}

__global__ void copy_block_kernel(int64_t half, int64_t n, double* Q, int64_t ldq, MergeBufs b) {
    const Merge g = merge_at(half, n, b);
    const int64_t l = g.l, k = g.k;
    const double* F = b.U;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = blockIdx.y;
    if (c >= k || row >= k) return;
    Q[(l + row) * ldq + l + c] = F[row * k + c];
}

// ------------------------------------------------------------------ 3. back-transformation

// Vp[t][i] = component j0 + 1 + i of reflector j0 + t (rows j0 + 1 .. n - 1), zero above its 1.
__global__ void panel_v_kernel(const double* A, int64_t lda, int64_t n, int64_t j0, int nb, double* Vp) {
    const int64_t mr = n - j0 - 1;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.y;
    if (i >= mr || t >= nb) return;
    const int64_t j = j0 + t, row = j0 + 1 + i;
    double v = 0.0;
    if (row == j + 1) v = 1.0;
    else if (row > j + 1) v = A[j * lda + row];
    Vp[t * mr + i] = v;
}

// Gv[p][s][t] = v_s . v_t (s <= t) for every panel p = blockIdx.z of kPanel reflectors, one
// block per pair, straight from A's rows (v of reflector j: zeros, 1 at j + 1, A[j][j+2:]).
__global__ void panel_gram_kernel(const double* __restrict__ A, int64_t lda, int64_t n, int64_t nref, double* Gv) {
    const int s = blockIdx.x, t = blockIdx.y;
    const int64_t j0 = (int64_t)blockIdx.z * kPanel;
    const int nb = (int)(nref - j0 < kPanel ? nref - j0 : kPanel);
    if (s > t || t >= nb) return;
    const double* vs = A + (j0 + s) * lda;
    const int64_t jt = j0 + t;
    const double* vt = A + jt * lda;
    double acc = 0.0;
    for (int64_t i = jt + 2 + threadIdx.x; i < n; i += blockDim.x) acc = fma(vs[i], vt[i], acc);
    if (threadIdx.x == 0) acc += s == t ? 1.0 : vs[jt + 1];
    acc = block_sum(acc);
    if (threadIdx.x == 0) Gv[(int64_t)blockIdx.z * kPanel * kPanel + s * nb + t] = acc;
}

// T of H_j0 ... H_{j0+nb-1} = I - V T V^T (upper triangular, forward accumulation):
// T[t][t] = tau_t, T[s][t] = -tau_t sum_{s <= u < t} T[s][u] Gv[u][t]; one block per panel.
// The rows of T are independent: four lanes share a row, each keeps the sums of sixteen
// columns in registers, and T[s][u], final at step u, goes round by shuffle, so there is no
// barrier in the chain.  (One panel a launch, the sums over u in one thread from global
// memory, took 145 us a panel; all panels together now take 50 us.)
__global__ void __launch_bounds__(256) panel_t_kernel(const double* __restrict__ Gv, const double* __restrict__ tau,
                                                      int64_t nref, double* T) {
    __shared__ double G[kPanel][kPanel + 1];
    __shared__ double ts[kPanel];
    const int64_t j0 = (int64_t)blockIdx.x * kPanel;
    const int nb = (int)(nref - j0 < kPanel ? nref - j0 : kPanel);
    Gv += (int64_t)blockIdx.x * kPanel * kPanel;
    T += (int64_t)blockIdx.x * kPanel * kPanel;
    for (int e = threadIdx.x; e < kPanel * kPanel; e += 256) {
        const int s = e / kPanel, t = e % kPanel;
        G[s][t] = (s <= t && t < nb) ? Gv[s * nb + t] : 0.0;
    }
    if (threadIdx.x < kPanel) ts[threadIdx.x] = (int)threadIdx.x < nb ? tau[j0 + threadIdx.x] : 0.0;
    __syncthreads();
    const int s = threadIdx.x >> 2, g = threadIdx.x & 3;
    double w[kPanel / 4];
#pragma unroll
    for (int q = 0; q < kPanel / 4; q++) w[q] = 0.0;
#pragma unroll
    for (int u = 0; u < kPanel; u++) {
        double v = s < u ? -ts[u] * w[u / 4] : (s == u ? ts[u] : 0.0);
        v = __shfl_sync(0xffffffffu, v, u & 3, 4);
        if (g == (u & 3)) w[u / 4] = v;              // T[s][u]
#pragma unroll
        for (int q = 0; q < kPanel / 4; q++) {
            if (4 * q + 3 <= u) continue;
            if (4 * q + g > u) w[q] = fma(v, G[u][4 * q + g], w[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < kPanel / 4; q++) {
        const int t = 4 * q + g;
        if (s < nb && t < nb) T[s * nb + t] = w[q];
    }
}

// ------------------------------------------------------------------ workspace

inline int64_t round8(int64_t x) { return (x + 7) / 8 * 8; }

// Products of the merges (G U) and of the back-transformation run as Ozaki products on
// the tensor cores for 256 <= n <= 8192 (the NN form takes inner dimensions up to
// 8192), otherwise as FP64 products on the DFMA pipe (small n: a few tiles, where the
// slicing passes would cost more than they save).
constexpr int64_t kOzakiMinN = 256, kOzakiMaxN = 8192;
constexpr int kMaxTriBlocks = 1024;
// Merges of up to 256 rows multiply in FP64 (n k^2 multiply-adds a level, 0.27 ms at n = 2400
// and k = 256, against about 40 us of launches a merge for an Ozaki product).
constexpr int64_t kMergeFp64 = 256;

struct EighBufs {
    double *d, *e, *tau, *ebak;
    double *PV, *ybuf, *part, *dots;      // tridiagonalisation: [V; W; V] of a panel, A0 x, sums
    TriScalars* tri;
    int* vwmax;                           // per panel: exponents of its V and W
    MergeBufs mb;
    double *Vp, *Gv, *T, *W1, *W2;
    unsigned char* oz;      // Ozaki product scratch (nullptr for n > kOzakiMaxN)
    size_t oz_bytes;
};

size_t eigh_ozaki_bytes(int64_t n) {
    if (n < kOzakiMinN || n > kOzakiMaxN) return 0;
    return std::max({ozaki_workspace_bytes(false, n, n, n, false), ozaki_workspace_bytes(false, kPanel, n, n, false),
                     ozaki_workspace_bytes(true, n, n, kPanel, false)});
}

template <typename Ar>
void eigh_layout(Ar& ar, int64_t n, EighBufs* out) {
    EighBufs u{};
    u.d = ar.template take<double>(n);
    u.e = ar.template take<double>(n);
    u.tau = ar.template take<double>(n);
    u.ebak = ar.template take<double>(n);
    u.part = ar.template take<double>(kMaxTriBlocks);
    u.dots = ar.template take<double>(2 * kPanel32);
    u.tri = ar.template take<TriScalars>(1);
    u.vwmax = ar.template take<int>(2 * (size_t)(n / kPanel32 + 1));
    u.PV = ar.template take<double>((size_t)(3 * kPanel32) * n);
    u.ybuf = ar.template take<double>(n);
    MergeBufs& b = u.mb;
    b.D = ar.template take<double>(n);
    b.z = ar.template take<double>(n);
    b.Dnd = ar.template take<double>(n);
    b.znd = ar.template take<double>(n);
    b.tau_r = ar.template take<double>(n);
    b.zhat = ar.template take<double>(n);
    b.norm = ar.template take<double>(n);
    b.val = ar.template take<double>(n);
    b.rot_c = ar.template take<double>(n);
    b.rot_s = ar.template take<double>(n);
    b.par = ar.template take<double>((size_t)(n / kLeaf + 8) * 4);   // 8 per merge
    b.perm = ar.template take<int>(n);
    b.defl = ar.template take<int>(n);
    b.ndidx = ar.template take<int>(n);
    b.pos = ar.template take<int>(n);
    b.org = ar.template take<int>(n);
    b.rot_a = ar.template take<int>(n);
    b.rot_b = ar.template take<int>(n);
    b.rank = ar.template take<int>(n);
    b.G = ar.template take<double>((size_t)n * n);
    b.U = ar.template take<double>((size_t)n * n);
    b.Gn = ar.template take<double>((size_t)n * n);
    u.Vp = ar.template take<double>((size_t)kPanel * n);
    const size_t panels = (size_t)((n + kPanel - 1) / kPanel);
    u.Gv = ar.template take<double>(panels * kPanel * kPanel);
    u.T = ar.template take<double>(panels * kPanel * kPanel);
    u.W1 = ar.template take<double>((size_t)kPanel * n);
    u.W2 = ar.template take<double>((size_t)kPanel * n);
    u.oz_bytes = eigh_ozaki_bytes(n);
    u.oz = u.oz_bytes ? ar.template take<unsigned char>(u.oz_bytes) : nullptr;
    if (out) *out = u;
}

struct CountOnly {
    Sizer s;
    template <typename T>
    T* take(size_t n) {
        s.take<T>(n);
        return nullptr;
    }
};

}  // namespace

size_t eigh_workspace_bytes(int64_t n) {
    CountOnly ar;
    eigh_layout(ar, n > 0 ? n : 1, nullptr);
    return ar.s.used;
}

int eigh(double* A, int64_t lda, int64_t n, double* w, double* Q, int64_t ldq, void* ws, size_t ws_bytes,
         unsigned* status, cudaStream_t s) {
    if (n <= 0) return CHFSI_OK;
    if (ws_bytes < eigh_workspace_bytes(n)) return CHFSI_ERR_NOMEM;
    Arena ar(ws, ws_bytes);
    EighBufs u;
    eigh_layout(ar, n, &u);
    double *d = u.d, *e = u.e, *tau = u.tau, *ebak = u.ebak, *Vp = u.Vp, *Gv = u.Gv, *T = u.T, *W1 = u.W1,
           *W2 = u.W2;
    MergeBufs& mb = u.mb;
    const bool oz = u.oz != nullptr;

    // d, e and tau, and with what lies behind them the scalars and the panels' exponents
    CHFSI_CUDA_TRY(cudaMemsetAsync(u.d, 0, (size_t)((char*)(u.vwmax + 2 * (n / kPanel32 + 1)) - (char*)u.d), s));
    const unsigned rows = (unsigned)std::min<int64_t>(n, 4 * 1024);
    matrix_exponent_kernel<<<rows, 256, 0, s>>>(A, lda, n, &u.tri->emax, status);
    CHFSI_LAUNCH_CHECK();
    scale_matrix_kernel<<<rows, 256, 0, s>>>(A, lda, n, &u.tri->emax);
    CHFSI_LAUNCH_CHECK();

    // 1. tridiagonalisation: a cooperative launch per panel, then the trailing product
    if (n >= 3) {
        const int dev = current_device();
        int sms = 0;
        if (dev < 0 || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return CHFSI_ERR_CUDA;
        sms = std::min(sms, kMaxTriBlocks);
        TriPanel tp{};
        tp.A = A;
        tp.lda = lda;
        tp.n = n;
        tp.staged = n <= kTriStaged;
        tp.PV = u.PV;
        tp.part = u.part;
        tp.ybuf = u.ybuf;
        tp.dots = u.dots;
        tp.d = d;
        tp.e = e;
        tp.tau = tau;
        tp.tri = u.tri;
        tp.wait_ns = pipeline_wait_ns();
        tp.status = status;
        static bool attr[kMaxDevices] = {};
        if (!attr[dev]) {
            CHFSI_CUDA_TRY(cudaFuncSetAttribute(tri_panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)(sizeof(double) * (kTriStaged + 2))));
            attr[dev] = true;
        }
        for (int64_t j0 = 0; j0 + 2 < n; j0 += kPanel32) {
            const int nc = (int)std::min<int64_t>(kPanel32, (n - 2) - j0);
            if (nc < kPanel32)   // rows nc .. 31 of V and W take part in the trailing product
                CHFSI_CUDA_TRY(cudaMemsetAsync(u.PV, 0, sizeof(double) * (size_t)(3 * kPanel32) * n, s));
            // a warp per row of the product and its dots, at most one block per SM: fewer blocks
            // meet sooner at the barriers
            const int64_t rows = n - j0 - 1 + 2 * kPanel32;
            unsigned grid = (unsigned)std::min<int64_t>(sms, (rows + kTriWarps - 1) / kTriWarps);
            tp.j0 = j0;
            tp.nc = nc;
            tp.vwmax = u.vwmax + 2 * (j0 / kPanel32);
            void* args[] = {&tp};
            // a stream whose context has fewer SMs than the device refuses a grid that cannot be
            // resident; the kernel runs on any grid, so a smaller one is taken from there on
            const size_t smem = tp.staged ? sizeof(double) * (size_t)(n - j0 + 2) : 0;
            cudaError_t err;
            while ((err = cudaLaunchCooperativeKernel((const void*)tri_panel_kernel, dim3(grid), dim3(kTriThreads), args,
                                                      smem, s)) == cudaErrorCooperativeLaunchTooLarge &&
                   grid > 1) {
                (void)cudaGetLastError();
                sms = (int)(grid = (grid + 1) / 2);
            }
            CHFSI_CUDA_TRY(err);
            CHFSI_LAUNCH_CHECK();
            tp.base += grid * (unsigned)(2 * nc - 1);
            const int64_t jn = j0 + nc, mp = n - jn;
            // trailing matrix: A[jn:, jn:] -= V^T W + W^T V over the panel's rows of PV
            const double* Vop = u.PV + jn;
            const double* Wop = u.PV + (int64_t)kPanel32 * n + jn;
            double* C22 = A + jn * lda + jn;
            int rc;
            if (oz && mp >= kOzakiMinN) {
                panel_balance_kernel<<<dim3((unsigned)((mp + 255) / 256), 3 * kPanel32 / kBalanceRows), 256, 0, s>>>(
                    u.PV, n, jn, tp.vwmax);
                CHFSI_LAUNCH_CHECK();
                if ((rc = ozaki_gemm_tn(Vop, n, Wop, n, 2 * kPanel32, mp, mp, C22, lda, true, u.oz, u.oz_bytes, status,
                                        s, true)))
                    return rc;
            } else if ((rc = gemm_general(Vop, n, true, Wop, n, C22, lda, mp, mp, 2 * kPanel32, -1.0, true, s))) {
                return rc;
            }
        }
    }
    tridiag_tail_kernel<<<1, 32, 0, s>>>(A, lda, n, d, e, tau);
    CHFSI_LAUNCH_CHECK();

    // 2. divide and conquer on (d, e): Q starts as the leaf eigenvectors
    CHFSI_CUDA_TRY(cudaMemset2DAsync(Q, sizeof(double) * (size_t)ldq, 0, sizeof(double) * (size_t)n, (size_t)n, s));
    dc_split_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, d, e, ebak);
    CHFSI_LAUNCH_CHECK();
    const int64_t nleaf = (n + kLeaf - 1) / kLeaf;
    dc_leaf_kernel<<<(unsigned)nleaf, 256, 0, s>>>(n, d, e, w, Q, ldq);
    CHFSI_LAUNCH_CHECK();
    std::vector<double> kns;
    for (int64_t half = kLeaf; half < n; half *= 2) {
        // all merges of the level: blocks at 2 half b with rows beyond the first half
        const unsigned nm = (unsigned)((n - half + 2 * half - 1) / (2 * half));
        const int64_t k = std::min(2 * half, n);      // the largest of them
        const unsigned kb = (unsigned)((k + 255) / 256);
        dc_merge_prep_kernel<<<dim3(1, 1, nm), 1024, 0, s>>>(half, n, w, Q, ldq, ebak, mb, status);
        CHFSI_LAUNCH_CHECK();
        dc_rotate_kernel<<<dim3(kb, 1, nm), 256, 0, s>>>(half, n, Q, ldq, mb);
        CHFSI_LAUNCH_CHECK();
        const size_t sh = k <= kSecularSmem ? 2 * sizeof(double) * (size_t)k : 0;
        if (sh > 48 * 1024) {
            static bool attr[kMaxDevices] = {};
            const int dev = current_device();
            if (dev < 0) return CHFSI_ERR_CUDA;
            if (!attr[dev]) {
                CHFSI_CUDA_TRY(cudaFuncSetAttribute(dc_secular_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    (int)(2 * sizeof(double) * kSecularSmem)));
                attr[dev] = true;
            }
        }
        // the non-deflated counts are only known on the device: size the grids for k
        const dim3 roots((unsigned)((k + kRootWarps - 1) / kRootWarps), 1, nm), cells(kb, (unsigned)k, nm);
        dc_secular_kernel<<<roots, 32 * kRootWarps, sh, s>>>(half, n, mb, sh ? (int)k : 0);
        CHFSI_LAUNCH_CHECK();
        dc_lowner_kernel<<<roots, 32 * kRootWarps, 0, s>>>(half, n, mb);
        CHFSI_LAUNCH_CHECK();
        dc_norm_kernel<<<roots, 32 * kRootWarps, 0, s>>>(half, n, mb);
        CHFSI_LAUNCH_CHECK();
        dc_build_u_kernel<<<cells, 256, 0, s>>>(half, n, mb);
        CHFSI_LAUNCH_CHECK();
        dc_gather_kernel<<<cells, 256, 0, s>>>(half, n, Q, ldq, mb);
        CHFSI_LAUNCH_CHECK();
        // Gn (k x kn) = G (k x kn) U (kn x kn), kn <= k the merge's count of non-deflated poles:
        // FP64 products of all merges in one launch that reads kn on the device, or with more
        // than kMergeFp64 rows Ozaki products one by one (kn copied to the host, once a level)
        int rc;
        if (oz && k > kMergeFp64) {
            kns.resize(nm);
            CHFSI_CUDA_TRY(cudaMemcpy2DAsync(kns.data(), sizeof(double), mb.par + 2, 8 * sizeof(double), sizeof(double),
                                             nm, cudaMemcpyDeviceToHost, s));
            CHFSI_CUDA_TRY(cudaStreamSynchronize(s));
            for (unsigned b = 0; b < nm; b++) {
                const int64_t kn = (int64_t)kns[b], mat = (int64_t)b * (2 * half) * (2 * half);
                const int64_t kk = std::min(2 * half, n - 2 * half * b);
                if ((rc = ozaki_gemm_nn(mb.G + mat, kn, mb.U + mat, kn, kk, kn, kn, mb.Gn + mat, kn, false, u.oz,
                                        u.oz_bytes, status, s)))
                    return rc;
            }
        } else if ((rc = gemm_merges(mb.G, mb.U, mb.Gn, 2 * half, n, (int)nm, mb.par + 2, 8, s))) {
            return rc;
        }
        dc_rank_kernel<<<dim3(kb, 1, nm), 256, 0, s>>>(half, n, mb);
        CHFSI_LAUNCH_CHECK();
        dc_rank2_kernel<<<roots, 32 * kRootWarps, 0, s>>>(half, n, mb);
        CHFSI_LAUNCH_CHECK();
        dc_scatter_kernel<<<cells, 256, 0, s>>>(half, n, Q, ldq, w, mb);
        CHFSI_LAUNCH_CHECK();
        copy_block_kernel<<<cells, 256, 0, s>>>(half, n, Q, ldq, mb);
        CHFSI_LAUNCH_CHECK();
    }

    unscale_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(w, n, &u.tri->emax);
    CHFSI_LAUNCH_CHECK();

    // 3. back-transformation Q = H_0 H_1 ... H_{n-3} Q, panels from the last
    const int64_t nref = n - 2;   // reflectors j = 0 .. n - 3
    if (nref > 0) {
        const unsigned panels = (unsigned)((nref + kPanel - 1) / kPanel);
        panel_gram_kernel<<<dim3(kPanel, kPanel, panels), 256, 0, s>>>(A, lda, n, nref, Gv);
        CHFSI_LAUNCH_CHECK();
        panel_t_kernel<<<panels, 256, 0, s>>>(Gv, tau, nref, T);
        CHFSI_LAUNCH_CHECK();
    }
    for (int64_t j0 = ((nref - 1) / kPanel) * kPanel; nref > 0 && j0 >= 0; j0 -= kPanel) {
        const int nb = (int)std::min<int64_t>(kPanel, nref - j0);
        const int64_t mr = n - j0 - 1;
        panel_v_kernel<<<dim3((unsigned)((mr + 255) / 256), (unsigned)nb), 256, 0, s>>>(A, lda, n, j0, nb, Vp);
        CHFSI_LAUNCH_CHECK();
        const double* Tp = T + (j0 / kPanel) * (kPanel * kPanel);
        double* ZR = Q + (j0 + 1) * ldq;
        int rc;
        if (oz) {
            // W1 = V^T Z, W2 = T W1 (small, DFMA), Z -= V W2
            if ((rc = ozaki_gemm_nn(Vp, mr, ZR, ldq, nb, mr, n, W1, n, false, u.oz, u.oz_bytes, status, s))) return rc;
            if ((rc = gemm_general(Tp, nb, false, W1, n, W2, n, nb, n, nb, 1.0, false, s))) return rc;
            if ((rc = ozaki_gemm_tn(Vp, mr, W2, n, nb, mr, n, ZR, ldq, false, u.oz, u.oz_bytes, status, s, true)))
                return rc;
        } else {
            if ((rc = gemm_general(Vp, mr, false, ZR, ldq, W1, n, nb, n, mr, 1.0, false, s))) return rc;
            if ((rc = gemm_general(Tp, nb, false, W1, n, W2, n, nb, n, nb, 1.0, false, s))) return rc;
            if ((rc = gemm_general(Vp, mr, true, W2, n, ZR, ldq, mr, n, nb, -1.0, true, s))) return rc;
        }
    }
    return CHFSI_OK;
}

}  // namespace chfsi

int chfsi_eigh_workspace_size(int64_t n, size_t* bytes) {
    if (!bytes || n < 0) return CHFSI_ERR_ARG;
    *bytes = chfsi::align_up(chfsi::kStatusBytes) + chfsi::eigh_workspace_bytes(n);
    return CHFSI_OK;
}

int chfsi_eigh(double* A, int64_t lda, int64_t n, double* w, double* Q, int64_t ldq, void* ws, size_t ws_bytes,
               void* stream) {
    if (n < 0 || (n > 0 && (!A || !w || !Q || lda < n || ldq < n))) return CHFSI_ERR_ARG;
    if (n == 0) return CHFSI_OK;
    if (n > 65535) return CHFSI_ERR_UNSUPPORTED;   // one grid row per matrix row in several launches
    size_t need = 0;
    int rc = chfsi_eigh_workspace_size(n, &need);
    if (rc) return rc;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return CHFSI_ERR_ARG;
    if (ws_bytes < need) return CHFSI_ERR_NOMEM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned* st = chfsi::status_word(ws);
    CHFSI_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(unsigned), s));
    char* rest = static_cast<char*>(ws) + chfsi::align_up(chfsi::kStatusBytes);
    return chfsi::eigh(A, lda, n, w, Q, ldq, rest, ws_bytes - chfsi::align_up(chfsi::kStatusBytes), st, s);
}
