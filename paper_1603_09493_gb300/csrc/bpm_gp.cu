// Efficient global optimisation (Sec. II.A; Jones, Schonlau, Welch 1998) on the
// GPU: maximin choice among random Latin hypercubes, the concentrated kriging
// likelihood for a batch of correlation-length vectors, the kriging fit, and
// the predictor, its mean squared error and the expected improvement over
// large candidate sets.  FP64 throughout: the kriging systems are small
// (n <= 2048 training designs) and nearly singular for long correlation
// lengths, where lower precision loses the variance.
//
//   R_ij = exp(-sum_k theta_k (x_ik - x_jk)^2) + nugget [i == j]
//   mu = 1'R^-1 y / 1'R^-1 1,  sigma2 = (y - mu)'R^-1(y - mu) / n,
//   nll = n ln sigma2 + ln det R
//   yhat(x) = mu + r'R^-1(y - mu),  s2 = sigma2 [1 - r'R^-1 r + (1 - 1'R^-1 r)^2 / 1'R^-1 1]
//   EI = (f_min - yhat) Phi(z) + s phi(z),  z = (f_min - yhat) / s
#include <algorithm>
#include <cmath>
#include <vector>

#include "bpm_internal.cuh"

namespace bpm {

struct Gp {
    int n = 0, d = 0;
    double mu = 0, sigma2 = 0, one_Ri_1 = 0;
    double* X = nullptr;      // [n][d]
    double* theta = nullptr;  // [d]
    double* Linv = nullptr;   // [n][n] inverse of the Cholesky factor (lower)
    double* a = nullptr;      // [n] R^-1 (y - mu)
    double* c = nullptr;      // [n] Linv 1
};

void free_gp(Gp* g) {
    if (!g) return;
    cudaFree(g->X);
    cudaFree(g->theta);
    cudaFree(g->Linv);
    cudaFree(g->a);
    cudaFree(g->c);
    delete g;
}

namespace {

constexpr int kGpThreads = 256;
constexpr int kGpMaxN = 2048, kGpMaxD = 64;

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// fixed-order CTA sum, result in every thread
__device__ double cta_sum(double v, double* red) {
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    return s;
}

// smallest squared distance between two points of each candidate design
__global__ void __launch_bounds__(kGpThreads) k_lhs_min_d2(const double* __restrict__ C, int n, int d,
                                                           double* __restrict__ out) {
    __shared__ double red[kGpThreads / 32];
    const double* X = C + (size_t)blockIdx.x * n * d;
    double m = INFINITY;
    for (int i = 0; i < n - 1; ++i)
        for (int j = i + 1 + threadIdx.x; j < n; j += blockDim.x) {
            double s = 0.0;
            for (int k = 0; k < d; ++k) {
                const double t = X[i * d + k] - X[j * d + k];
                s += t * t;
            }
            m = fmin(m, s);
        }
    for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double r = INFINITY;
        for (int w = 0; w < kGpThreads / 32; ++w) r = fmin(r, red[w]);
        out[blockIdx.x] = r;
    }
}

// ---------------------------------------------------------------------------
// Cholesky factors of the correlation matrices of a batch of theta vectors, blocked over the whole GPU.
// Matrix t is A[t] [n + 2][n], the lower triangle of R with two more rows, y and 1: factoring the first
// n rows turns them into z = L^-1 y and w = L^-1 1, so the solves cost no pass of their own.  Per block
// of 32 columns one launch factors the diagonal block (every CTA for itself) and solves 32 rows below
// it a CTA, one launch subtracts the block's products from 32 x 32 tiles to its right.  The factored
// diagonal blocks have a place of their own, D[t] [block][32][32]: a CTA of the matrix may start after
// another has finished, so the block they all load is never written.  An element's products are
// subtracted in the order of k, one rounding each, as an unblocked factorisation does; the row solve
// rounds a factor's quotient once more.
// An SM does two FP64 multiply-adds a cycle: n = 160, 32 vectors are 22 M for the factors and as many
// for the correlations, 0.08 ms spread over the GPU.  One CTA a matrix, unblocked from global memory,
// took 1.40 ms; 0.47 ms now.
// ---------------------------------------------------------------------------
constexpr int kPB = 32;

// doubles of a matrix's factored diagonal blocks
__host__ __device__ __forceinline__ size_t diag_doubles(int n) { return (size_t)((n + kPB - 1) / kPB) * kPB * kPB; }

// rows 0 .. n - 1: the lower triangle of R; row n: y; row n + 1: ones
__global__ void __launch_bounds__(kGpThreads) k_gp_matrix(const double* __restrict__ X, const double* __restrict__ y,
                                                          int n, int d, const double* __restrict__ theta,
                                                          double nugget, double* __restrict__ Aall) {
    const int j = blockIdx.x * kPB + (threadIdx.x & 31), t = blockIdx.z;
    if ((int)blockIdx.x > (int)blockIdx.y && (int)(blockIdx.y + 1) * kPB < n) return;   // above the diagonal
    double* A = Aall + (size_t)t * (n + 2) * n;
    const double* th = theta + (size_t)t * d;
    for (int i = blockIdx.y * kPB + (threadIdx.x >> 5); i < min(n + 2, (int)(blockIdx.y + 1) * kPB);
         i += kGpThreads / 32) {
        if (j >= n || (i < n && j > i)) continue;
        double v;
        if (i >= n) {
            v = i == n ? y[j] : 1.0;
        } else {
            double s = 0.0;
            for (int k = 0; k < d; ++k) {
                const double u = X[i * d + k] - X[j * d + k];
                s += th[k] * u * u;
            }
            v = exp(-s) + (i == j ? nugget : 0.0);
        }
        A[(size_t)i * n + j] = v;
    }
}

// Columns k0 .. k0 + 31: factor the diagonal block (CTA 0 of the matrix writes it to Dall), solve the
// 32 rows of this CTA below it.  A non-positive pivot marks the matrix as failed.
__global__ void __launch_bounds__(kGpThreads) k_gp_panel(int n, int k0, double* __restrict__ Aall,
                                                         double* __restrict__ Dall, int* __restrict__ fail) {
    __shared__ double D[kPB][kPB + 1], P[kPB][kPB + 1], inv[kPB];
    __shared__ int s_bad;
    const int t = blockIdx.y, nb = min(kPB, n - k0), r0 = k0 + nb + kPB * blockIdx.x;
    // one thread reads the mark, which another CTA of the matrix may set meanwhile
    if (threadIdx.x == 0) s_bad = *(volatile int*)(fail + t);
    __syncthreads();
    if (s_bad) return;
    double* A = Aall + (size_t)t * (n + 2) * n;
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w == 0) inv[l] = 0.0;
    for (int i = w; i < kPB; i += kGpThreads / 32) {
        D[i][l] = i < nb && l <= i ? A[(size_t)(k0 + i) * n + k0 + l] : 0.0;
        P[i][l] = r0 + i < n + 2 && l < nb ? A[(size_t)(r0 + i) * n + k0 + l] : 0.0;
    }
    __syncthreads();
    for (int k = 0; k < nb; ++k) {
        if (w == 0) {                                       // one warp: an FP64 root or quotient costs every lane
            const double piv = D[k][k];
            double iv = 0.0;
            if (l == 0) {
                iv = rsqrt(piv);                            // one chain of FP64 latencies for root and quotient
                inv[k] = iv;
                if (!(piv > 0.0)) s_bad = 1;
            }
            iv = __shfl_sync(0xffffffffu, iv, 0);
            __syncwarp();
            if (l >= k && l < nb) D[l][k] *= iv;            // L_kk = piv / sqrt(piv)
        }
        __syncthreads();
        if (s_bad) {
            if (threadIdx.x == 0) fail[t] = 1;              // every CTA of the matrix writes the same
            return;
        }
        for (int i = k + 1 + w; i < nb; i += kGpThreads / 32)
            if (l > k && l <= i) D[i][l] -= D[i][k] * D[l][k];
        __syncthreads();
    }
    if (blockIdx.x == 0) {
        double* F = Dall + (size_t)t * diag_doubles(n) + (size_t)k0 * kPB;
        for (int i = w; i < kPB; i += kGpThreads / 32) F[i * kPB + l] = D[i][l];
    }
    // row solve: a warp per four rows, lane = column.  The right-hand sides stay unscaled, the quotients
    // go into the factor's columns (one multiply-add an element and step) and into the result.
    double a[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = P[4 * w + q][l];
    for (int k = 0; k < nb; ++k) {
        const double c = l > k ? -D[l][k] * inv[k] : 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] += __shfl_sync(0xffffffffu, a[q], k) * c;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = r0 + 4 * w + q;
        if (i < n + 2 && l < nb) A[(size_t)i * n + k0 + l] = a[q] * inv[l];
    }
}

// Tiles right of the panel: A[i][j] -= sum over its columns of A[i][k] A[j][k] (j <= i for the rows of R)
__global__ void __launch_bounds__(kGpThreads) k_gp_update(int n, int k0, double* __restrict__ Aall,
                                                          const int* __restrict__ fail) {
    __shared__ double Ri[kPB][kPB + 1], Rj[kPB][kPB + 1];
    const int t = blockIdx.z, j0 = k0 + kPB * (1 + blockIdx.x), i0 = k0 + kPB * (1 + blockIdx.y);
    if ((i0 + kPB <= n && i0 < j0) || j0 >= n || fail[t]) return;   // above the diagonal; the last row block has y and 1
    double* A = Aall + (size_t)t * (n + 2) * n;
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int r = w; r < kPB; r += kGpThreads / 32) {
        Ri[r][l] = i0 + r < n + 2 ? A[(size_t)(i0 + r) * n + k0 + l] : 0.0;
        Rj[r][l] = j0 + r < n ? A[(size_t)(j0 + r) * n + k0 + l] : 0.0;
    }
    __syncthreads();
    const int j = j0 + l;
    double acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + 4 * w + q;
        acc[q] = i < n + 2 && j < n ? A[(size_t)i * n + j] : 0.0;
    }
#pragma unroll 8
    for (int k = 0; k < kPB; ++k) {
        const double b = Rj[l][k];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] -= Ri[4 * w + q][k] * b;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + 4 * w + q;
        if (i < n + 2 && j < n && (i >= n || j <= i)) A[(size_t)i * n + j] = acc[q];
    }
}

// nll = n ln sigma2 + ln det R from the factored matrix (one CTA each); +inf where it failed
__global__ void __launch_bounds__(kGpThreads) k_gp_stats(int n, const double* __restrict__ Aall,
                                                         const double* __restrict__ Dall,
                                                         const int* __restrict__ fail, double* __restrict__ nll,
                                                         double* __restrict__ stats) {
    __shared__ double red[kGpThreads / 32];
    const int t = blockIdx.x;
    if (fail[t]) {
        if (threadIdx.x == 0) nll[t] = INFINITY;
        return;
    }
    const double* A = Aall + (size_t)t * (n + 2) * n;
    const double *z = A + (size_t)n * n, *w = z + n, *D = Dall + (size_t)t * diag_doubles(n);
    double ww = 0.0, wz = 0.0, ld = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        ww += w[i] * w[i];
        wz += w[i] * z[i];
        ld += log(D[(size_t)i * kPB + (i & (kPB - 1))]);
    }
    ww = cta_sum(ww, red);
    wz = cta_sum(wz, red);
    ld = cta_sum(ld, red);
    const double mu = wz / ww;
    double rr = 0.0;                           // |L^-1 (y - mu 1)|^2 = (y - mu)'R^-1(y - mu)
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double r = z[i] - mu * w[i];
        rr += r * r;
    }
    rr = cta_sum(rr, red);
    if (threadIdx.x == 0) {
        const double sigma2 = rr / n;
        nll[t] = sigma2 > 0.0 ? n * log(sigma2) + 2.0 * ld : INFINITY;
        if (stats) {
            stats[3 * t] = mu;
            stats[3 * t + 1] = sigma2;
            stats[3 * t + 2] = ww;        // 1'R^-1 1
        }
    }
}

// factors and likelihoods of T matrices (A: T (n + 2) n doubles, D: T diag_doubles(n), fail: T ints)
int gp_factor(cudaStream_t s, const double* X, const double* y, int n, int d, const double* theta, int T,
              double nugget, double* A, double* D, int* fail, double* nll, double* stats) {
    const int nblk = (n + kPB - 1) / kPB, nrow = (n + 2 + kPB - 1) / kPB;
    BPM_CK(cudaMemsetAsync(fail, 0, T * sizeof(int), s));
    for (int t0 = 0; t0 < T; t0 += 32768) {                 // grid y and z limit
        const int m = std::min(32768, T - t0);
        double *At = A + (size_t)t0 * (n + 2) * n, *Dt = D + (size_t)t0 * diag_doubles(n);
        k_gp_matrix<<<dim3(nblk, nrow, m), kGpThreads, 0, s>>>(X, y, n, d, theta + (size_t)t0 * d, nugget, At);
        for (int p = 0; p < nblk; ++p) {
            const int k0 = p * kPB, below = n + 2 - std::min(n, k0 + kPB);
            k_gp_panel<<<dim3((below + kPB - 1) / kPB, m), kGpThreads, 0, s>>>(n, k0, At, Dt, fail + t0);
            if (p + 1 < nblk)
                k_gp_update<<<dim3(nblk - p - 1, nrow - p - 1, m), kGpThreads, 0, s>>>(n, k0, At, fail + t0);
        }
        k_gp_stats<<<m, kGpThreads, 0, s>>>(n, At, Dt, fail + t0, nll + t0,
                                            stats ? stats + 3 * (size_t)t0 : nullptr);
    }
    BPM_CK(cudaGetLastError());
    return BPM_OK;
}

// Block row i0 .. i0 + 31 of Linv = L^-1 (L: [n + 2][n] below its diagonal blocks, which are D): 32 columns
// a CTA, products of the block rows above (in the order of k) first, then the triangular solve within the
// block; Linv_ij = -s / L_ii.
// (One thread per column walked the whole triangle: 0.81 ms at n = 160; 0.26 ms now.)
__global__ void __launch_bounds__(kGpThreads) k_gp_linv(const double* __restrict__ L,
                                                        const double* __restrict__ D, int n, int i0,
                                                        double* __restrict__ Linv) {
    __shared__ double Lb[kPB][kPB + 1], Xb[kPB][kPB + 1];
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5, j = blockIdx.x * kPB + l;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k0 = blockIdx.x * kPB; k0 < i0; k0 += kPB) {   // rows of Linv above column block: zero
        __syncthreads();
        for (int r = w; r < kPB; r += kGpThreads / 32) {
            Lb[r][l] = i0 + r < n ? L[(size_t)(i0 + r) * n + k0 + l] : 0.0;
            Xb[r][l] = j < n ? Linv[(size_t)(k0 + r) * n + j] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < kPB; ++k)
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] += Lb[4 * w + q][k] * Xb[k][l];
    }
    __syncthreads();
    for (int r = w; r < kPB; r += kGpThreads / 32)
        Lb[r][l] = D[(size_t)(i0 + r) * kPB + l];           // zeros above the diagonal and past n
#pragma unroll
    for (int q = 0; q < 4; ++q) Xb[4 * w + q][l] = s[q];
    __syncthreads();
    if (w) return;
    const double dinv = i0 + l < n ? 1.0 / Lb[l][l] : 0.0;  // of every row at once
    for (int r = 0; r < kPB && i0 + r < n; ++r) {           // one warp, lane = column
        const int i = i0 + r;
        double u[4] = {Xb[r][l], 0.0, 0.0, 0.0};            // four sums: a chain of FP64 latencies otherwise
        int k = 0;
        for (; k + 4 <= r; k += 4)
#pragma unroll
            for (int e = 0; e < 4; ++e) u[e] += Lb[r][k + e] * Xb[k + e][l];
        for (; k < r; ++k) u[0] += Lb[r][k] * Xb[k][l];
        const double q = __shfl_sync(0xffffffffu, dinv, r);
        const double v = i == j ? q : i > j ? -((u[0] + u[1]) + (u[2] + u[3])) * q : 0.0;
        Xb[r][l] = v;
        if (j < n) Linv[(size_t)i * n + j] = v;
    }
}

// u = Linv (y - mu 1) and c = Linv 1 (one thread per row)
__global__ void k_gp_rows(const double* __restrict__ Linv, const double* __restrict__ y, double mu, int n,
                          double* __restrict__ u, double* __restrict__ c) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double su = 0.0, sc = 0.0;
    for (int j = 0; j <= i; ++j) {
        const double l = Linv[(size_t)i * n + j];
        su += l * (y[j] - mu);
        sc += l;
    }
    u[i] = su;
    c[i] = sc;
}

// a = Linv' u = R^-1 (y - mu 1) (one thread per column)
__global__ void k_gp_cols(const double* __restrict__ Linv, const double* __restrict__ u, int n,
                          double* __restrict__ a) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double s = 0.0;
    for (int i = j; i < n; ++i) s += Linv[(size_t)i * n + j] * u[i];
    a[j] = s;
}

// Rc[c][i] = exp(-sum_k theta_k (C_ck - X_ik)^2)
__global__ void k_gp_corr(const double* __restrict__ C, const double* __restrict__ X,
                          const double* __restrict__ theta, int N, int n, int d, double* __restrict__ Rc) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (long long)N * n) return;
    const int c = (int)(q / n), i = (int)(q % n);
    double s = 0.0;
    for (int k = 0; k < d; ++k) {
        const double t = C[(size_t)c * d + k] - X[(size_t)i * d + k];
        s += theta[k] * t * t;
    }
    Rc[q] = exp(-s);
}

// V[N][n] = Rc[N][n] * Linv[n][n]^T, FP64, 32 x 64 tiles, 2 x 4 outputs per thread (64 x 64 tiles of
// 4000 candidates and n = 160 were 189 CTAs of unequal depth on 152 SMs: 329 us, 236 now).  B lower
// triangular: row r of B is zero past column r, so output columns n0 .. n0 + 63 need K only up
// to n0 + 64 (the skipped products are exact zeros; the sums are unchanged)
constexpr int kTM = 32, kTN = 64, kTK = 16;
__global__ void __launch_bounds__(256) k_gp_gemm_nt(const double* __restrict__ A, const double* __restrict__ B,
                                                    int M, int N, int K, double* __restrict__ Cout) {
    __shared__ double As[kTK][kTM + 1];
    __shared__ double Bs[kTK][kTN + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * kTM, n0 = blockIdx.x * kTN;
    double acc[2][4] = {};
    const int kend = min(K, n0 + kTN);
    for (int k0 = 0; k0 < kend; k0 += kTK) {
        for (int e = threadIdx.x; e < kTN * kTK; e += 256) {
            const int r = e / kTK, kk = e % kTK;
            if (r < kTM) As[kk][r] = (m0 + r < M && k0 + kk < K) ? A[(size_t)(m0 + r) * K + k0 + kk] : 0.0;
            Bs[kk][r] = (n0 + r < N && k0 + kk < K) ? B[(size_t)(n0 + r) * K + k0 + kk] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kTK; ++kk) {
            double av[2], bv[4];
#pragma unroll
            for (int q = 0; q < 2; ++q) av[q] = As[kk][ty + 16 * q];
#pragma unroll
            for (int q = 0; q < 4; ++q) bv[q] = Bs[kk][tx + 16 * q];
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] += av[p] * bv[q];
        }
        __syncthreads();
    }
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = m0 + ty + 16 * p, col = n0 + tx + 16 * q;
            if (r < M && col < N) Cout[(size_t)r * N + col] = acc[p][q];
        }
}

// predictor, MSE and expected improvement (one warp per candidate)
__global__ void k_gp_ei(const double* __restrict__ Rc, const double* __restrict__ V, const double* __restrict__ a,
                        const double* __restrict__ cvec, int N, int n, double mu, double sigma2, double one_Ri_1,
                        double f_min, double* __restrict__ yhat, double* __restrict__ s_out,
                        double* __restrict__ ei) {
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (c >= N) return;
    double sy = 0.0, q = 0.0, p = 0.0;
    for (int i = lane; i < n; i += 32) {
        const double v = V[(size_t)c * n + i];
        sy += Rc[(size_t)c * n + i] * a[i];
        q += v * v;
        p += cvec[i] * v;
    }
    sy = warp_sum(sy);
    q = warp_sum(q);
    p = warp_sum(p);
    if (lane == 0) {
        const double yh = mu + sy;
        const double s2 = sigma2 * (1.0 - q + (1.0 - p) * (1.0 - p) / one_Ri_1);
        const double s = s2 > 0.0 ? sqrt(s2) : 0.0;
        double e;
        if (s > 0.0) {
            const double z = (f_min - yh) / s;
            e = (f_min - yh) * 0.5 * (1.0 + erf(z * 0.70710678118654752)) +
                s * exp(-0.5 * z * z) * 0.39894228040143268;
        } else {
            e = fmax(f_min - yh, 0.0);
        }
        if (yhat) yhat[c] = yh;
        if (s_out) s_out[c] = s;
        if (ei) ei[c] = e;
    }
}

}  // namespace
}  // namespace bpm

using namespace bpm;

namespace {

template <typename T>
int upload(T* d, const T* h, size_t count, cudaStream_t s) {
    BPM_CK(cudaMemcpyAsync(d, h, count * sizeof(T), cudaMemcpyHostToDevice, s));
    return BPM_OK;
}

int check_design(const double* X, const double* y, int n, int d) {
    if (!X || !y || n < 2 || n > kGpMaxN || d < 1 || d > kGpMaxD) {
        set_error("kriging data: 2 <= n <= %d training designs, 1 <= d <= %d parameters", kGpMaxN, kGpMaxD);
        return BPM_ERR_ARG;
    }
    return BPM_OK;
}

int gp_of(bpm_ctx* ctx, int id, Gp** out) {
    if (!ctx || id < 0 || id >= (int)ctx->gps.size() || !ctx->gps[id]) {
        set_error("unknown kriging model %d", id);
        return BPM_ERR_ARG;
    }
    *out = ctx->gps[id];
    return BPM_OK;
}

}  // namespace

extern "C" int bpm_lhs_maximin(bpm_ctx* ctx, const double* cands, int32_t T, int32_t n, int32_t d, int32_t* best,
                               double* min_d2) {
    if (!ctx || !cands || !best || T < 1 || n < 2 || d < 1) {
        set_error("bad Latin hypercube arguments");
        return BPM_ERR_ARG;
    }
    BPM_CK(cudaSetDevice(ctx->device));
    cudaStream_t s = ctx->stream;
    CallBuffers sc(ctx);
    double *dC = nullptr, *dD = nullptr;
    sc.take(&dC, (size_t)T * n * d);
    sc.take(&dD, T);
    BPM_TRY(sc.reserve());
    BPM_TRY(upload(dC, cands, (size_t)T * n * d, s));
    k_lhs_min_d2<<<T, kGpThreads, 0, s>>>(dC, n, d, dD);
    BPM_CK(cudaGetLastError());
    std::vector<double> h(T);
    BPM_CK(cudaMemcpyAsync(h.data(), dD, T * sizeof(double), cudaMemcpyDeviceToHost, s));
    BPM_CK(cudaStreamSynchronize(s));
    int b = 0;
    for (int t = 1; t < T; ++t)
        if (h[t] > h[b]) b = t;
    *best = b;
    if (min_d2) std::copy(h.begin(), h.end(), min_d2);
    return BPM_OK;
}

extern "C" int bpm_gp_nll(bpm_ctx* ctx, const double* X, const double* y, int32_t n, int32_t d,
                          const double* theta, int32_t T, double nugget, double* nll) {
    if (!ctx || !theta || !nll || T < 1 || !(nugget >= 0)) {
        set_error("bad likelihood arguments");
        return BPM_ERR_ARG;
    }
    BPM_TRY(check_design(X, y, n, d));
    BPM_CK(cudaSetDevice(ctx->device));
    cudaStream_t s = ctx->stream;
    // theta vectors per launch: their factors together stay under 1 GiB
    const int chunk = (int)std::max<size_t>(1, std::min<size_t>(T, (size_t(1) << 30) / (8 * ((size_t)(n + 2) * n + diag_doubles(n)))));
    CallBuffers sc(ctx);
    double *dX = nullptr, *dy = nullptr, *dth = nullptr, *A = nullptr, *D = nullptr, *dn = nullptr;
    int* fail = nullptr;
    sc.take(&dX, (size_t)n * d);
    sc.take(&dy, n);
    sc.take(&dth, (size_t)T * d);
    sc.take(&A, (size_t)chunk * (n + 2) * n);
    sc.take(&D, (size_t)chunk * diag_doubles(n));
    sc.take(&fail, chunk);
    sc.take(&dn, T);
    BPM_TRY(sc.reserve());
    BPM_TRY(upload(dX, X, (size_t)n * d, s));
    BPM_TRY(upload(dy, y, n, s));
    BPM_TRY(upload(dth, theta, (size_t)T * d, s));
    for (int t0 = 0; t0 < T; t0 += chunk)
        BPM_TRY(gp_factor(s, dX, dy, n, d, dth + (size_t)t0 * d, std::min(chunk, T - t0), nugget, A, D, fail,
                          dn + t0, nullptr));
    BPM_CK(cudaMemcpyAsync(nll, dn, T * sizeof(double), cudaMemcpyDeviceToHost, s));
    BPM_CK(cudaStreamSynchronize(s));
    return BPM_OK;
}

extern "C" int bpm_gp_create(bpm_ctx* ctx, const double* X, const double* y, int32_t n, int32_t d,
                             const double* theta, double nugget, int32_t* gp_id, double* mu_sigma2) {
    if (!ctx || !theta || !gp_id || !(nugget >= 0)) {
        set_error("bad kriging fit arguments");
        return BPM_ERR_ARG;
    }
    BPM_TRY(check_design(X, y, n, d));
    BPM_CK(cudaSetDevice(ctx->device));
    cudaStream_t s = ctx->stream;
    CallBuffers sc(ctx);
    double *dy = nullptr, *A = nullptr, *D = nullptr, *dn = nullptr, *st = nullptr, *u = nullptr;
    int* dfail = nullptr;
    Gp* g = new Gp();
    g->n = n;
    g->d = d;
    auto fail = [&](int r) {
        free_gp(g);
        return r;
    };
    int r = BPM_OK;
    sc.take(&dy, n);
    sc.take(&A, (size_t)(n + 2) * n);
    sc.take(&D, diag_doubles(n));
    sc.take(&dn, 1);
    sc.take(&st, 3);
    sc.take(&u, n);
    sc.take(&dfail, 1);
    if ((r = sc.reserve()) || (r = upload(dy, y, n, s))) return fail(r);
    cudaError_t e = cudaMalloc(&g->X, (size_t)n * d * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&g->theta, d * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&g->Linv, (size_t)n * n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&g->a, n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&g->c, n * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpyAsync(g->X, X, (size_t)n * d * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(g->theta, theta, d * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) {
        set_error("kriging model buffers: %s", cudaGetErrorString(e));
        return fail(BPM_ERR_OOM);
    }
    if ((r = gp_factor(s, g->X, dy, n, d, g->theta, 1, nugget, A, D, dfail, dn, st))) return fail(r);
    double hst[3] = {0, 0, 0}, hn = 0;
    e = cudaMemcpyAsync(hst, st, sizeof(hst), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hn, dn, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        set_error("kriging factor: %s", cudaGetErrorString(e));
        return fail(BPM_ERR_CUDA);
    }
    if (!std::isfinite(hn)) {
        set_error("correlation matrix is not positive definite at this theta and nugget");
        return fail(BPM_ERR_NONFINITE);
    }
    g->mu = hst[0];
    g->sigma2 = hst[1];
    g->one_Ri_1 = hst[2];
    const int nb = (n + 127) / 128;
    for (int i0 = 0; i0 < n; i0 += kPB)
        k_gp_linv<<<(n + kPB - 1) / kPB, kGpThreads, 0, s>>>(A, D, n, i0, g->Linv);
    k_gp_rows<<<nb, 128, 0, s>>>(g->Linv, dy, g->mu, n, u, g->c);
    k_gp_cols<<<nb, 128, 0, s>>>(g->Linv, u, n, g->a);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        set_error("kriging fit: %s", cudaGetErrorString(e));
        return fail(BPM_ERR_CUDA);
    }
    ctx->gps.push_back(g);
    *gp_id = (int32_t)ctx->gps.size() - 1;
    if (mu_sigma2) {
        mu_sigma2[0] = g->mu;
        mu_sigma2[1] = g->sigma2;
    }
    return BPM_OK;
}

extern "C" int bpm_gp_predict(bpm_ctx* ctx, int32_t gp_id, const double* C, int64_t N, double f_min, double* yhat,
                              double* s_out, double* ei) {
    Gp* g = nullptr;
    BPM_TRY(gp_of(ctx, gp_id, &g));
    if (!C || N < 0) {
        set_error("bad prediction arguments");
        return BPM_ERR_ARG;
    }
    if (N == 0) return BPM_OK;
    BPM_CK(cudaSetDevice(ctx->device));
    cudaStream_t s = ctx->stream;
    const int n = g->n, d = g->d;
    const int chunk = (int)std::min<int64_t>(N, 32768);
    CallBuffers sc(ctx);
    double *dC = nullptr, *Rc = nullptr, *V = nullptr, *dy = nullptr, *ds = nullptr, *de = nullptr;
    sc.take(&dC, (size_t)chunk * d);
    sc.take(&Rc, (size_t)chunk * n);
    sc.take(&V, (size_t)chunk * n);
    sc.take(&dy, chunk);
    sc.take(&ds, chunk);
    sc.take(&de, chunk);
    BPM_TRY(sc.reserve());
    for (int64_t c0 = 0; c0 < N; c0 += chunk) {
        const int m = (int)std::min<int64_t>(chunk, N - c0);
        BPM_CK(cudaMemcpyAsync(dC, C + c0 * d, (size_t)m * d * sizeof(double), cudaMemcpyHostToDevice, s));
        const long long cells = (long long)m * n;
        k_gp_corr<<<(unsigned)((cells + 255) / 256), 256, 0, s>>>(dC, g->X, g->theta, m, n, d, Rc);
        k_gp_gemm_nt<<<dim3((n + kTN - 1) / kTN, (m + kTM - 1) / kTM), 256, 0, s>>>(Rc, g->Linv, m, n, n, V);
        k_gp_ei<<<(m + 7) / 8, 256, 0, s>>>(Rc, V, g->a, g->c, m, n, g->mu, g->sigma2, g->one_Ri_1, f_min, dy, ds,
                                             de);
        BPM_CK(cudaGetLastError());
        if (yhat) BPM_CK(cudaMemcpyAsync(yhat + c0, dy, m * sizeof(double), cudaMemcpyDeviceToHost, s));
        if (s_out) BPM_CK(cudaMemcpyAsync(s_out + c0, ds, m * sizeof(double), cudaMemcpyDeviceToHost, s));
        if (ei) BPM_CK(cudaMemcpyAsync(ei + c0, de, m * sizeof(double), cudaMemcpyDeviceToHost, s));
        BPM_CK(cudaStreamSynchronize(s));
    }
    return BPM_OK;
}

extern "C" int bpm_gp_destroy(bpm_ctx* ctx, int32_t gp_id) {
    Gp* g = nullptr;
    BPM_TRY(gp_of(ctx, gp_id, &g));
    cudaSetDevice(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    free_gp(g);
    ctx->gps[gp_id] = nullptr;
    return BPM_OK;
}
