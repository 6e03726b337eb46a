// One-time FP64 assembly of an island's operators on the GPU.
//
// P1 tetrahedral FEM (Sec. II.A: finite-element micromagnetics of the island;
// the discretisation itself is the textbook one): lumped nodal volumes, nodal
// Ms/Ku, the exchange stiffness K_ij = sum_t A_t vol_t grad(phi_i).grad(phi_j)
// and the exchange operator S = 2 K / (Ms V).  Demagnetising field by the
// hybrid FEM/BEM method (Sec. II.A) in the Fredkin-Koehler form:
//   u1: Neumann Poisson problem with source div(M) (zero-mean gauge),
//   u2 = (D + diag(Omega/4pi - 1)) u1 on the boundary, D the double-layer
//        matrix of Lindholm's closed-form weights for linear densities,
//   u2 harmonic inside (Dirichlet problem),
//   H = -grad(u1 + u2) per tet, lumped to the nodes.
// The map M -> H is formed as a matrix.  Its source div(M) and its gradient are
// sparse, so the solves are done for the n nodal sources rather than for the
// 3n magnetisation components: G = K^+ (Neumann; a null vector per body of the
// mesh), the harmonic extension E of the boundary values (Dirichlet),
// Q = G + E (D + diag(..)) G_boundary, and N = P Q R with the sparse R (source)
// and P (projected gradient).  Both solves
// run as Jacobi-preconditioned CG over row-major blocks of right-hand sides: a
// CTA owns one or two columns and runs their iterations in shared memory, with
// reductions in a fixed order so that results are bit-reproducible.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>

#include "bpm_internal.cuh"

namespace bpm {

namespace {

// buffers of one assembly; zeroing and uploads are ordered on its stream
struct DevPool {
    cudaStream_t st = nullptr;
    std::vector<void*> ptrs;
    explicit DevPool(cudaStream_t s) : st(s) {}
    ~DevPool() {
        for (void* p : ptrs) cudaFree(p);
    }
    template <class T>
    int alloc(T** p, size_t count, bool zero = true) {
        void* q = nullptr;
        if (count == 0) count = 1;
        cudaError_t e = cudaMalloc(&q, count * sizeof(T));
        if (e != cudaSuccess) {
            set_error("device allocation of %zu bytes failed: %s", count * sizeof(T),
                      cudaGetErrorString(e));
            return BPM_ERR_OOM;
        }
        ptrs.push_back(q);
        if (zero) {
            e = cudaMemsetAsync(q, 0, count * sizeof(T), st);
            if (e != cudaSuccess) {
                set_error("cudaMemsetAsync failed: %s", cudaGetErrorString(e));
                return BPM_ERR_CUDA;
            }
        }
        *p = static_cast<T*>(q);
        return BPM_OK;
    }
};

// A stream forked from `main` at fork() and joined into it by join().  Left on an early return it is
// drained before its stream goes, so that its kernels never outlive the buffers they use (declare it
// after the pool that owns them).
struct SideStream {
    cudaStream_t s = nullptr;
    cudaEvent_t e = nullptr;
    int fork(cudaStream_t main) {
        BPM_CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
        BPM_CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        BPM_CK(cudaEventRecord(e, main));
        BPM_CK(cudaStreamWaitEvent(s, e, 0));
        return BPM_OK;
    }
    int join(cudaStream_t main) {
        BPM_CK(cudaEventRecord(e, s));
        BPM_CK(cudaStreamWaitEvent(main, e, 0));
        return BPM_OK;
    }
    ~SideStream() {
        if (s) {
            cudaStreamSynchronize(s);
            cudaStreamDestroy(s);
        }
        if (e) cudaEventDestroy(e);
    }
};

template <class T>
int upload(DevPool& pool, T** dst, const std::vector<T>& src) {
    BPM_TRY(pool.alloc(dst, src.size(), false));
    BPM_CK(cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, pool.st));
    return BPM_OK;
}

// ---------------------------------------------------------------- vectors
struct V3 {
    double x, y, z;
};
__host__ __device__ inline V3 mk(double x, double y, double z) { return V3{x, y, z}; }
__host__ __device__ inline V3 sub(V3 a, V3 b) { return mk(a.x - b.x, a.y - b.y, a.z - b.z); }
__host__ __device__ inline V3 add(V3 a, V3 b) { return mk(a.x + b.x, a.y + b.y, a.z + b.z); }
__host__ __device__ inline V3 scl(V3 a, double s) { return mk(a.x * s, a.y * s, a.z * s); }
__host__ __device__ inline double dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__host__ __device__ inline V3 cross(V3 a, V3 b) {
    return mk(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__host__ __device__ inline double nrm(V3 a) { return sqrt(dot(a, a)); }
__host__ __device__ inline V3 ld3(const double* p) { return mk(p[0], p[1], p[2]); }

// ---------------------------------------------------------------- FEM kernels
__global__ void k_tet_geom(int nt, const double* __restrict__ xyz, const int* __restrict__ tets,
                           double* __restrict__ vol, double* __restrict__ grads) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    V3 x0 = ld3(xyz + 3 * tets[4 * t + 0]);
    V3 e1 = sub(ld3(xyz + 3 * tets[4 * t + 1]), x0);
    V3 e2 = sub(ld3(xyz + 3 * tets[4 * t + 2]), x0);
    V3 e3 = sub(ld3(xyz + 3 * tets[4 * t + 3]), x0);
    V3 c23 = cross(e2, e3), c31 = cross(e3, e1), c12 = cross(e1, e2);
    double det = dot(e1, c23);
    // rows of J^{-1} (J = [e1 e2 e3]) are the gradients of phi_1..phi_3
    V3 g1 = scl(c23, 1.0 / det), g2 = scl(c31, 1.0 / det), g3 = scl(c12, 1.0 / det);
    V3 g0 = scl(add(add(g1, g2), g3), -1.0);
    vol[t] = fabs(det) / 6.0;
    double* g = grads + 12 * t;
    V3 gs[4] = {g0, g1, g2, g3};
    for (int a = 0; a < 4; ++a) {
        g[3 * a + 0] = gs[a].x;
        g[3 * a + 1] = gs[a].y;
        g[3 * a + 2] = gs[a].z;
    }
}

// position of a node in a tet, -1 if the tet does not hold it
__device__ inline int tet_slot(const int* tet, int node) {
    for (int a = 0; a < 4; ++a)
        if (tet[a] == node) return a;
    return -1;
}

__global__ void k_node_lumped(int n, const int* __restrict__ n2t_ptr, const int* __restrict__ n2t,
                              const int* __restrict__ region, const double* __restrict__ vol,
                              const double* __restrict__ mat_Ms, const double* __restrict__ mat_Ku,
                              double* __restrict__ V, double* __restrict__ Ms, double* __restrict__ Ku) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = 0, ms = 0, ku = 0;
    for (int e = n2t_ptr[i]; e < n2t_ptr[i + 1]; ++e) {
        int t = n2t[e];
        double q = 0.25 * vol[t];
        v += q;
        ms += q * mat_Ms[region[t]];
        ku += q * mat_Ku[region[t]];
    }
    V[i] = v;
    Ms[i] = ms / v;
    Ku[i] = ku / v;
}

// One warp per row, a lane per CSR entry (i, j): the lane walks the tets around i in order and
// adds those that hold j, so every entry is summed in the same order as a serial loop over the
// row would.  (One thread per row: 197 us at 481 nodes, two CTAs' worth of threads; now 24 us.)
__global__ void k_csr_values(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                             const int* __restrict__ n2t_ptr, const int* __restrict__ n2t,
                             const int* __restrict__ tets, const int* __restrict__ region,
                             const double* __restrict__ mat_A, const double* __restrict__ vol,
                             const double* __restrict__ grads, double* __restrict__ KA,
                             double* __restrict__ KL) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= n) return;
    for (int pos = rowptr[i] + lane; pos < rowptr[i + 1]; pos += 32) {
        const int j = col[pos];
        double kl = 0, ka = 0;
        for (int e = n2t_ptr[i]; e < n2t_ptr[i + 1]; ++e) {
            const int t = n2t[e];
            const int* tt = tets + 4 * t;
            const int b = tet_slot(tt, j);
            if (b < 0) continue;
            const int a = tet_slot(tt, i);
            const double* g = grads + 12 * t;
            const double gg = g[3 * a] * g[3 * b] + g[3 * a + 1] * g[3 * b + 1] + g[3 * a + 2] * g[3 * b + 2];
            kl += vol[t] * gg;
            ka += mat_A[region[t]] * vol[t] * gg;
        }
        KL[pos] = kl;
        KA[pos] = ka;
    }
}

// exchange operator, difference form: c_ij = -2e18 K_A,ij / (Ms_i V_i) for j != i
// (nm -> m: K carries 1e-9, V carries 1e-27)
__global__ void k_exchange_values(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                                  const double* __restrict__ KA, const double* __restrict__ V,
                                  const double* __restrict__ Ms, float* __restrict__ c) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = -2.0e18 / (Ms[i] * V[i]);
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) c[e] = (col[e] == i) ? 0.f : (float)(s * KA[e]);
}

// the same values in FP64, kept for the plain FP64 form
__global__ void k_exchange_values64(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                                    const double* __restrict__ KA, const double* __restrict__ V,
                                    const double* __restrict__ Ms, double* __restrict__ c) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = -2.0e18 / (Ms[i] * V[i]);
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) c[e] = (col[e] == i) ? 0.0 : s * KA[e];
}

__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double s = 0;
    int nw = blockDim.x >> 5;
    for (int k = 0; k < nw; ++k) s += red[k];
    return s;
}

// A CSR matrix in slices of 32 rows (diagonal included): entry e of row 32 s + l sits at
// off[s] + 32 e + l, so that a warp reads a slice's values and columns coalesced; padding
// entries hold the row itself (or node 0) with the value 0.
struct Sliced {
    const int* off;      // [n_slices + 1]
    const int* col;      // node of the entry
    const int* src;      // its CSR entry, -1 for padding
    int len;
};

// sliced values of a CSR matrix; with d: d_i v_ij d_j; with mask: rows and columns outside it zero
__global__ void k_sliced_values(Sliced A, const int* __restrict__ rows, const double* __restrict__ v,
                                const double* __restrict__ d, const unsigned char* __restrict__ mask,
                                double* __restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= A.len) return;
    const int e = A.src[k], i = rows[k], j = A.col[k];
    double x = e >= 0 ? v[e] : 0.0;
    if (d) x *= d[i] * d[j];
    if (mask && !(mask[i] && mask[j])) x = 0.0;
    out[k] = x;
}

__global__ void k_exchange_scale(int n, const double* __restrict__ V, const double* __restrict__ Ms,
                                 double* __restrict__ d) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) d[i] = sqrt(2.0e18 / (Ms[i] * V[i]));
}

// K_ii^-1/2 of every node, and the same with zeros off the interior
__global__ void k_diag_scale(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                             const double* __restrict__ K, const unsigned char* __restrict__ interior,
                             double* __restrict__ d, double* __restrict__ d_in) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double kii = 0;
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e)
        if (col[e] == i) kii = K[e];
    d[i] = 1.0 / sqrt(kii);
    d_in[i] = interior[i] ? d[i] : 0.0;
}

__device__ __forceinline__ double sliced_row(const Sliced& A, const double* __restrict__ val, const double* x, int i) {
    const int lo = A.off[i >> 5] + (i & 31), hi = A.off[(i >> 5) + 1];
    double s = 0;
#pragma unroll 4
    for (int k = lo; k < hi; k += 32) s += val[k] * x[A.col[k]];
    return s;
}

// Largest eigenvalue of S = D K_A (D = 2e18/(Ms V)) by power iteration on the similar symmetric
// matrix D^1/2 K_A D^1/2 (sliced values in `val`), Rayleigh quotient of the last iterate.  A cluster
// of 8 CTAs holds both vectors in every CTA's shared memory; a CTA forms an eighth of
// the rows, four lanes a row, and writes them to all eight copies, with one cluster barrier per iteration.  Every CTA
// normalises its own copy every 8 steps (the direction does not depend on when).  An SM does two
// FP64 multiply-adds a cycle, so one CTA alone was bound by them: 5.9 ms for 1500 steps at 481 nodes,
// 3.4 ms with the cluster, and it runs beside the demag assembly.  (With square roots and divisions
// formed per entry, rows read uncoalesced and three reductions a step: 116 ms.)
constexpr int kPowCluster = 8, kPowThreads = 512;

__global__ void __cluster_dims__(kPowCluster, 1, 1) __launch_bounds__(kPowThreads)
    k_power_iteration(int n, Sliced A, const double* __restrict__ val, int iters, double* __restrict__ lam_out) {
    namespace cgr = cooperative_groups;
    extern __shared__ double vec[];
    __shared__ double red[32];
    cgr::cluster_group cl = cgr::this_cluster();
    const int rank = (int)cl.block_rank();
    const int n_slices = (n + 31) / 32, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *x = vec, *y = vec + n;
    for (int i = threadIdx.x; i < n; i += kPowThreads) x[i] = ((i & 1) ? 1.0 : -1.0) + 0.3 * sin(0.7 * i);
    cl.sync();
    for (int it = 1; it < iters; ++it) {
        // a warp takes 8 rows of a slice, four lanes a row; each lane sends the sum to two CTAs
        for (int u = rank + kPowCluster * warp; u < 4 * n_slices; u += kPowCluster * (kPowThreads / 32)) {
            const int i = 8 * u + (lane & 7), part = lane >> 3;
            double v = 0;
            if (i < n) {
                const int hi = A.off[(i >> 5) + 1];
#pragma unroll 2
                for (int k = A.off[i >> 5] + (i & 31) + 32 * part; k < hi; k += 128) v += val[k] * x[A.col[k]];
            }
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            if (i < n) {
                cl.map_shared_rank(y, 2 * part)[i] = v;
                cl.map_shared_rank(y, 2 * part + 1)[i] = v;
            }
        }
        cl.sync();
        double* t = x;
        x = y;
        y = t;
        if ((it & 7) == 0) {
            double nn = 0;
            for (int i = threadIdx.x; i < n; i += kPowThreads) nn += x[i] * x[i];
            const double inv = 1.0 / sqrt(block_sum(nn, red));
            for (int i = threadIdx.x; i < n; i += kPowThreads) x[i] *= inv;
            __syncthreads();
        }
    }
    double xy = 0, xx = 0;
    if (rank == 0) {
        for (int i = threadIdx.x; i < n; i += kPowThreads) {
            xy += x[i] * sliced_row(A, val, x, i);
            xx += x[i] * x[i];
        }
        xy = block_sum(xy, red);
        xx = block_sum(xx, red);
        if (threadIdx.x == 0) *lam_out = xy / xx;
    }
}

// (R M)_j = int M . grad(phi_j) for nodal P1 M, by columns: RT[c][pos] = R[j][c n + k] for CSR entry
// pos = (k, j).  A lane per entry, tets in order, as in k_csr_values.
__global__ void k_source(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                         const int* __restrict__ n2t_ptr, const int* __restrict__ n2t,
                         const int* __restrict__ tets, const double* __restrict__ vol,
                         const double* __restrict__ grads, int nnz, double* __restrict__ RT) {
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (k >= n) return;
    for (int pos = rowptr[k] + lane; pos < rowptr[k + 1]; pos += 32) {
        const int j = col[pos];
        double s[3] = {0, 0, 0};
        for (int e = n2t_ptr[k]; e < n2t_ptr[k + 1]; ++e) {
            const int t = n2t[e];
            const int a = tet_slot(tets + 4 * t, j);
            if (a < 0) continue;
            const double* g = grads + 12 * t;
            const double q = 0.25 * vol[t];
            for (int c = 0; c < 3; ++c) s[c] += q * g[3 * a + c];
        }
        for (int c = 0; c < 3; ++c) RT[(size_t)c * nnz + pos] = s[c];
    }
}

// U = Q R: U[i][c n + k] = sum over the neighbours j of k of Q[i][j] R[j][c n + k] (RT sliced: rv[c][entry])
__global__ void k_apply_source(int n, Sliced A, const double* __restrict__ rv, const double* __restrict__ Q,
                               double* __restrict__ U) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (k >= n) return;
    const double* q = Q + (size_t)i * n;
    double s0 = 0, s1 = 0, s2 = 0;
    const int lo = A.off[k >> 5] + (k & 31), hi = A.off[(k >> 5) + 1];
#pragma unroll 4
    for (int e = lo; e < hi; e += 32) {
        const double v = q[A.col[e]];
        s0 += v * rv[e];
        s1 += v * rv[A.len + e];
        s2 += v * rv[2 * (size_t)A.len + e];
    }
    double* u = U + (size_t)i * 3 * n + k;
    u[0] = s0;
    u[n] = s1;
    u[2 * (size_t)n] = s2;
}

// right-hand sides of the nodal sources of the Neumann problem: e_j less its mean over the body that holds
// j (body: per node; ptr: first node of each body in an order by bodies).  The Laplacian has a null vector
// per body of the mesh, so a source has to sum to zero over each; div M does, and its potential's constant
// on a body drops out of u1 + u2.
__global__ void k_unit_sources(int n, const int* __restrict__ body, const int* __restrict__ ptr,
                               double* __restrict__ B) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (j >= n) return;
    const int p = body[i];
    B[(size_t)i * n + j] = (i == j ? 1.0 : 0.0) - (body[j] == p ? 1.0 / (ptr[p + 1] - ptr[p]) : 0.0);
}

// right-hand sides -K_IB of the harmonic extension (interior rows; B zeroed before)
__global__ void k_boundary_sources(int n, int nb, const int* __restrict__ rowptr, const int* __restrict__ col,
                                   const double* __restrict__ K, const unsigned char* __restrict__ interior,
                                   const int* __restrict__ bidx, double* __restrict__ B) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= n || !interior[i]) return;
    for (int e = rowptr[i] + lane; e < rowptr[i + 1]; e += 32)
        if (!interior[col[e]]) B[(size_t)i * nb + bidx[col[e]]] = -K[e];
}

// the extension on the boundary itself is the identity
__global__ void k_boundary_identity(int nb, const int* __restrict__ bnodes, double* __restrict__ E) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nb) E[(size_t)bnodes[b] * nb + b] = 1.0;
}

// ---------------------------------------------------------------- batched CG
// kCgSteps iterations of CG on C columns of the right-hand side block, one CTA: p, q and r of its
// columns in shared memory ([n][C]), x in global memory (each thread its own rows).  The matrix is
// scaled to a unit diagonal (d K d, d = K_ii^-1/2: Jacobi preconditioning); b and x are scaled on the
// way in and out.  The columns are independent, so an iteration needs
// no grid-wide step.  The matrix (sliced, 12 B an entry) comes from L1/L2, once for the C columns.
// The bound is the FP64 rate, two multiply-adds a cycle and SM: about 25 per node, column and
// iteration.  Hence one warp adds up the CTA's partial sums and divides (all threads doing so cost a
// third of the iteration), while the others update x.  Measured at 481 nodes, 481 columns: 20 us an
// iteration (28 us with all threads reducing and two columns a CTA; one kernel per vector operation
// with one thread per column in the dot products took 330 us for the 1443 columns of 3n sources).
constexpr int kCgThreads = 256, kCgSteps = 16;

// sum over the CTA of C values per thread: partial sums to shared memory, warp 0 adds them
template <int C>
__device__ __forceinline__ void put_partial(const double (&v)[C], double* part) {
#pragma unroll
    for (int c = 0; c < C; ++c) part[c * kCgThreads + threadIdx.x] = v[c];
}
template <int C>
__device__ __forceinline__ void warp_total(const double* part, double (&v)[C]) {
#pragma unroll
    for (int c = 0; c < C; ++c) {
        double s = 0;
        for (int k = threadIdx.x; k < kCgThreads; k += 32) s += part[c * kCgThreads + k];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        v[c] = s;
    }
}

template <int C>
__global__ void __launch_bounds__(kCgThreads) k_cg_steps(int n, int ncol, Sliced A, const double* __restrict__ val,
                                                         const double* __restrict__ d,
                                                         const double* __restrict__ b, int first,
                                                         double* __restrict__ x, double* __restrict__ rg,
                                                         double* __restrict__ pg, double* __restrict__ rzg,
                                                         double* __restrict__ bbg, double* __restrict__ rrg) {
    extern __shared__ double cg[];
    __shared__ double part[kCgThreads * C], coef[C], rz_s[C], floor_s[C];
    double *p = cg, *q = cg + (size_t)n * C, *r = q + (size_t)n * C;
    const int c0 = blockIdx.x * C;
    double v[C], s[C];
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = s[c] = 0;
    for (int i = threadIdx.x; i < n; i += kCgThreads) {
        const double di = d[i];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const bool in = c0 + c < ncol;
            const size_t k = (size_t)i * ncol + c0 + c;
            const double bv = in && first ? b[k] : 0.0;
            const double rv = first ? di * bv : (in ? rg[k] : 0.0);
            r[i * C + c] = rv;
            p[i * C + c] = first ? rv : (in ? pg[k] : 0.0);
            if (first) {
                if (in) x[k] = 0.0;
                v[c] += rv * rv;
                s[c] += bv * bv;
            }
        }
    }
    // a column at rounding level stays where it is: steps beyond it would only follow the null space
    // of the Neumann problem (a mesh of a few dozen nodes is there before the first check)
    put_partial<C>(v, part);
    __syncthreads();
    if (threadIdx.x < 32) {
        warp_total<C>(part, v);
        if (threadIdx.x == 0)
            for (int c = 0; c < C; ++c) {
                const bool in = c0 + c < ncol;
                if (in && first) rzg[ncol + c0 + c] = v[c];
                rz_s[c] = first ? v[c] : (in ? rzg[c0 + c] : 0.0);
                floor_s[c] = 1e-31 * (first ? v[c] : (in ? rzg[ncol + c0 + c] : 0.0));
            }
    }
    if (first) {
        __syncthreads();
        put_partial<C>(s, part);
        __syncthreads();
        if (threadIdx.x < 32) {
            warp_total<C>(part, s);
            if (threadIdx.x == 0)
                for (int c = 0; c < C && c0 + c < ncol; ++c) bbg[c0 + c] = s[c];
        }
    }
    for (int it = 0; it < kCgSteps; ++it) {
        __syncthreads();                                   // p of every row is in place
        double pq[C], rr[C];
#pragma unroll
        for (int c = 0; c < C; ++c) pq[c] = rr[c] = 0;
        for (int i = threadIdx.x; i < n; i += kCgThreads) {
            const int lo = A.off[i >> 5] + (i & 31), hi = A.off[(i >> 5) + 1];
            double t[C];
#pragma unroll
            for (int c = 0; c < C; ++c) t[c] = 0;
#pragma unroll 4
            for (int k = lo; k < hi; k += 32) {
                const double a = val[k];
                const double* pj = p + A.col[k] * C;
#pragma unroll
                for (int c = 0; c < C; ++c) t[c] += a * pj[c];
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {
                q[i * C + c] = t[c];
                pq[c] += p[i * C + c] * t[c];
            }
        }
        put_partial<C>(pq, part);
        __syncthreads();
        if (threadIdx.x < 32) {
            warp_total<C>(part, pq);
            if (threadIdx.x == 0)
                for (int c = 0; c < C; ++c) coef[c] = pq[c] > 0 && rz_s[c] > floor_s[c] ? rz_s[c] / pq[c] : 0.0;
        }
        __syncthreads();
        double a[C];
#pragma unroll
        for (int c = 0; c < C; ++c) a[c] = coef[c];
        for (int i = threadIdx.x; i < n; i += kCgThreads)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const double rv = r[i * C + c] - a[c] * q[i * C + c];
                r[i * C + c] = rv;
                rr[c] += rv * rv;
            }
        put_partial<C>(rr, part);
        __syncthreads();
        if (threadIdx.x < 32) {
            warp_total<C>(part, rr);
            if (threadIdx.x == 0)
                for (int c = 0; c < C; ++c) {
                    coef[c] = rz_s[c] > 0 ? rr[c] / rz_s[c] : 0.0;
                    rz_s[c] = rr[c];
                }
        }
        for (int i = threadIdx.x; i < n; i += kCgThreads)
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (c0 + c < ncol) x[(size_t)i * ncol + c0 + c] += a[c] * p[i * C + c];
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += kCgThreads)
#pragma unroll
            for (int c = 0; c < C; ++c) p[i * C + c] = r[i * C + c] + coef[c] * p[i * C + c];
    }
#pragma unroll
    for (int c = 0; c < C; ++c) s[c] = 0;
    for (int i = threadIdx.x; i < n; i += kCgThreads) {
        const double di = d[i];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const double rv = r[i * C + c], u = di > 0 ? rv / di : 0.0;
            s[c] += u * u;
            if (c0 + c < ncol) {
                rg[(size_t)i * ncol + c0 + c] = rv;
                pg[(size_t)i * ncol + c0 + c] = p[i * C + c];
            }
        }
    }
    __syncthreads();
    put_partial<C>(s, part);
    __syncthreads();
    if (threadIdx.x < 32) {
        warp_total<C>(part, s);
        if (threadIdx.x == 0)
            for (int c = 0; c < C && c0 + c < ncol; ++c) {
                rrg[c0 + c] = s[c];
                rzg[c0 + c] = rz_s[c];
            }
    }
}

// x = d x', out of the scaled system
__global__ void k_scale_rows(int ncol, const double* __restrict__ d, double* __restrict__ X) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (c < ncol) X[(size_t)i * ncol + c] *= d[i];
}

__global__ void k_max_ratio(int ncol, const double* __restrict__ rr, const double* __restrict__ bb,
                            double* __restrict__ out) {
    __shared__ double red[32];
    double m = 0;
    for (int c = threadIdx.x; c < ncol; c += blockDim.x) {
        double v = bb[c] > 0 ? sqrt(rr[c] / bb[c]) : 0.0;
        if (!(v == v)) v = 1e300;  // NaN propagates as "not converged"
        m = fmax(m, v);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s = fmax(s, red[k]);
        *out = s;
    }
}

// subtract each column's mean over a body's rows (rows of all bodies, by body): 32 columns of a body a CTA, 8
// warps over the rows, partial sums in a fixed order
__global__ void __launch_bounds__(256) k_col_mean_sub(const int* __restrict__ rows, const int* __restrict__ ptr,
                                                      int ncol, double* __restrict__ X) {
    __shared__ double part[8][32];
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + l;
    const int lo = ptr[blockIdx.y], hi = ptr[blockIdx.y + 1];
    double s = 0;
    if (c < ncol)
        for (int i = lo + w; i < hi; i += 8) s += X[(size_t)rows[i] * ncol + c];
    part[w][l] = s;
    __syncthreads();
    s = 0;
    for (int k = 0; k < 8; ++k) s += part[k][l];
    s /= hi - lo;
    if (c < ncol)
        for (int i = lo + w; i < hi; i += 8) X[(size_t)rows[i] * ncol + c] -= s;
}

template <int C>
int cg_launch(cudaStream_t st, int n, int ncol, const Sliced& A, const double* val, const double* d,
              const double* b, int first, double* x, double* r, double* p, double* rz, double* bb, double* rr) {
    const int smem = 3 * (int)sizeof(double) * n * C;
    BPM_CK(cudaFuncSetAttribute(k_cg_steps<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    k_cg_steps<C><<<(ncol + C - 1) / C, kCgThreads, smem, st>>>(n, ncol, A, val, d, b, first, x, r, p, rz, bb, rr);
    BPM_CK(cudaGetLastError());
    return BPM_OK;
}

int pcg(cudaStream_t st, DevPool& pool, int n, int ncol, const Sliced& A, const double* val, const double* d,
        const double* b, double* x, double tol, int maxit, int* iters_out, double* resid_out) {
    const size_t N = (size_t)n * ncol;
    double *r, *p, *rz, *bb, *rr, *mx;
    BPM_TRY(pool.alloc(&r, N, false));
    BPM_TRY(pool.alloc(&p, N, false));
    BPM_TRY(pool.alloc(&rz, 2 * (size_t)ncol));   // current and initial r . z
    BPM_TRY(pool.alloc(&bb, ncol));
    BPM_TRY(pool.alloc(&rr, ncol));
    BPM_TRY(pool.alloc(&mx, 1));
    // columns a CTA: two share the matrix loads where there are enough columns to fill the SMs either
    // way, and while three vectors of both fit shared memory (4096 nodes: 196608 B)
    const bool two = n <= 4096 && ncol >= 1024;
    double res = 1.0;
    int it = 0;
    while (it < maxit) {
        BPM_TRY(two ? cg_launch<2>(st, n, ncol, A, val, d, b, it == 0, x, r, p, rz, bb, rr)
                    : cg_launch<1>(st, n, ncol, A, val, d, b, it == 0, x, r, p, rz, bb, rr));
        it += kCgSteps;
        k_max_ratio<<<1, 1024, 0, st>>>(ncol, rr, bb, mx);
        BPM_CK(cudaGetLastError());
        BPM_CK(cudaMemcpyAsync(&res, mx, sizeof(double), cudaMemcpyDeviceToHost, st));
        BPM_CK(cudaStreamSynchronize(st));
        if (!(res < 1e300)) {
            set_error("CG produced a non-finite residual");
            return BPM_ERR_NONFINITE;
        }
        if (res < tol) break;
    }
    k_scale_rows<<<dim3((ncol + 127) / 128, n), 128, 0, st>>>(ncol, d, x);
    BPM_CK(cudaGetLastError());
    *iters_out = it;
    *resid_out = res;
    if (res >= tol) {
        set_error("CG did not converge: relative residual %.3e after %d iterations", res, maxit);
        return BPM_ERR_UNSTABLE;
    }
    return BPM_OK;
}

// ---------------------------------------------------------------- BEM
// signed solid angle of triangle (r1, r2, r3) seen from the origin (van Oosterom & Strackee)
__device__ double solid_angle(V3 r1, V3 r2, V3 r3) {
    double l1 = nrm(r1), l2 = nrm(r2), l3 = nrm(r3);
    double num = dot(r1, cross(r2, r3));
    double den = l1 * l2 * l3 + dot(r1, r2) * l3 + dot(r1, r3) * l2 + dot(r2, r3) * l1;
    return 2.0 * atan2(num, den);
}

// w_k = int_T phi_k(y) n.(y - x)/|y - x|^3 dS, Lindholm's closed form (see header of this file)
__device__ void lindholm(V3 x, const V3 y[3], double w[3]) {
    V3 rho[3], xi[3];
    double s[3], lr[3];
    for (int k = 0; k < 3; ++k) {
        rho[k] = sub(y[k], x);
        lr[k] = nrm(rho[k]);
        V3 e = sub(y[(k + 1) % 3], y[k]);
        s[k] = nrm(e);
        xi[k] = scl(e, 1.0 / s[k]);
    }
    V3 cr = cross(sub(y[1], y[0]), sub(y[2], y[0]));
    double two_area = nrm(cr);
    V3 n = scl(cr, 1.0 / two_area);
    double zeta = dot(n, rho[0]);
    double eta[3], P[3];
    for (int k = 0; k < 3; ++k) {
        eta[k] = dot(cross(n, xi[k]), rho[k]);
        double ls = lr[k] + lr[(k + 1) % 3];
        P[k] = log((ls + s[k]) / (ls - s[k]));
    }
    double om = solid_angle(rho[0], rho[1], rho[2]);
    for (int k = 0; k < 3; ++k) {
        int k1 = (k + 1) % 3;
        double gp = 0;
        for (int j = 0; j < 3; ++j) gp += dot(xi[k1], xi[j]) * P[j];
        w[k] = s[k1] / two_area * (-eta[k1] * om + zeta * gp);
    }
}

__global__ void k_interior_angles(int nb, const int* __restrict__ bnodes, const int* __restrict__ n2t_ptr,
                                  const int* __restrict__ n2t, const int* __restrict__ tets,
                                  const double* __restrict__ xyz, double* __restrict__ omega) {
    int ib = blockIdx.x * blockDim.x + threadIdx.x;
    if (ib >= nb) return;
    int i = bnodes[ib];
    V3 x = ld3(xyz + 3 * i);
    double s = 0;
    for (int e = n2t_ptr[i]; e < n2t_ptr[i + 1]; ++e) {
        const int* tt = tets + 4 * n2t[e];
        V3 r[3];
        int k = 0;
        for (int a = 0; a < 4; ++a)
            if (tt[a] != i) r[k++] = sub(ld3(xyz + 3 * tt[a]), x);
        s += fabs(solid_angle(r[0], r[1], r[2]));
    }
    omega[ib] = s;
}

// Lindholm weights of every (observer, face) pair, W[ib][3 f + k] for vertex k of face f; zero where
// the observer is a vertex of the face (it lies in the face's plane).  One evaluation gives all three
// weights of a face (evaluated per (observer, node) pair each face was computed three times and two
// of its weights dropped: 584 us at 272 boundary nodes).
__global__ void k_bem_weights(int i0, int rows, int nf, const int* __restrict__ bnodes,
                              const double* __restrict__ xyz, const int* __restrict__ faces,
                              double* __restrict__ W) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x, ib = blockIdx.y;
    if (f >= nf || ib >= rows) return;
    const int i = bnodes[i0 + ib];
    const int* fc = faces + 3 * f;
    double w[3] = {0, 0, 0};
    if (fc[0] != i && fc[1] != i && fc[2] != i) {
        const V3 y[3] = {ld3(xyz + 3 * fc[0]), ld3(xyz + 3 * fc[1]), ld3(xyz + 3 * fc[2])};
        lindholm(ld3(xyz + 3 * i), y, w);
    }
    double* o = W + ((size_t)ib * nf + f) * 3;
    o[0] = w[0];
    o[1] = w[1];
    o[2] = w[2];
}

// Bmat[ib][jb] = D_ij + delta_ij (Omega_i/4pi - 1),
// D_ij = -(1/4pi) sum over boundary faces T containing node j of w_j(x_i; T)
__global__ void k_bem_matrix(int i0, int nb, int nf, const int* __restrict__ bnodes, const int* __restrict__ faces,
                             const int* __restrict__ b2f_ptr, const int* __restrict__ b2f,
                             const double* __restrict__ omega, const double* __restrict__ W,
                             double* __restrict__ Bmat) {
    const int jb = blockIdx.x * blockDim.x + threadIdx.x, ib = i0 + blockIdx.y;
    if (jb >= nb) return;
    const int j = bnodes[jb];
    double s = 0;
    for (int e = b2f_ptr[jb]; e < b2f_ptr[jb + 1]; ++e) {
        const int* f = faces + 3 * b2f[e];
        const int loc = (f[0] == j) ? 0 : ((f[1] == j) ? 1 : 2);
        s += W[((size_t)blockIdx.y * nf + b2f[e]) * 3 + loc];
    }
    double v = -s / (4.0 * M_PI);
    if (ib == jb) v += omega[ib] / (4.0 * M_PI) - 1.0;
    Bmat[(size_t)ib * nb + jb] = v;
}

__global__ void k_gather_rows(int nb, int ncol, const int* __restrict__ rows, const double* __restrict__ src,
                              double* __restrict__ dst) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    int ib = blockIdx.y;
    if (c >= ncol) return;
    dst[(size_t)ib * ncol + c] = src[(size_t)rows[ib] * ncol + c];
}

// C[M][N] (+)= A[M][K] B[K][N] (row-major, FP64), 32x32 tiles
__global__ void k_dgemm(int M, int N, int K, const double* __restrict__ A, const double* __restrict__ B, int add,
                        double* __restrict__ C) {
    __shared__ double As[32][33], Bs[32][33];
    int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    int row0 = blockIdx.y * 32, col = blockIdx.x * 32 + tx;
    double acc[4] = {0, 0, 0, 0};
    for (int k0 = 0; k0 < K; k0 += 32) {
        for (int r = ty; r < 32; r += 8) {
            int gr = row0 + r, gk = k0 + tx;
            As[r][tx] = (gr < M && gk < K) ? A[(size_t)gr * K + gk] : 0.0;
            int bk = k0 + r;
            Bs[r][tx] = (bk < K && col < N) ? B[(size_t)bk * N + col] : 0.0;
        }
        __syncthreads();
        for (int kk = 0; kk < 32; ++kk) {
            double bv = Bs[kk][tx];
            for (int q = 0; q < 4; ++q) acc[q] += As[ty + 8 * q][kk] * bv;
        }
        __syncthreads();
    }
    for (int q = 0; q < 4; ++q) {
        int gr = row0 + ty + 8 * q;
        if (gr < M && col < N) C[(size_t)gr * N + col] = add ? C[(size_t)gr * N + col] + acc[q] : acc[q];
    }
}

// P_c[e] = (1/V_i) sum_{t ni i, k} (vol_t / 4) grad(phi_k)|_t [c] for CSR entry e = (i, k); a lane per
// entry, tets in order, as in k_csr_values
__global__ void k_proj_values(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                              const int* __restrict__ n2t_ptr, const int* __restrict__ n2t,
                              const int* __restrict__ tets, const double* __restrict__ vol,
                              const double* __restrict__ grads, const double* __restrict__ V, int nnz,
                              double* __restrict__ P) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= n) return;
    for (int pos = rowptr[i] + lane; pos < rowptr[i + 1]; pos += 32) {
        const int j = col[pos];
        double s[3] = {0, 0, 0};
        for (int e = n2t_ptr[i]; e < n2t_ptr[i + 1]; ++e) {
            const int t = n2t[e];
            const int b = tet_slot(tets + 4 * t, j);
            if (b < 0) continue;
            const double* g = grads + 12 * t;
            const double q = 0.25 * vol[t] / V[i];
            for (int c = 0; c < 3; ++c) s[c] += q * g[3 * b + c];
        }
        for (int c = 0; c < 3; ++c) P[(size_t)c * nnz + pos] = s[c];
    }
}

// N64[(c n + i)][col] = sum_e P_c[e] U[col_e][col]   (H = -N M with u = U M)
__global__ void k_demag_rows(int n, int ncol, const int* __restrict__ rowptr, const int* __restrict__ col,
                             const double* __restrict__ P, int nnz, const double* __restrict__ U,
                             double* __restrict__ N64) {
    int cc = blockIdx.x * blockDim.x + threadIdx.x;
    int i = blockIdx.y;
    if (cc >= ncol) return;
    double s0 = 0, s1 = 0, s2 = 0;
    for (int e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        double u = U[(size_t)col[e] * ncol + cc];
        s0 += P[e] * u;
        s1 += P[(size_t)nnz + e] * u;
        s2 += P[2 * (size_t)nnz + e] * u;
    }
    N64[((size_t)0 * n + i) * ncol + cc] = s0;
    N64[((size_t)1 * n + i) * ncol + cc] = s1;
    N64[((size_t)2 * n + i) * ncol + cc] = s2;
}

// kernel operand [K][K]: W[r][q] = -mu0 1e6 N[(c n + i)][(c' n + k)], r = c pitch + i, q = c' pitch + k; zero
// in the other rows and columns
__global__ void k_demag_convert(int n, int pitch, int K, const double* __restrict__ N64, float* __restrict__ W32,
                                __nv_bfloat16* __restrict__ Whi, __nv_bfloat16* __restrict__ Wlo) {
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    int r = blockIdx.y;
    if (q >= K) return;
    int c = r / pitch, i = r % pitch, c2 = q / pitch, k = q % pitch;
    double v = 0;
    if (c < 3 && c2 < 3 && i < n && k < n) v = -kMu0 * 1e6 * N64[((size_t)c * n + i) * (3 * (size_t)n) + (size_t)c2 * n + k];
    size_t o = (size_t)r * K + q;
    W32[o] = (float)v;
    __nv_bfloat16 hi = __float2bfloat16_rn((float)v);
    Whi[o] = hi;
    Wlo[o] = __float2bfloat16_rn((float)(v - (double)__bfloat162float(hi)));
}

// Sliced-ELL places of the exchange entries: fills the slices' offsets *off [slices + 1] and returns the CSR
// entry e of each place, ~e for padding (node col[e], value 0).  Entry c of a slice's 32 rows is one gather of
// the stage kernels, lane l from bank (node mod 32).  Column by column every row, the longest first, takes
// the neighbour that meets fewest others in its bank so far, and waits for a later column where even that
// one would lengthen the gather and its row is shorter than the slice; padding reads a node of its row that
// meets fewest.  1.26 instead of 1.93 wavefronts a gather on the census mesh in row order.
// An interval of 4096 islands 24.46 -> 24.16 ms, of 1024 islands 6.60 -> 6.48 ms.
std::vector<int> gather_order(int n, const std::vector<int>& rowptr, const std::vector<int>& col,
                              std::vector<int>* off) {
    const int ns = (n + 31) / 32;
    off->assign(ns + 1, 0);
    for (int q = 0; q < ns; ++q) {
        int w = 0;
        for (int i = 32 * q; i < std::min(n, 32 * q + 32); ++i) w = std::max(w, rowptr[i + 1] - rowptr[i] - 1);
        (*off)[q + 1] = (*off)[q] + 32 * w;
    }
    std::vector<int> slot((*off)[ns]), seen(n, -1), order;
    std::vector<int> left[32];
    for (int q = 0; q < ns; ++q) {
        const int w = ((*off)[q + 1] - (*off)[q]) / 32, rows = std::min(32, n - 32 * q);
        for (int l = 0; l < rows; ++l) {
            left[l].clear();
            for (int e = rowptr[32 * q + l]; e < rowptr[32 * q + l + 1]; ++e)
                if (col[e] != 32 * q + l) left[l].push_back(e);
        }
        order.resize(rows);
        for (int l = 0; l < rows; ++l) order[l] = l;
        std::stable_sort(order.begin(), order.end(),
                         [&](int x, int y) { return left[x].size() > left[y].size(); });
        for (int c = 0; c < w; ++c) {
            const int tag = (*off)[q] / 32 + c;           // of this column, in seen
            int bank[32] = {}, deep = 0, any = -1;        // distinct nodes of the column in each bank, their most
            int* out = &slot[(*off)[q] + 32 * c];
            auto others = [&](int e) { return bank[col[e] & 31] - (seen[col[e]] == tag ? 1 : 0); };
            auto place = [&](int e) {
                if (seen[col[e]] == tag) return;
                seen[col[e]] = tag;
                deep = std::max(deep, ++bank[col[e] & 31]);
            };
            unsigned padded = 0;
            for (int l : order) {
                std::vector<int>& v = left[l];
                size_t best = 0;
                int least = 1 << 30;
                for (size_t k = 0; k < v.size() && least > 0; ++k)
                    if (const int o = others(v[k]); o < least) least = o, best = k;
                if (v.empty() || ((int)v.size() < w - c && least >= std::max(1, deep))) {
                    padded |= 1u << l;
                    continue;
                }
                any = out[l] = v[best];
                place(out[l]);
                v.erase(v.begin() + best);
            }
            for (int l = 0; l < 32; ++l) {
                if (l >= rows) out[l] = ~any;
                if (l >= rows || !(padded >> l & 1)) continue;
                int pick = rowptr[32 * q + l], least = others(pick);
                for (int e = pick + 1; e < rowptr[32 * q + l + 1] && least > 0; ++e)
                    if (const int o = others(e); o < least) least = o, pick = e;
                place(pick);
                out[l] = ~pick;
            }
        }
    }
    return slot;
}

}  // namespace

void free_mesh(Mesh* M) {
    if (!M) return;
    cudaFree(M->node_pos);
    cudaFree(M->node_mat);
    cudaFree(M->sell_off);
    cudaFree(M->sell_ent);
    cudaFree(M->sell_il);
    cudaFree(M->N32);
    cudaFree(M->Nhi);
    cudaFree(M->Nlo);
    cudaFree(M->N64);
    cudaFree(M->csr_rowptr);
    cudaFree(M->csr_col);
    cudaFree(M->csr_c64);
    cudaFree(M->node64);
    cudaFree(M->mat64);
    delete M;
}

int assemble_mesh(bpm_ctx* ctx, Mesh* M, const double* xyz, const int32_t* tets_in, int32_t nt,
                  const int32_t* region, const bpm_region_mat* mats, int32_t nreg, uint32_t flags) {
    const int n = M->n;
    cudaStream_t st = ctx->stream;
    // ---------------- host topology ----------------
    std::vector<int> tets(tets_in, tets_in + 4 * (size_t)nt);
    for (int t = 0; t < nt; ++t) {
        for (int a = 0; a < 4; ++a)
            if (tets[4 * t + a] < 0 || tets[4 * t + a] >= n) {
                set_error("tet %d references node %d outside [0, %d)", t, tets[4 * t + a], n);
                return BPM_ERR_ARG;
            }
        if (region[t] < 0 || region[t] >= nreg) {
            set_error("tet %d has region %d outside [0, %d)", t, region[t], nreg);
            return BPM_ERR_ARG;
        }
        V3 x0 = ld3(xyz + 3 * tets[4 * t]);
        V3 e1 = sub(ld3(xyz + 3 * tets[4 * t + 1]), x0), e2 = sub(ld3(xyz + 3 * tets[4 * t + 2]), x0),
           e3 = sub(ld3(xyz + 3 * tets[4 * t + 3]), x0);
        double det = dot(e1, cross(e2, e3));
        double h = std::max(nrm(e1), std::max(nrm(e2), nrm(e3)));
        if (!(fabs(det) > 1e-10 * h * h * h)) {
            set_error("tet %d is degenerate", t);
            return BPM_ERR_ARG;
        }
    }
    // node -> tets
    std::vector<int> n2t_ptr(n + 1, 0), n2t(4 * (size_t)nt);
    for (int k = 0; k < 4 * nt; ++k) n2t_ptr[tets[k] + 1]++;
    for (int i = 0; i < n; ++i) n2t_ptr[i + 1] += n2t_ptr[i];
    {
        std::vector<int> fill(n2t_ptr.begin(), n2t_ptr.end() - 1);
        for (int t = 0; t < nt; ++t)
            for (int a = 0; a < 4; ++a) n2t[fill[tets[4 * t + a]]++] = t;
    }
    for (int i = 0; i < n; ++i)
        if (n2t_ptr[i + 1] == n2t_ptr[i]) {
            set_error("node %d belongs to no tetrahedron", i);
            return BPM_ERR_ARG;
        }
    // CSR pattern (sorted, incl. diagonal)
    std::vector<int>& rowptr = M->rowptr;
    std::vector<int>& col = M->col;
    rowptr.assign(n + 1, 0);
    col.clear();
    {
        std::vector<int> nb;
        for (int i = 0; i < n; ++i) {
            nb.clear();
            for (int e = n2t_ptr[i]; e < n2t_ptr[i + 1]; ++e)
                for (int a = 0; a < 4; ++a) nb.push_back(tets[4 * n2t[e] + a]);
            std::sort(nb.begin(), nb.end());
            nb.erase(std::unique(nb.begin(), nb.end()), nb.end());
            col.insert(col.end(), nb.begin(), nb.end());
            rowptr[i + 1] = (int)col.size();
        }
    }
    const int nnz = (int)col.size();
    // bodies of the mesh (connected parts of the node graph), in the order of their first nodes: body of
    // each node, nodes by body (ascending), first of each body
    std::vector<int> body(n, -1), by_body, body_ptr(1, 0);
    by_body.reserve(n);
    for (int i = 0; i < n; ++i) {
        if (body[i] >= 0) continue;
        const int p = (int)body_ptr.size() - 1;
        body[i] = p;
        by_body.push_back(i);
        for (size_t q = body_ptr[p]; q < by_body.size(); ++q)
            for (int e = rowptr[by_body[q]]; e < rowptr[by_body[q] + 1]; ++e)
                if (body[col[e]] < 0) {
                    body[col[e]] = p;
                    by_body.push_back(col[e]);
                }
        std::sort(by_body.begin() + body_ptr[p], by_body.end());
        body_ptr.push_back((int)by_body.size());
    }
    const int n_bodies = (int)body_ptr.size() - 1;
    // boundary faces: faces of exactly one tet, oriented outward
    struct Face {
        uint64_t key;                      // sorted corners, 21 bits each
        int a, b, c, opposite;
    };
    std::vector<Face> fl;
    fl.reserve(4 * (size_t)nt);
    for (int t = 0; t < nt; ++t)
        for (int k = 0; k < 4; ++k) {
            int f[3], q = 0;
            for (int a = 0; a < 4; ++a)
                if (a != k) f[q++] = tets[4 * t + a];
            int o[3] = {f[0], f[1], f[2]};
            std::sort(o, o + 3);
            fl.push_back(Face{(uint64_t)o[0] << 42 | (uint64_t)o[1] << 21 | (uint64_t)o[2], f[0], f[1], f[2],
                              tets[4 * t + k]});
        }
    std::sort(fl.begin(), fl.end(), [](const Face& x, const Face& y) { return x.key < y.key; });
    std::vector<int> faces;
    for (size_t i = 0, j; i < fl.size(); i = j) {
        for (j = i + 1; j < fl.size() && fl[j].key == fl[i].key; ++j) {}
        if (j - i != 1) continue;
        int a = fl[i].a, b = fl[i].b, c = fl[i].c, d = fl[i].opposite;
        V3 ya = ld3(xyz + 3 * a);
        V3 nrmv = cross(sub(ld3(xyz + 3 * b), ya), sub(ld3(xyz + 3 * c), ya));
        if (dot(nrmv, sub(ld3(xyz + 3 * d), ya)) > 0) std::swap(b, c);
        faces.push_back(a);
        faces.push_back(b);
        faces.push_back(c);
    }
    const int nf = (int)faces.size() / 3;
    if (nf == 0) {
        set_error("the mesh has no boundary face: every face belongs to two or more tetrahedra");
        return BPM_ERR_ARG;
    }
    std::vector<int> bnodes(faces.begin(), faces.end());
    std::sort(bnodes.begin(), bnodes.end());
    bnodes.erase(std::unique(bnodes.begin(), bnodes.end()), bnodes.end());
    const int nb = (int)bnodes.size();
    std::vector<int> bidx(n, -1);
    for (int k = 0; k < nb; ++k) bidx[bnodes[k]] = k;
    std::vector<int> b2f_ptr(nb + 1, 0), b2f(3 * (size_t)nf);
    for (int k = 0; k < 3 * nf; ++k) b2f_ptr[bidx[faces[k]] + 1]++;
    for (int k = 0; k < nb; ++k) b2f_ptr[k + 1] += b2f_ptr[k];
    {
        std::vector<int> fill(b2f_ptr.begin(), b2f_ptr.end() - 1);
        for (int f = 0; f < nf; ++f)
            for (int a = 0; a < 3; ++a) b2f[fill[bidx[faces[3 * f + a]]]++] = f;
    }
    std::vector<unsigned char> interior(n, 1);
    for (int k = 0; k < nb; ++k) interior[bnodes[k]] = 0;
    std::vector<double> mat_Ms(nreg), mat_Ku(nreg), mat_A(nreg);
    for (int r = 0; r < nreg; ++r) {
        mat_Ms[r] = mats[r].Ms_A_per_m;
        mat_Ku[r] = mats[r].Ku_J_per_m3;
        mat_A[r] = mats[r].A_J_per_m;
        if (!(mat_Ms[r] > 0)) {
            set_error("region %d has Ms <= 0", r);
            return BPM_ERR_ARG;
        }
    }

    // ---------------- device assembly ----------------
    DevPool pool(st);
    double *d_xyz, *d_vol, *d_grads, *d_V, *d_Ms, *d_Ku, *d_KA, *d_KL, *d_mMs, *d_mKu, *d_mA;
    int *d_tets, *d_reg, *d_n2tp, *d_n2t, *d_rowptr, *d_col, *d_bnodes, *d_faces, *d_b2fp, *d_b2f;
    unsigned char* d_int;
    std::vector<double> xyzv(xyz, xyz + 3 * (size_t)n);
    std::vector<int> regv(region, region + nt);
    BPM_TRY(upload(pool, &d_xyz, xyzv));
    BPM_TRY(upload(pool, &d_tets, tets));
    BPM_TRY(upload(pool, &d_reg, regv));
    BPM_TRY(upload(pool, &d_n2tp, n2t_ptr));
    BPM_TRY(upload(pool, &d_n2t, n2t));
    BPM_TRY(upload(pool, &d_rowptr, rowptr));
    BPM_TRY(upload(pool, &d_col, col));
    BPM_TRY(upload(pool, &d_bnodes, bnodes));
    BPM_TRY(upload(pool, &d_faces, faces));
    BPM_TRY(upload(pool, &d_b2fp, b2f_ptr));
    BPM_TRY(upload(pool, &d_b2f, b2f));
    BPM_TRY(upload(pool, &d_int, interior));
    BPM_TRY(upload(pool, &d_mMs, mat_Ms));
    BPM_TRY(upload(pool, &d_mKu, mat_Ku));
    BPM_TRY(upload(pool, &d_mA, mat_A));
    BPM_TRY(pool.alloc(&d_vol, nt));
    BPM_TRY(pool.alloc(&d_grads, 12 * (size_t)nt));
    BPM_TRY(pool.alloc(&d_V, n));
    BPM_TRY(pool.alloc(&d_Ms, n));
    BPM_TRY(pool.alloc(&d_Ku, n));
    BPM_TRY(pool.alloc(&d_KA, nnz));
    BPM_TRY(pool.alloc(&d_KL, nnz));
    const int T = 256;
    k_tet_geom<<<(nt + T - 1) / T, T, 0, st>>>(nt, d_xyz, d_tets, d_vol, d_grads);
    k_node_lumped<<<(n + T - 1) / T, T, 0, st>>>(n, d_n2tp, d_n2t, d_reg, d_vol, d_mMs, d_mKu, d_V, d_Ms, d_Ku);
    const int gRow = (32 * n + T - 1) / T;   // a warp per row
    k_csr_values<<<gRow, T, 0, st>>>(n, d_rowptr, d_col, d_n2tp, d_n2t, d_tets, d_reg, d_mA, d_vol, d_grads, d_KA,
                                     d_KL);
    BPM_CK(cudaGetLastError());
    // exchange operator values (FP32) and lambda_max
    float* d_c;
    BPM_TRY(pool.alloc(&d_c, nnz));
    k_exchange_values<<<(n + T - 1) / T, T, 0, st>>>(n, d_rowptr, d_col, d_KA, d_V, d_Ms, d_c);
    BPM_CK(cudaMalloc(&M->csr_rowptr, (n + 1) * sizeof(int)));
    BPM_CK(cudaMalloc(&M->csr_col, nnz * sizeof(int)));
    BPM_CK(cudaMalloc(&M->csr_c64, nnz * sizeof(double)));
    BPM_CK(cudaMemcpyAsync(M->csr_rowptr, d_rowptr, (n + 1) * sizeof(int), cudaMemcpyDeviceToDevice, st));
    BPM_CK(cudaMemcpyAsync(M->csr_col, d_col, nnz * sizeof(int), cudaMemcpyDeviceToDevice, st));
    k_exchange_values64<<<(n + T - 1) / T, T, 0, st>>>(n, d_rowptr, d_col, d_KA, d_V, d_Ms, M->csr_c64);
    // the matrix pattern in 32-row slices, for the power iteration and CG
    const int n_sl = (n + 31) / 32;
    std::vector<int> soff(n_sl + 1, 0);
    for (int q = 0; q < n_sl; ++q) {
        int w = 0;
        for (int i = 32 * q; i < std::min(n, 32 * q + 32); ++i) w = std::max(w, rowptr[i + 1] - rowptr[i]);
        soff[q + 1] = soff[q] + 32 * w;
    }
    Sliced A{};
    A.len = soff[n_sl];
    std::vector<int> scol(A.len), ssrc(A.len), srow(A.len);
    for (int q = 0; q < n_sl; ++q)
        for (int k = soff[q]; k < soff[q + 1]; ++k) {
            const int i = 32 * q + ((k - soff[q]) & 31), e = i < n ? rowptr[i] + (k - soff[q]) / 32 : 0;
            const bool in = i < n && e < rowptr[i + 1];
            srow[k] = i < n ? i : 0;
            scol[k] = in ? col[e] : srow[k];
            ssrc[k] = in ? e : -1;
        }
    int *d_soff, *d_scol, *d_ssrc, *d_srow;
    double *d_sval, *d_sval_in, *d_sval_x, *d_dx, *d_lam;
    BPM_TRY(upload(pool, &d_soff, soff));
    BPM_TRY(upload(pool, &d_scol, scol));
    BPM_TRY(upload(pool, &d_ssrc, ssrc));
    BPM_TRY(upload(pool, &d_srow, srow));
    A.off = d_soff;
    A.col = d_scol;
    A.src = d_ssrc;
    BPM_TRY(pool.alloc(&d_sval, A.len, false));
    BPM_TRY(pool.alloc(&d_sval_in, A.len, false));
    BPM_TRY(pool.alloc(&d_sval_x, A.len, false));
    BPM_TRY(pool.alloc(&d_dx, n, false));
    BPM_TRY(pool.alloc(&d_lam, 1, false));
    const int gS = (A.len + T - 1) / T;
    k_exchange_scale<<<(n + T - 1) / T, T, 0, st>>>(n, d_V, d_Ms, d_dx);
    k_sliced_values<<<gS, T, 0, st>>>(A, d_srow, d_KA, d_dx, nullptr, d_sval_x);
    BPM_CK(cudaGetLastError());
    // lambda_max on a stream of its own, beside the demag assembly
    SideStream side;
    BPM_TRY(side.fork(st));
    const int psmem = 2 * (int)sizeof(double) * n;
    BPM_CK(cudaFuncSetAttribute(k_power_iteration, cudaFuncAttributeMaxDynamicSharedMemorySize, psmem));
    k_power_iteration<<<kPowCluster, kPowThreads, psmem, side.s>>>(n, A, d_sval_x, 1500, d_lam);
    BPM_CK(cudaGetLastError());
    M->exch_val.resize(nnz);
    M->V.resize(n);
    M->Ms.resize(n);
    M->Ku.resize(n);
    BPM_CK(cudaMemcpyAsync(M->exch_val.data(), d_c, nnz * sizeof(float), cudaMemcpyDeviceToHost, st));
    BPM_CK(cudaMemcpyAsync(M->V.data(), d_V, n * sizeof(double), cudaMemcpyDeviceToHost, st));
    BPM_CK(cudaMemcpyAsync(M->Ms.data(), d_Ms, n * sizeof(double), cudaMemcpyDeviceToHost, st));
    BPM_CK(cudaMemcpyAsync(M->Ku.data(), d_Ku, n * sizeof(double), cudaMemcpyDeviceToHost, st));

    // ---------------- Fredkin-Koehler demag ----------------
    const int ncol = 3 * n;
    const size_t NN = (size_t)n * n, NB = (size_t)n * nb;
    double *d_RT, *d_rv;
    BPM_TRY(pool.alloc(&d_RT, 3 * (size_t)nnz, false));
    BPM_TRY(pool.alloc(&d_rv, 3 * (size_t)A.len, false));
    k_source<<<gRow, T, 0, st>>>(n, d_rowptr, d_col, d_n2tp, d_n2t, d_tets, d_vol, d_grads, nnz, d_RT);
    for (int c = 0; c < 3; ++c)
        k_sliced_values<<<gS, T, 0, st>>>(A, d_srow, d_RT + (size_t)c * nnz, nullptr, nullptr,
                                          d_rv + (size_t)c * A.len);
    BPM_CK(cudaGetLastError());
    // the Laplacian scaled to a unit diagonal, whole and with interior rows and columns only
    double *d_sc, *d_sc_in;
    BPM_TRY(pool.alloc(&d_sc, n, false));
    BPM_TRY(pool.alloc(&d_sc_in, n, false));
    k_diag_scale<<<(n + T - 1) / T, T, 0, st>>>(n, d_rowptr, d_col, d_KL, d_int, d_sc, d_sc_in);
    k_sliced_values<<<gS, T, 0, st>>>(A, d_srow, d_KL, d_sc, nullptr, d_sval);
    k_sliced_values<<<gS, T, 0, st>>>(A, d_srow, d_KL, d_sc, d_int, d_sval_in);
    BPM_CK(cudaGetLastError());
    int it1 = 0, it2 = 0;
    double res1 = 0, res2 = 0;
    // G = K^+ for the nodal sources, zero-mean gauge on each body
    int *d_body, *d_by_body, *d_body_ptr;
    BPM_TRY(upload(pool, &d_body, body));
    BPM_TRY(upload(pool, &d_by_body, by_body));
    BPM_TRY(upload(pool, &d_body_ptr, body_ptr));
    double *d_b, *d_G;
    BPM_TRY(pool.alloc(&d_b, NN, false));
    BPM_TRY(pool.alloc(&d_G, NN, false));
    k_unit_sources<<<dim3((n + 127) / 128, n), 128, 0, st>>>(n, d_body, d_body_ptr, d_b);
    BPM_TRY(pcg(st, pool, n, n, A, d_sval, d_sc, d_b, d_G, 1e-12, 20000, &it1, &res1));
    k_col_mean_sub<<<dim3((n + 31) / 32, n_bodies), 256, 0, st>>>(d_by_body, d_body_ptr, n, d_G);
    // boundary values of u2 from u1
    double *d_omega, *d_Bmat;
    BPM_TRY(pool.alloc(&d_omega, nb, false));
    BPM_TRY(pool.alloc(&d_Bmat, (size_t)nb * nb, false));
    k_interior_angles<<<(nb + 127) / 128, 128, 0, st>>>(nb, d_bnodes, d_n2tp, d_n2t, d_tets, d_xyz, d_omega);
    {   // observers in blocks whose weights stay within 256 MB
        double* d_W;
        const int rows = std::max(1, std::min(nb, (int)((size_t(256) << 20) / (3 * sizeof(double) * (size_t)nf))));
        BPM_TRY(pool.alloc(&d_W, 3 * (size_t)rows * nf, false));
        for (int i0 = 0; i0 < nb; i0 += rows) {
            const int m = std::min(rows, nb - i0);
            k_bem_weights<<<dim3((nf + 127) / 128, m), 128, 0, st>>>(i0, m, nf, d_bnodes, d_xyz, d_faces, d_W);
            k_bem_matrix<<<dim3((nb + 127) / 128, m), 128, 0, st>>>(i0, nb, nf, d_bnodes, d_faces, d_b2fp, d_b2f,
                                                                    d_omega, d_W, d_Bmat);
        }
    }
    // harmonic extension E of unit boundary values: K_II E_I = -K_IB, identity on the boundary
    double *d_bD, *d_E, *d_F, *d_GB;
    int* d_bidx;
    BPM_TRY(upload(pool, &d_bidx, bidx));
    BPM_TRY(pool.alloc(&d_bD, NB));
    BPM_TRY(pool.alloc(&d_E, NB));
    if (nb < n) {
        k_boundary_sources<<<gRow, T, 0, st>>>(n, nb, d_rowptr, d_col, d_KL, d_int, d_bidx, d_bD);
        BPM_TRY(pcg(st, pool, n, nb, A, d_sval_in, d_sc_in, d_bD, d_E, 1e-12, 20000, &it2, &res2));
    }
    k_boundary_identity<<<(nb + T - 1) / T, T, 0, st>>>(nb, d_bnodes, d_E);
    // Q = G + (E B) G_boundary: potential u1 + u2 of the nodal sources
    BPM_TRY(pool.alloc(&d_F, NB, false));
    BPM_TRY(pool.alloc(&d_GB, (size_t)nb * n, false));
    const dim3 gemm_threads(32, 8);
    k_gather_rows<<<dim3((n + 127) / 128, nb), 128, 0, st>>>(nb, n, d_bnodes, d_G, d_GB);
    k_dgemm<<<dim3((nb + 31) / 32, (n + 31) / 32), gemm_threads, 0, st>>>(n, nb, nb, d_E, d_Bmat, 0, d_F);
    k_dgemm<<<dim3((n + 31) / 32, (n + 31) / 32), gemm_threads, 0, st>>>(n, n, nb, d_F, d_GB, 1, d_G);
    // U = Q R, N = P U
    double *d_U, *d_P;
    BPM_TRY(pool.alloc(&d_U, (size_t)n * ncol, false));
    BPM_TRY(pool.alloc(&d_P, 3 * (size_t)nnz, false));
    k_apply_source<<<dim3((n + 127) / 128, n), 128, 0, st>>>(n, A, d_rv, d_G, d_U);
    k_proj_values<<<gRow, T, 0, st>>>(n, d_rowptr, d_col, d_n2tp, d_n2t, d_tets, d_vol, d_grads, d_V, nnz, d_P);
    BPM_CK(cudaGetLastError());
    double* N64 = nullptr;
    BPM_CK(cudaMalloc(&N64, (size_t)ncol * ncol * sizeof(double)));
    M->N64 = N64;  // freed below unless kept
    k_demag_rows<<<dim3((ncol + 127) / 128, n), 128, 0, st>>>(n, ncol, d_rowptr, d_col, d_P, nnz, d_U, N64);
    const int K = M->K();
    BPM_CK(cudaMalloc(&M->N32, (size_t)K * K * sizeof(float)));
    BPM_CK(cudaMalloc(&M->Nhi, (size_t)K * K * sizeof(__nv_bfloat16)));
    BPM_CK(cudaMalloc(&M->Nlo, (size_t)K * K * sizeof(__nv_bfloat16)));
    k_demag_convert<<<dim3((K + 127) / 128, K), 128, 0, st>>>(n, M->pitch, K, N64, M->N32, M->Nhi, M->Nlo);
    BPM_CK(cudaGetLastError());
    double lam = 0;
    BPM_TRY(side.join(st));
    std::vector<int> off;
    const std::vector<int> slot = gather_order(n, rowptr, col, &off);   // on the host beside the kernels above
    M->n_slices = (int)off.size() - 1;
    BPM_CK(cudaMemcpyAsync(&lam, d_lam, sizeof(double), cudaMemcpyDeviceToHost, st));
    BPM_CK(cudaStreamSynchronize(st));
    if (!(flags & BPM_MESH_KEEP_F64)) {
        cudaFree(M->N64);
        M->N64 = nullptr;
    }

    // ---------------- node data and sliced-ELL exchange ----------------
    const int np = M->n_pad;
    double Vsum = 0;
    for (int i = 0; i < n; ++i) Vsum += M->V[i];
    std::vector<float4> pos(np, make_float4(0, 0, 0, 0)), nm(np, make_float4(0, 0, 0, 0));
    double an_max = 0, ms_max = 0;
    for (int i = 0; i < n; ++i) {
        pos[i] = make_float4((float)xyz[3 * i], (float)xyz[3 * i + 1], (float)xyz[3 * i + 2],
                             (float)(M->V[i] / Vsum));

        double an = 2.0 * M->Ku[i] / M->Ms[i];
        nm[i] = make_float4((float)an, (float)(M->Ms[i] * 1e-6), 0.f, 0.f);
        an_max = std::max(an_max, an);
        ms_max = std::max(ms_max, M->Ms[i]);
    }
    std::vector<int2> ent(std::max<size_t>(1, slot.size()), make_int2(0, 0));
    for (size_t k = 0; k < slot.size(); ++k) {
        const float v = slot[k] < 0 ? 0.f : M->exch_val[slot[k]];
        ent[k] = make_int2(col[slot[k] < 0 ? ~slot[k] : slot[k]], *reinterpret_cast<const int*>(&v));
    }
    std::vector<int2> ent_il(ent.size());
    for (size_t k = 0; k < ent.size(); ++k) {
        const int j = ent[k].x;
        ent_il[k] = make_int2(4 * ((j >> 5) * 96 * kIlIslands + (j & 31)), ent[k].y);
    }
    std::vector<NodeF64> node64(n);
    std::vector<double2> mat64(n);
    for (int i = 0; i < n; ++i) {
        node64[i] = NodeF64{xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], M->V[i] / Vsum};
        mat64[i] = make_double2(2.0 * M->Ku[i] / M->Ms[i], M->Ms[i]);
    }
    BPM_CK(cudaMalloc(&M->node64, n * sizeof(NodeF64)));
    BPM_CK(cudaMalloc(&M->mat64, n * sizeof(double2)));
    BPM_CK(cudaMemcpy(M->node64, node64.data(), n * sizeof(NodeF64), cudaMemcpyHostToDevice));
    BPM_CK(cudaMemcpy(M->mat64, mat64.data(), n * sizeof(double2), cudaMemcpyHostToDevice));
    BPM_CK(cudaMalloc(&M->node_pos, np * sizeof(float4)));
    BPM_CK(cudaMalloc(&M->node_mat, np * sizeof(float4)));
    BPM_CK(cudaMalloc(&M->sell_off, off.size() * sizeof(int)));
    BPM_CK(cudaMalloc(&M->sell_ent, ent.size() * sizeof(int2)));
    BPM_CK(cudaMalloc(&M->sell_il, ent_il.size() * sizeof(int2)));
    BPM_CK(cudaMemcpy(M->node_pos, pos.data(), np * sizeof(float4), cudaMemcpyHostToDevice));
    BPM_CK(cudaMemcpy(M->node_mat, nm.data(), np * sizeof(float4), cudaMemcpyHostToDevice));
    BPM_CK(cudaMemcpy(M->sell_off, off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice));
    BPM_CK(cudaMemcpy(M->sell_ent, ent.data(), ent.size() * sizeof(int2), cudaMemcpyHostToDevice));
    BPM_CK(cudaMemcpy(M->sell_il, ent_il.data(), ent_il.size() * sizeof(int2), cudaMemcpyHostToDevice));

    M->nb = nb;
    M->nnz = nnz;
    bpm_mesh_info& I = M->info;
    I.n_nodes = n;
    I.n_pad = np;
    I.k_pad = M->k_pad;
    I.n_tets = nt;
    I.n_boundary = nb;
    I.nnz = nnz;
    I.cg_iters_neumann = it1;
    I.cg_iters_dirichlet = it2;
    I.volume_nm3 = Vsum;
    I.exchange_lambda_max_T = lam;
    I.field_bound_T = lam + an_max + kMu0 * ms_max;
    M->an_max = an_max;
    M->ms_max = ms_max;
    I.cg_residual_neumann = res1;
    I.cg_residual_dirichlet = res2;
    return BPM_OK;
}

}  // namespace bpm
