// CUDA-core demag GEMMs: C[M][N] = A[M][K] * W[N][K]^T (both operands K-major).
//
// The FP32 kernel is the plain (single-precision) form of the demag product
// H_d = N' (Ms m); the BF16x3 kernel evaluates, on CUDA cores, the same three
// split products hi*hi + lo*hi + hi*lo that the tensor-core kernel computes,
// and serves to validate it.
#include "bpm_internal.cuh"

namespace bpm {

namespace {

constexpr int BM = 128, BN = 128, BK = 8;

// FP32 product.  Both operands are contiguous along K, so tiles go to shared memory as they are, by
// 16-byte cp.async into a ring of kFStages stages of 32 k, and a thread reads four k of a row at once.
// The pairs (k, k + 1) of those reads are the lanes of packed FMAs (fma.rn.f32x2), and two groups of
// warps take the fours of k in turn: an output has four sums, added at the end, and nothing is shuffled
// into pairs.  A warp holds TM rows of A (its loads are broadcasts) by 32 TN rows of W; rows of 36 words
// put the eight rows of a quarter warp's load in distinct banks.
// The bound is the FP32 FMA rate (80 TFLOP/s).  64 x 128 outputs of 2 x 8 warps: 200 rows of a 4672 x
// 4672 operator are 148 CTAs, one an SM, 0.29 ms (0.32 with one group: two warps a scheduler do not
// cover the FMAs' latency; 1.04 with 128 x 128 tiles, 74 CTAs, and scalar loads and FMAs).  Up to 32 rows
// take 16 x 32 tiles, so that their few rows still give every SM a CTA.  The sum of an output does not
// depend on the tile.
constexpr int kFK = 32, kFLd = kFK + 4, kFStages = 4;

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool in) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    const int bytes = in ? 16 : 0;                         // rows past the end are zero
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void fma2(float2& c, float2 a, float2 b) {
    unsigned long long& cc = reinterpret_cast<unsigned long long&>(c);
    asm("fma.rn.f32x2 %0, %1, %2, %0;"
        : "+l"(cc)
        : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
}

template <int WARPS, int TM, int TN>
__global__ void __launch_bounds__(64 * WARPS) k_gemm_f32(int M, int N, int K, const float* __restrict__ A, int lda,
                                                         const float* __restrict__ W, int ldw, float* __restrict__ C,
                                                         int ldc) {
    constexpr int BM = WARPS * TM, BN = 32 * TN, kFThreads = 64 * WARPS;
    extern __shared__ float fs[];
    constexpr int stage = (BM + BN) * kFLd;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) % WARPS, group = (threadIdx.x >> 5) / WARPS;
    auto load = [&](int kb) {
        float* d = fs + (kb % kFStages) * stage;
        const int k0 = kb * kFK;
        for (int e = threadIdx.x; e < (BM + BN) * (kFK / 4); e += kFThreads) {
            const int r = e / (kFK / 4), c = 4 * (e % (kFK / 4));
            const bool is_a = r < BM;
            const int g = is_a ? m0 + r : n0 + r - BM;
            const bool in = g < (is_a ? M : N);
            const float* src = is_a ? A + (size_t)(in ? g : 0) * lda : W + (size_t)(in ? g : 0) * ldw;
            cp_async16(d + r * kFLd + c, src + k0 + c, in);
        }
    };
    float2 acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
    const int nk = K / kFK;
    for (int p = 0; p < kFStages - 1; ++p) {
        if (p < nk) load(p);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int kb = 0; kb < nk; ++kb) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kFStages - 2) : "memory");
        __syncthreads();                                   // stage kb landed; stage kb - 1 is free
        if (kb + kFStages - 1 < nk) load(kb + kFStages - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float* as = fs + (kb % kFStages) * stage + warp * TM * kFLd + 4 * group;
        const float* ws = fs + (kb % kFStages) * stage + (BM + lane) * kFLd + 4 * group;
#pragma unroll
        for (int k = 0; k < kFK; k += 8) {
            float4 a[TM], w[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(as + i * kFLd + k);
#pragma unroll
            for (int j = 0; j < TN; ++j) w[j] = *reinterpret_cast<const float4*>(ws + j * 32 * kFLd + k);
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    fma2(acc[i][j], make_float2(a[i].x, a[i].y), make_float2(w[j].x, w[j].y));
                    fma2(acc[i][j], make_float2(a[i].z, a[i].w), make_float2(w[j].z, w[j].w));
                }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                       // the ring is free: the second group's sums pass through it
    float* part = fs + warp * TM * BN + lane;
    static_assert(BM * BN <= kFStages * stage, "the sums fit the ring");
    if (group == 1) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) part[i * BN + 32 * j] = acc[i][j].x + acc[i][j].y;
    }
    __syncthreads();
    if (group == 1) return;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int gm = m0 + warp * TM + i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int gn = n0 + lane + 32 * j;
            if (gn < N) C[(size_t)gm * ldc + gn] = (acc[i][j].x + acc[i][j].y) + part[i * BN + 32 * j];
        }
    }
}

// reference of the split products: 128x128 output tile per CTA, 256 threads with an 8x8 register tile
// each, K staged through shared memory 8 at a time
__global__ void __launch_bounds__(256) k_gemm_split_ref(int M, int N, int K, const __nv_bfloat16* __restrict__ Ahi,
                                                        const __nv_bfloat16* __restrict__ Alo,
                                                        const __nv_bfloat16* __restrict__ Whi,
                                                        const __nv_bfloat16* __restrict__ Wlo, int products,
                                                        float* __restrict__ C) {
    __shared__ float As[BK][BM + 4], Ws[BK][BN + 4], Als[BK][BM + 4], Wls[BK][BN + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    float acc[8][8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int p = 0; p < 8; ++p) acc[q][p] = 0.f;
    // loader: thread handles row lr (0..127) and k-half lk (0 or 4)
    const int lr = tid >> 1, lk = (tid & 1) * 4;
    for (int k0 = 0; k0 < K; k0 += BK) {
        int gm = m0 + lr, gn = n0 + lr;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int gk = k0 + lk + u;
            bool okk = gk < K;
            As[lk + u][lr] = (gm < M && okk) ? __bfloat162float(Ahi[(size_t)gm * K + gk]) : 0.f;
            Als[lk + u][lr] = (gm < M && okk) ? __bfloat162float(Alo[(size_t)gm * K + gk]) : 0.f;
            Ws[lk + u][lr] = (gn < N && okk) ? __bfloat162float(Whi[(size_t)gn * K + gk]) : 0.f;
            Wls[lk + u][lr] = (gn < N && okk) ? __bfloat162float(Wlo[(size_t)gn * K + gk]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[8], w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) a[q] = As[kk][ty + 16 * q];
#pragma unroll
            for (int p = 0; p < 8; ++p) w[p] = Ws[kk][tx + 16 * p];
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int p = 0; p < 8; ++p) acc[q][p] = fmaf(a[q], w[p], acc[q][p]);
            if (products > 1) {
                float al[8], wl[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) al[q] = Als[kk][ty + 16 * q];
#pragma unroll
                for (int p = 0; p < 8; ++p) wl[p] = Wls[kk][tx + 16 * p];
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        acc[q][p] = fmaf(al[q], w[p], acc[q][p]);
                        acc[q][p] = fmaf(a[q], wl[p], acc[q][p]);
                    }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        int gm = m0 + ty + 16 * q;
        if (gm >= M) continue;
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            int gn = n0 + tx + 16 * p;
            if (gn < N) C[(size_t)gm * N + gn] = acc[q][p];
        }
    }
}

template <int WARPS, int TM, int TN>
int launch_f32(cudaStream_t s, int M, int N, int K, const float* A, int lda, const float* W, int ldw, float* C,
               int ldc) {
    constexpr int BM = WARPS * TM, BN = 32 * TN, smem = kFStages * (BM + BN) * kFLd * (int)sizeof(float);
    BPM_CK(cudaFuncSetAttribute(k_gemm_f32<WARPS, TM, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    k_gemm_f32<WARPS, TM, TN><<<dim3((N + BN - 1) / BN, (M + BM - 1) / BM), 64 * WARPS, smem, s>>>(M, N, K, A, lda, W,
                                                                                                    ldw, C, ldc);
    BPM_CK(cudaGetLastError());
    return BPM_OK;
}

}  // namespace

int gemm_f32_nt(cudaStream_t s, int M, int N, int K, const float* A, int lda, const float* W, int ldw, float* C,
                int ldc) {
    if (K % kFK || lda % 4 || ldw % 4 || (reinterpret_cast<uintptr_t>(A) & 15) || (reinterpret_cast<uintptr_t>(W) & 15)) {
        set_error("FP32 GEMM needs K %% %d == 0 and 16-byte aligned rows (K=%d lda=%d ldw=%d)", kFK, K, lda, ldw);
        return BPM_ERR_ARG;
    }
    return M <= 32 ? launch_f32<4, 4, 1>(s, M, N, K, A, lda, W, ldw, C, ldc)
                   : launch_f32<8, 8, 4>(s, M, N, K, A, lda, W, ldw, C, ldc);
}

int gemm_bf16x3_simt(cudaStream_t s, int M, int N, int K, const __nv_bfloat16* Ahi, const __nv_bfloat16* Alo,
                     const __nv_bfloat16* Whi, const __nv_bfloat16* Wlo, float* C, int products) {
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
    k_gemm_split_ref<<<grid, 256, 0, s>>>(M, N, K, Ahi, Alo, Whi, Wlo, products, C);
    BPM_CK(cudaGetLastError());
    return BPM_OK;
}

}  // namespace bpm
