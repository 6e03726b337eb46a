// Tensor-core GEMM with fused epilogues (tcgen05, sm_103a), used by the surrogate MLP:
//   C[M][N] = A[M][K] * W[N][K]^T, BF16 operands, FP32 accumulate in TMEM
// (the batched demag product uses the persistent grouped kernel in
// bpm_gemm_grouped.cu).
//
// One CTA computes a 128-row output tile of 32 to 256 columns (by epilogue and
// size, see Cfg and gemm_tc).  Warp 0 (one elected lane) streams the k-blocks (64
// BF16 = one 128-byte swizzle atom) of both operand tiles with TMA into a ring of
// shared-memory stages, warp 1 (one elected lane) issues the tcgen05.mma
// instructions into a TMEM accumulator of 128 lanes, and after the last k-block
// all eight warps read the accumulator back with tcgen05.ld and store it.
// Every mbarrier wait is bounded; on timeout the kernel records an error flag,
// drains its own copies and MMAs, frees TMEM and exits.
#include <cuda.h>

#include "bpm_tc_ptx.cuh"

namespace bpm {

namespace {

using namespace tc;

// warp 0 issues the TMA loads and warp 1 the MMAs; all eight warps run the epilogue, warp w
// on TMEM lane quarter w % 4 (rows) and every second 32 columns, from 32 (w / 4)
constexpr int kThreads = 256;

// The forward layers of the MLP (bias+GELU and output epilogues) have K <= 256, at most four
// k-blocks: two stages keep their ring full and halve the shared memory, so that two CTAs share
// an SM and one CTA's epilogue runs beside the other's MMAs.  The other GEMMs (K = batch rows)
// keep the deep ring.
// Column tiles: the widest whose CTAs fill the SMs (tile_width), narrow ones where they would not.  The sums do
// not depend on the tile.  The epilogues bound the small layers, which want every SM; wide tiles read the
// row operand fewer times, which bounds the large ones.  4096 rows of 256 features: forward 64 wide 17 us
// a layer (128 CTAs; 128 wide 27), input gradient 64 wide 23 us (256 wide, 32 CTAs, 71), weight gradient
// 32 wide 20 us in 16 CTAs beside the input gradients (its K is the batch, a serial walk; 256 wide two
// CTAs of 27 us).  Inference of 65536 samples, 64 / 128 / 256 wide: width 512 445 / 407 / 462 us, width 2048
// 1127 / 894 / 954, width 4096 3132 / 2306 / 2384.  A training step of 4096 rows of 2048 features: input
// gradient 64 / 128 / 256 wide 592 / 541 / 519 us, weight gradient 32 / 64 / 128 / 256 wide 592 / 525 / 492 / 485.
template <int TN, int EPI>
struct Cfg {
    static constexpr int W_TILE = Tile<TN>::W_TILE;
    static constexpr int stage_bytes = A_TILE + W_TILE;
    static constexpr bool forward_layer = EPI == 1 || EPI == 2;   // TC_EPI_BIAS_GELU, TC_EPI_BIAS_OUT
    static constexpr int stages = forward_layer ? 2 : (192 * 1024) / stage_bytes;   // 2, or 4 (256 wide) .. 9 (32 wide)
    static constexpr int smem = stages * stage_bytes + 1024 /*align*/ + 256 /*barriers*/;
};

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Epilogue of one thread: row `row`, 32 accumulator columns starting at `col`.
template <int EPI>
__device__ __forceinline__ void epilogue32(const TcEpilogue& e, int M, int N, int row, int col, const uint32_t (&r)[32],
                                           float (&colsum)[32]) {
    const bool rok = row < M && row < e.rows_valid;
    if (EPI == TC_EPI_STORE) {
        if (!rok || col >= N) return;
        if (e.cols_valid >= N && (e.ldc % 4) == 0) {
            float4* dst = reinterpret_cast<float4*>(e.C + (size_t)row * e.ldc + col);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (col + 4 * q < N)
                    dst[q] = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                                         __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
        } else {
#pragma unroll
            for (int q = 0; q < 32; ++q)
                if (col + q < e.cols_valid) e.C[(size_t)row * e.ldc + col + q] = __uint_as_float(r[q]);
        }
    } else if (EPI == TC_EPI_BIAS_GELU) {
        // z = acc + b; keep z (for the backward pass, optional) and h = GELU(z) row-major and,
        // optionally, transposed.  N is a multiple of 32 and the rows of z and H are 16-byte aligned, so
        // a thread's 32 columns of z and h go out in 16-byte stores (a lane's row is a line of its own:
        // scalar ones cost a sector each).
        if (col >= N || row >= M) return;
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
            float z[8], h[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = col + q + u;
                z[u] = __uint_as_float(r[q + u]) + (c < e.cols_valid ? e.bias[c] : 0.f);
                // rows past the valid batch are written as zeros so that no stale value travels on
                h[u] = (rok && c < e.cols_valid) ? gelu(z[u]) : 0.f;
                if (e.HT) e.HT[(size_t)c * e.ldht + row] = __float2bfloat16_rn(h[u]);
            }
            if (e.C && rok) {
                float4* zd = reinterpret_cast<float4*>(e.C + (size_t)row * e.ldc + col + q);
                zd[0] = make_float4(z[0], z[1], z[2], z[3]);
                zd[1] = make_float4(z[4], z[5], z[6], z[7]);
            }
            *reinterpret_cast<uint4*>(e.H + (size_t)row * e.ldh + col + q) =
                make_uint4(pack2(h[0], h[1]), pack2(h[2], h[3]), pack2(h[4], h[5]), pack2(h[6], h[7]));
        }
    } else if (EPI == TC_EPI_BIAS_OUT) {
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            const int c = col + q;
            if (!rok || c >= e.cols_valid) break;
            const float z = __uint_as_float(r[q]) + e.bias[c];
            e.C[(size_t)row * e.ldc + c] = e.sigmoid ? 1.f / (1.f + expf(-z)) : z;
        }
    } else if (EPI == TC_EPI_GELU_BWD) {
        // dz = dh * GELU'(z) in both layouts (16-byte loads and stores along the row), plus per-column
        // sums for the bias gradient
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
            float z[8], dz[8];
            if (rok && col + q < N) {
                const float4* zs = reinterpret_cast<const float4*>(e.Zin + (size_t)row * e.ldz + col + q);
                const float4 lo = zs[0], hi = zs[1];
                z[0] = lo.x; z[1] = lo.y; z[2] = lo.z; z[3] = lo.w;
                z[4] = hi.x; z[5] = hi.y; z[6] = hi.z; z[7] = hi.w;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c = col + q + u;
                dz[u] = 0.f;
                if (rok && c < e.cols_valid) dz[u] = __uint_as_float(r[q + u]) * gelu_grad(z[u]);
                colsum[q + u] = dz[u];
                if (c < N && e.HT && row < M) e.HT[(size_t)c * e.ldht + row] = __float2bfloat16_rn(dz[u]);
            }
            if (col + q < N && row < M)
                *reinterpret_cast<uint4*>(e.H + (size_t)row * e.ldh + col + q) =
                    make_uint4(pack2(dz[0], dz[1]), pack2(dz[2], dz[3]), pack2(dz[4], dz[5]), pack2(dz[6], dz[7]));
        }
    }
}

// sums over the warp's lanes of 32 values per lane, value q to lane q: the exchange halves the values
// held at every step (31 shuffles; a tree per value is 160), and adds the same pairs as those trees
__device__ __forceinline__ float warp_colsums(float (&v)[32], int lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int q = 0; q < o; ++q) {
            const float mine = up ? v[q + o] : v[q], other = up ? v[q] : v[q + o];
            v[q] = mine + __shfl_xor_sync(0xffffffffu, other, o);
        }
    }
    return v[0];
}

template <int EPI, int TN>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mW, int M, int N, int K,
              const TcEpilogue e, int* err) {
    using CF = Cfg<TN, EPI>;
    constexpr int S = CF::stages;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;             // 1024 B alignment for the swizzle atoms
    uint8_t* gbase = smem_raw + (base - raw);
    const uint32_t bar0 = base + S * CF::stage_bytes;         // full[S], empty[S], done, tmem slot
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    const uint32_t done_bar = bar0 + 8u * (2 * S);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + S * CF::stage_bytes + 8 * (2 * S + 1));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * TN, m0 = blockIdx.y * TM;
    const int nk = K / TK;
    {   // an earlier launch gave up: skip (decided once per CTA, so that no thread is left at a barrier)
        __shared__ int s_abort;
        if (threadIdx.x == 0) s_abort = *(volatile int*)err;
        __syncthreads();
        if (s_abort) return;
    }

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    auto sA = [&](int s) { return base + s * CF::stage_bytes; };
    auto sW = [&](int s) { return base + s * CF::stage_bytes + A_TILE; };

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        int issued = 0;
        bool ok = true;
        for (int kb = 0; kb < nk && ok; ++kb) {
            const int s = kb % S;
            if (kb >= S) ok = mbar_wait(empty_bar(s), ((kb / S) - 1) & 1, err, 1);
            if (!ok) break;
            mbar_expect_tx(full_bar(s), CF::stage_bytes);
            const int kc = kb * TK;
            tma_load_2d(sA(s), &mA, kc, m0, full_bar(s));
            tma_load_2d(sW(s), &mW, kc, n0, full_bar(s));
            issued = kb + 1;
        }
        // drain: every stage armed so far must have landed before the CTA may exit
        for (int kb = (issued > S ? issued - S : 0); kb < issued; ++kb)
            mbar_drain(full_bar(kb % S), (kb / S) & 1, err, 2);
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer ----------------
        bool ok = true;
        for (int kb = 0; kb < nk && ok; ++kb) {
            const int s = kb % S;
            ok = mbar_wait(full_bar(s), (kb / S) & 1, err, 3);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int k = 0; k < TK / 16; ++k) {
                const uint32_t koff = 32u * k;
                mma_bf16<TN>(tmem, sw128_desc(sA(s) + koff), sw128_desc(sW(s) + koff), (kb > 0 || k > 0) ? 1u : 0u);
            }
            mma_commit(empty_bar(s));
        }
        mma_commit(done_bar);       // tracks every MMA issued above, also on the error path
    }
    __syncwarp();
    // ---------------- epilogue: TMEM -> registers -> global ----------------
    const bool have = mbar_drain(done_bar, 0, err, 4);   // also on the error path: MMAs land before TMEM is freed
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // tcgen05.ld is warp-collective: take the decision once per warp
    const int go = __shfl_sync(0xffffffffu, (have && *(volatile int*)err == 0) ? 1 : 0, 0);
    if (go) {
        const int quarter = warp & 3, half = warp >> 2;
        const int row = m0 + quarter * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
        for (int c = 32 * half; c < TN; c += 64) {
            uint32_t r[32];
            float colsum[32];
            tmem_ld32(lane_addr + (uint32_t)c, r);
            const int col = n0 + c;
            epilogue32<EPI>(e, M, N, row, col, r, colsum);
            if (EPI == TC_EPI_GELU_BWD && e.colsum && col < N) {
                // fixed-order warp sums -> one partial per (row block of 32, column)
                const float v = warp_colsums(colsum, lane);
                if (col + lane < N) e.colsum[(size_t)(blockIdx.y * 4 + quarter) * e.ldcs + col + lane] = v;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TN) : "memory");
    }
}

template <int EPI, int TN>
int launch(cudaStream_t s, int M, int N, int K, const __nv_bfloat16* A, const __nv_bfloat16* W, const TcEpilogue& e,
           int* err) {
    static bool configured = false;
    if (!configured) {
        BPM_CK(cudaFuncSetAttribute(k_gemm_tc<EPI, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    Cfg<TN, EPI>::smem));
        configured = true;
    }
    CUtensorMap mA, mW;
    BPM_TRY(make_bf16_tensor_map(&mA, A, K, M, TM));
    BPM_TRY(make_bf16_tensor_map(&mW, W, K, N, TN));
    dim3 grid((N + TN - 1) / TN, M / TM);
    k_gemm_tc<EPI, TN><<<grid, kThreads, Cfg<TN, EPI>::smem, s>>>(mA, mW, M, N, K, e, err);
    BPM_CK(cudaGetLastError());
    return BPM_OK;
}

}  // namespace

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

int make_bf16_tensor_map(CUtensorMap* map, const void* ptr, int inner, int rows, int box_rows, int box_inner) {
    if (box_inner != 64 && box_inner != 32) {
        set_error("TMA box depth must be 64 or 32 elements (got %d)", box_inner);
        return BPM_ERR_ARG;
    }
    EncodeTiledFn fn = encode_fn();
    if (!fn) {
        set_error("cuTensorMapEncodeTiled is not available from the driver");
        return BPM_ERR_CUDA;
    }
    if ((reinterpret_cast<uintptr_t>(ptr) & 15u) || (inner % 8)) {
        set_error("TMA operand not 16-byte aligned (ptr %p, inner %d)", ptr, inner);
        return BPM_ERR_ARG;
    }
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)inner * 2};
    // rows of box_inner BF16 elements: 128 B rows with the 128-byte swizzle, 64 B rows with the 64-byte one
    cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    const CUtensorMapSwizzle sw = box_inner == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d)", (int)r);
        return BPM_ERR_CUDA;
    }
    return BPM_OK;
}

// the widest column tile, halved from `most` down to `least`, of which the M x N outputs have `ctas` or more
static int tile_width(int M, int N, int most, int least, int ctas) {
    int t = most;
    while (t > least && (long long)(M / tc::TM) * ((N + t - 1) / t) < ctas) t /= 2;
    return t;
}

int gemm_tc(cudaStream_t s, int epi, int M, int N, int K, const __nv_bfloat16* A, const __nv_bfloat16* W,
            const TcEpilogue& e, int sm_count, int* err_flag) {
    if (M % TM || K % TK || N % 16 || M <= 0 || N <= 0) {
        set_error("tensor-core GEMM needs M %% %d == 0, K %% %d == 0, N %% 16 == 0 (M=%d N=%d K=%d)", TM, TK, M, N, K);
        return BPM_ERR_ARG;
    }
    // The forward layers alone on the GPU take 128 columns where that gives every SM a CTA (128 CTAs: width
    // 512 at 4096 rows 108 us 64 wide, 111 so; 256 CTAs: 134 and 123).  The gradients share it, and take the widest
    // tile with a CTA for every second SM (64 CTAs of 256 columns, width 1024 at 2048 rows: 271 us a step, 259 at
    // 128; 128 CTAs, 4096 rows: 372 and 386).
    switch (epi) {
        case TC_EPI_STORE:
            switch (tile_width(M, N, 256, 32, sm_count / 2)) {
                case 256: return launch<TC_EPI_STORE, 256>(s, M, N, K, A, W, e, err_flag);
                case 128: return launch<TC_EPI_STORE, 128>(s, M, N, K, A, W, e, err_flag);
                case 64: return launch<TC_EPI_STORE, 64>(s, M, N, K, A, W, e, err_flag);
                default: return launch<TC_EPI_STORE, 32>(s, M, N, K, A, W, e, err_flag);
            }
        case TC_EPI_BIAS_GELU:
            return tile_width(M, N, 128, 64, sm_count) == 128
                       ? launch<TC_EPI_BIAS_GELU, 128>(s, M, N, K, A, W, e, err_flag)
                       : launch<TC_EPI_BIAS_GELU, 64>(s, M, N, K, A, W, e, err_flag);
        case TC_EPI_BIAS_OUT: return launch<TC_EPI_BIAS_OUT, 128>(s, M, N, K, A, W, e, err_flag);
        case TC_EPI_GELU_BWD:
            switch (tile_width(M, N, 256, 64, sm_count / 2)) {
                case 256: return launch<TC_EPI_GELU_BWD, 256>(s, M, N, K, A, W, e, err_flag);
                case 128: return launch<TC_EPI_GELU_BWD, 128>(s, M, N, K, A, W, e, err_flag);
                default: return launch<TC_EPI_GELU_BWD, 64>(s, M, N, K, A, W, e, err_flag);
            }
        default: set_error("unknown epilogue %d", epi); return BPM_ERR_ARG;
    }
}

}  // namespace bpm
