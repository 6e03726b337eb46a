// Surrogate forward pass in one kernel (tcgen05, sm_103a), for networks up to 256 wide.
//
// Layer by layer the forward pass wrote 128 MB of activations a layer and read them back, each layer a
// launch of its own: 262144 samples took 772 us, of which the matrix products are 55 us.  Here a CTA
// (one per SM) carries tiles of 128 samples through every layer: the activations stay in shared memory
// (BF16, the MMA's A operand), the accumulators in TMEM, and only inputs and results touch HBM.  Two
// tiles are in flight, so that one tile's products and weight loads run under the other's epilogue.
// Warp roles:
//   warps 0-15  inputs (FP32 -> BF16) into a tile's activations, then per layer bias + GELU of its
//               accumulator back into them; warp w takes rows 32 (w % 4) .. and columns 64 (w / 4) ..,
//               one 64-column k-block of the next layer's operand; last layer: logits or probabilities
//   warp 16     streams the weights, a k-block (64 columns of W_l) per stage of a three-stage ring, once
//               per tile and layer: 0.45 MB a tile from L2
//   warp 17     TMEM and the MMAs
// The bound is the erf-form GELU with its bias and conversions, about 35 instructions for each of the 1024
// hidden values of a sample.  262144 samples: 352 us (452 with a column test and a scalar bias load per
// value).  The products, their order and the roundings between layers are those of
// the layer-by-layer path (bpm_gemm_tc.cu), so the results are bitwise its own.
// Waits are bounded as in the other tensor-core kernels.
#include <algorithm>

#include "bpm_mlp_forward.cuh"
#include "bpm_tc_ptx.cuh"

namespace bpm {

namespace {

using namespace tc;

constexpr int kFThreads = 18 * 32, kFEpiWarps = 16, kFSlots = 2, kFStages = 3;
constexpr int kActBytes = 4 * A_TILE;                     // 128 rows x 256 columns
constexpr int kStageBytes = 256 * TK * 2;                 // 256 weight rows x 64 columns
constexpr int kFwdSmem = kFSlots * kActBytes + kFStages * kStageBytes + 1024 + 256;

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }

__device__ __forceinline__ void st_shared16(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// shared address of columns 8 q .. 8 q + 7 of a row of k-block kb (128-byte rows, 128-byte swizzle)
__device__ __forceinline__ uint32_t act_addr(uint32_t act, int kb, int row, int q) {
    return act + (uint32_t)(kb * A_TILE + row * 128 + ((q ^ (row & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}

__global__ void __launch_bounds__(kFThreads, 1) k_mlp_forward(const __grid_constant__ MlpForward p, int* err) {
    extern __shared__ uint8_t smem_raw[];
    {   // an earlier launch gave up: skip (decided once per CTA, so that no thread is left at a barrier)
        __shared__ int s_abort;
        if (threadIdx.x == 0) s_abort = *(volatile int*)err;
        __syncthreads();
        if (s_abort) return;
    }
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t ring = base + kFSlots * kActBytes;
    const uint32_t bar0 = ring + kFStages * kStageBytes;
    auto act = [&](int s) { return base + (uint32_t)(s * kActBytes); };
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kFStages + s); };
    auto act_bar = [&](int s) { return bar0 + 8u * (2 * kFStages + s); };
    auto acc_bar = [&](int s) { return bar0 + 8u * (2 * kFStages + kFSlots + s); };
    const uint32_t done_bar = bar0 + 8u * (2 * kFStages + 2 * kFSlots);
    uint32_t* tmem_slot =
        reinterpret_cast<uint32_t*>(smem_raw + (bar0 - raw) + 8 * (2 * kFStages + 2 * kFSlots + 1));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kFStages; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int s = 0; s < kFSlots; ++s) {
            mbar_init(act_bar(s), kFEpiWarps);
            mbar_init(acc_bar(s), 1);
        }
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 17) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int tiles = (int)((p.N + TM - 1) / TM);

    if (warp < kFEpiWarps) {
        const int quarter = warp & 3, cg = warp >> 2, row = 32 * quarter + lane;
        int unit[kFSlots] = {0, 0};                        // accumulators of the slot read so far
        bool ok = true;
        for (long long t0 = blockIdx.x; t0 < tiles && ok; t0 += (long long)kFSlots * gridDim.x) {
            const int ns = t0 + gridDim.x < tiles ? 2 : 1;
            for (int s = 0; s < ns; ++s) {
                // inputs of the slot's next tile; its activations are free (the last layer's MMAs are done)
                const long long r0 = (t0 + (long long)s * gridDim.x) * TM;
                const int chunks = p.k_pad[0] / 8;
                for (int e = threadIdx.x; e < TM * chunks; e += 32 * kFEpiWarps) {
                    const int r = e / chunks, q = e % chunks;
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int c = 8 * q + u;
                        v[u] = c < p.n_in && r0 + r < p.N ? __ldg(p.X + (r0 + r) * p.n_in + c) : 0.f;
                    }
                    st_shared16(act_addr(act(s), q >> 3, r, q & 7),
                                make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                                           pack_bf16(v[6], v[7])));
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(act_bar(s));
            }
            for (int l = 0; l < p.L && ok; ++l)
                for (int s = 0; s < ns && ok; ++s) {
                    const bool have = mbar_wait(acc_bar(s), unit[s] & 1, err, 24);
                    ++unit[s];
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    ok = __shfl_sync(0xffffffffu, have ? 1 : 0, 0) != 0;
                    if (!ok) break;
                    const uint32_t lane_addr = tmem + (uint32_t)(256 * s) + ((uint32_t)(32 * quarter) << 16);
                    const float* bias = p.bias[l];
                    const int nr = p.n_real[l];
                    if (l + 1 < p.L) {
                        // 64 real columns with their biases on a 16-byte boundary (layers of 4 n columns)
                        const bool whole = 64 * cg + 64 <= nr && (reinterpret_cast<uintptr_t>(bias) & 15) == 0;
                        if (64 * cg < p.n_pad[l])
#pragma unroll 1
                            for (int h = 0; h < 2; ++h) {
                                uint32_t r[32];
                                const int c0 = 64 * cg + 32 * h;
                                tmem_ld32(lane_addr + (uint32_t)c0, r);
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    float v[8];
                                    if (whole) {
                                        const float4* b4 = reinterpret_cast<const float4*>(bias + c0 + 8 * q);
                                        const float4 lo = __ldg(b4), hi = __ldg(b4 + 1);
                                        const float bv[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                                        for (int u = 0; u < 8; ++u) v[u] = gelu(__uint_as_float(r[8 * q + u]) + bv[u]);
                                    } else {
#pragma unroll
                                        for (int u = 0; u < 8; ++u) {
                                            const int c = c0 + 8 * q + u;
                                            v[u] = 0.f;
                                            if (c < nr) v[u] = gelu(__uint_as_float(r[8 * q + u]) + __ldg(bias + c));
                                        }
                                    }
                                    st_shared16(act_addr(act(s), cg, row, 4 * h + q),
                                                make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]),
                                                           pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7])));
                                }
                            }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(act_bar(s));
                    } else {
                        const long long gr = (t0 + (long long)s * gridDim.x) * TM + row;
#pragma unroll 1
                        for (int c0 = 32 * cg; c0 < nr; c0 += 128) {
                            uint32_t r[32];
                            tmem_ld32(lane_addr + (uint32_t)c0, r);
                            if (gr < p.N)
#pragma unroll
                                for (int u = 0; u < 32; ++u)
                                    if (c0 + u < nr) {
                                        const float z = __uint_as_float(r[u]) + __ldg(bias + c0 + u);
                                        p.out[gr * nr + c0 + u] = p.sigmoid ? 1.f / (1.f + expf(-z)) : z;
                                    }
                        }
                    }
                }
        }
    } else if (warp == 16 && lane == 0) {
        // ---------------- weights ----------------
        int kbg = 0;
        bool ok = true;
        for (long long t0 = blockIdx.x; t0 < tiles && ok; t0 += (long long)kFSlots * gridDim.x) {
            const int ns = t0 + gridDim.x < tiles ? 2 : 1;
            for (int l = 0; l < p.L && ok; ++l)
                for (int s = 0; s < ns && ok; ++s)
                    for (int kb = 0; kb < p.k_pad[l] / TK; ++kb, ++kbg) {
                        const int st = kbg % kFStages;
                        if (kbg >= kFStages) ok = mbar_wait(empty_bar(st), ((kbg / kFStages) - 1) & 1, err, 21);
                        if (!ok) break;
                        mbar_expect_tx(full_bar(st), (uint32_t)(p.n_mma[l] * TK * 2));
                        tma_load_2d(ring + (uint32_t)(st * kStageBytes), &p.w[l], kb * TK, 0, full_bar(st));
                    }
        }
        // drain: the last armed phase of every stage must land before exit
        for (int k = (kbg > kFStages ? kbg - kFStages : 0); k < kbg; ++k)
            mbar_drain(full_bar(k % kFStages), (k / kFStages) & 1, err, 22);
    } else if (warp == 17 && lane == 0) {
        // ---------------- MMAs ----------------
        int kbg = 0, unit[kFSlots] = {0, 0};
        bool ok = true;
        for (long long t0 = blockIdx.x; t0 < tiles && ok; t0 += (long long)kFSlots * gridDim.x) {
            const int ns = t0 + gridDim.x < tiles ? 2 : 1;
            for (int l = 0; l < p.L && ok; ++l) {
                const uint32_t idesc = idesc_n<256>(p.n_mma[l]);
                for (int s = 0; s < ns && ok; ++s) {
                    ok = mbar_wait(act_bar(s), unit[s] & 1, err, 23);
                    ++unit[s];
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    for (int kb = 0; kb < p.k_pad[l] / TK; ++kb, ++kbg) {
                        const int st = kbg % kFStages;
                        ok = mbar_wait(full_bar(st), (kbg / kFStages) & 1, err, 25);
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                        for (int k = 0; k < TK / 16; ++k)
                            mma_bf16_desc(tmem + (uint32_t)(256 * s),
                                          sw128_desc(act(s) + (uint32_t)(kb * A_TILE) + 32u * k),
                                          sw128_desc(ring + (uint32_t)(st * kStageBytes) + 32u * k), idesc,
                                          (kb > 0 || k > 0) ? 1u : 0u);
                        mma_commit(empty_bar(st));
                    }
                    if (ok) mma_commit(acc_bar(s));
                }
            }
        }
        mma_commit(done_bar);       // tracks every MMA issued above, also on the error path
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 17) {
        mbar_drain(done_bar, 0, err, 26);     // every MMA has completed before TMEM is released
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

}  // namespace

bool mlp_forward_fits(int L, const int* k_pad, const int* n_pad) {
    if (L < 2 || L > kMaxMlpLayers) return false;
    for (int l = 0; l < L; ++l)
        if (k_pad[l] > 256 || n_pad[l] > 256) return false;
    return true;
}

int mlp_forward_launch(cudaStream_t s, const MlpForward& p, int sm_count, int* err) {
    BPM_CK(cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem));
    const long long tiles = (p.N + tc::TM - 1) / tc::TM;
    if (tiles > (1 << 30)) {
        set_error("surrogate batch of %lld samples", p.N);
        return BPM_ERR_ARG;
    }
    k_mlp_forward<<<(int)std::min<long long>(tiles, sm_count), kFThreads, kFwdSmem, s>>>(p, err);
    BPM_CK(cudaGetLastError());
    return BPM_OK;
}

}  // namespace bpm
