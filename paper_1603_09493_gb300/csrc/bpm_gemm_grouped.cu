// Persistent, grouped demag GEMM on the tensor cores (tcgen05, sm_103a).
//
// One launch computes, for every mesh group g of a batch (uneven mesh sizes),
//   C_g[M_g][N_g] = sum of the BF16 split products of A_g[M_g][K_g] and W_g[N_g][K_g]^T
// (3 products hi*hi + lo*hi + hi*lo, or 1), FP32 accumulate in TMEM: M_g islands,
// N_g = K_g operator rows.  The operator's rows are the MMA's M side (128 a tile),
// the islands its N side, nb of them a tile, any multiple of 16 up to TN.  Island
// counts are what varies (one island to thousands, ragged over design variants),
// and an MMA costs nearly in proportion to N, so no tile computes padding beyond
// 15 islands (with the islands on the M side a group of 135 took 256 rows: eight
// design variants of 135 islands 35.1 ms an interval, 30.2 so).  A tile's accumulator holds operator rows in lanes, so a warp
// stores 128 contiguous bytes of an island's field per instruction.
//
// K is cut into up to four slices (gemm_slices), from K alone, and an element is the
// sum of its slices in order, so that an island's field has the same bits in every
// batch, whatever else is in it and whichever kernel forms it.  A group of at most
// 128 islands has only N_g / 128 tiles, each a serial walk over K: there a slice is
// an item of its own writing its own plane of C, and the stage kernels add the
// planes (one island of 209 nodes: 374 -> 172 us an interval of 6 steps; nine of 481
// nodes: 689 -> 330 us of 8 steps; 60 of 1547 nodes: 5.2 -> 2.7 ms of 28 steps).
// Otherwise an item is a tile's whole K: the slices go to the two accumulators in
// turn, and the epilogue adds them in registers (eight warps of 128 sums a thread, no
// store before the accumulator is free again; against four warps that stored as they
// read, one sum of all of K: an interval of 4096 islands of 1547 nodes 24.3 -> 23.9 ms,
// of 600 of 481 nodes 606 -> 556 us).
//
// The items of all groups are dealt to the CTAs (one per SM) when the GEMM is set
// up: an item costs its K, so each goes, longest first, to the CTA with the least
// so far (a walk of the list with the grid as stride left the longest items of
// eight uneven variants to the last, two-thirds full round: 31.1 ms an interval,
// 30.9 so, the product then being bound by reading 1.6 GB of operators).  Items of
// equal cost keep the list's order, one after the other over the CTAs.  Within a group the tiles run M-major or N-major (chosen
// per group), so that a wave of CTAs shares the larger operand's rows in L2 and it
// is read from HBM once.  Warp roles:
//   warp 0  one lane streams the k-blocks of every item with TMA into a ring of
//           shared-memory stages (the ring runs across item boundaries);
//   warp 1  allocates two TMEM accumulators; one lane issues the MMAs, slice i of
//           the CTA's items into accumulator i % 2;
//   warps 2-9  read an accumulator back (tcgen05.ld; a warp 32 operator rows by half of
//           the tile's islands), add an item's slices and store them, while the MMAs
//           of the next slice run into the other accumulator.
// Per-group tensor maps live in a device array (64-byte aligned entries).
// Every wait is bounded; on timeout the kernel raises the error flag, drains
// its copies and MMAs, frees TMEM and exits, and later launches return at once.
// The waits of normal progress take the launch's limit (wait_ns); the drains
// always take the fixed limit, so that copies and MMAs land before shared
// memory or TMEM is given up.
#include <algorithm>
#include <cstring>
#include <functional>
#include <queue>

#include "bpm_tc_ptx.cuh"

namespace bpm {

namespace {

using namespace tc;

constexpr int kGThreads = 320, kGEpiWarps = 8;

// KB: K depth of a stage (64: 128 B rows, 128-byte swizzle; 32: 64 B rows, 64-byte swizzle)
// TN: islands per tile at most
template <int P, int TN, int KB>
struct GCfg {
    static constexpr int W_BYTES = TM * KB * 2;
    static constexpr int A_BYTES = TN * KB * 2;
    static constexpr int stage_bytes = (P == 3 ? 2 : 1) * (A_BYTES + W_BYTES);
    static constexpr int stages = (192 * 1024) / stage_bytes;
    static constexpr int smem = stages * stage_bytes + 1024 + 256;
    static_assert(8 * (2 * stages + 5) + 4 <= 256, "barrier area");
};

template <int KB>
__device__ __forceinline__ uint64_t kmajor_desc(uint32_t addr) {
    return KB == 64 ? sw128_desc(addr) : sw64_desc(addr);
}

__device__ __forceinline__ int find_group(const GemmGroupDev* __restrict__ G, int ng, int t) {
    int g = 0;
    while (g + 1 < ng && t >= G[g + 1].tile_begin) ++g;
    return g;
}

// item it of group gg -> first island, first operator row, slice of K that it begins with (0 if it has all)
__device__ __forceinline__ void item_origin(const GemmGroupDev& gg, int it, int& b0, int& r0, int& slice) {
    slice = it % gg.splits;
    const int lt = it / gg.splits;
    const int mt = gg.n_major ? lt % gg.tiles_m : lt / gg.tiles_n;
    const int nt = gg.n_major ? lt / gg.tiles_m : lt % gg.tiles_n;
    b0 = mt * gg.nb;
    r0 = nt * TM;
}

template <int P, int TN, int KB>
__global__ void __launch_bounds__(kGThreads, 1)
    k_gemm_grouped(const GemmGroupDev* __restrict__ G, int ng, const int* __restrict__ sched, int* err,
                   unsigned long long wait_ns) {
    using CF = GCfg<P, TN, KB>;
    constexpr int S = CF::stages;
    constexpr int A_TILE = CF::A_BYTES;
    constexpr int W_TILE = CF::W_BYTES;
    extern __shared__ uint8_t smem_raw[];
    {   // an earlier launch gave up: skip (decided once per CTA, so that no thread is left at a barrier)
        __shared__ int s_abort;
        pdl_trigger();
        if (threadIdx.x == 0) s_abort = *(volatile int*)err;
        __syncthreads();
        if (s_abort) {
            pdl_wait();
            return;
        }
    }
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - raw);
    const uint32_t bar0 = base + S * CF::stage_bytes;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
    auto accf_bar = [&](int a) { return bar0 + 8u * (2 * S + a); };
    auto acce_bar = [&](int a) { return bar0 + 8u * (2 * S + 2 + a); };
    const uint32_t done_bar = bar0 + 8u * (2 * S + 4);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + S * CF::stage_bytes + 8 * (2 * S + 5));
    auto sWhi = [&](int s) { return base + s * CF::stage_bytes; };
    auto sAhi = [&](int s) { return base + s * CF::stage_bytes + W_TILE; };
    auto sWlo = [&](int s) { return base + s * CF::stage_bytes + W_TILE + A_TILE; };
    auto sAlo = [&](int s) { return base + s * CF::stage_bytes + 2 * W_TILE + A_TILE; };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this CTA's items: sched holds gridDim.x + 1 offsets into the list behind them
    const int* items = sched + gridDim.x + 1;
    const int q0 = sched[blockIdx.x], q1 = sched[blockIdx.x + 1];
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(accf_bar(a), 1);
            mbar_init(acce_bar(a), kGEpiWarps);     // one arrival per epilogue warp
        }
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(2 * TN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        int kbg = 0;
        bool ok = true;
        for (int qi = q0; qi < q1 && ok; ++qi) {
            const int t = items[qi];
            const int g = find_group(G, ng, t);
            const GemmGroupDev& gg = G[g];
            int b0, r0, sl;
            item_origin(gg, t - gg.tile_begin, b0, r0, sl);
            const int kb1 = min(gg.K, (sl + gg.segs) * gg.slice_k) / KB;
            const uint32_t bytes = (P == 3 ? 2u : 1u) * (uint32_t)(W_TILE + gg.nb * KB * 2);
            int kb = sl * gg.slice_k / KB;
            auto load_w = [&](int s, int kc) {
                mbar_expect_tx(full_bar(s), bytes);
                tma_load_2d(sWhi(s), &gg.whi, kc, r0, full_bar(s));
                if (P == 3) tma_load_2d(sWlo(s), &gg.wlo, kc, r0, full_bar(s));
            };
            auto load_a = [&](int s, int kc) {
                tma_load_2d(sAhi(s), &gg.ahi, kc, b0, full_bar(s));
                if (P == 3) tma_load_2d(sAlo(s), &gg.alo, kc, b0, full_bar(s));
            };
            if (qi == q0) {
                // the first ring of operator tiles, which no kernel writes, ahead of the wait for the
                // kernel that writes the islands' operand
                const int pre = min(S, kb1 - kb);
                for (int s = 0; s < pre; ++s) load_w(s, (kb + s) * KB);
                pdl_wait();
                for (int s = 0; s < pre; ++s) load_a(s, (kb + s) * KB);
                kb += pre;
                kbg = pre;
            }
            for (; kb < kb1; ++kb, ++kbg) {
                const int s = kbg % S;
                if (kbg >= S) ok = mbar_wait(empty_bar(s), ((kbg / S) - 1) & 1, err, 11, true, wait_ns);
                if (!ok) break;
                load_w(s, kb * KB);
                load_a(s, kb * KB);
            }
        }
        // drain: the last armed phase of every stage must land before exit
        const int armed = kbg;
        for (int k = (armed > S ? armed - S : 0); k < armed; ++k) mbar_drain(full_bar(k % S), (k / S) & 1, err, 12);
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer ----------------
        int kbg = 0, i = 0;
        bool ok = true;
        for (int qi = q0; qi < q1 && ok; ++qi) {
            const int t = items[qi];
            const int g = find_group(G, ng, t);
            const GemmGroupDev& gg = G[g];
            int b0, r0, sl;
            item_origin(gg, t - gg.tile_begin, b0, r0, sl);
            const uint32_t idesc = idesc_n<TN>(gg.nb);
            for (int u = sl; u < sl + gg.segs && ok; ++u, ++i) {
                const int kb0 = u * gg.slice_k / KB, kb1 = min(gg.K, (u + 1) * gg.slice_k) / KB;
                const int a = i & 1;
                if (i >= 2) ok = mbar_wait(acce_bar(a), ((i >> 1) - 1) & 1, err, 13, true, wait_ns);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem + (uint32_t)(a * TN);
                for (int kb = kb0; kb < kb1; ++kb, ++kbg) {
                    const int s = kbg % S;
                    ok = mbar_wait(full_bar(s), (kbg / S) & 1, err, 14, true, wait_ns);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (int k = 0; k < KB / 16; ++k) {
                        const uint32_t koff = 32u * k;    // 16 BF16 further along the swizzled row
                        const uint64_t ahi = kmajor_desc<KB>(sAhi(s) + koff), whi = kmajor_desc<KB>(sWhi(s) + koff);
                        mma_bf16_desc(acc, whi, ahi, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
                        if (P == 3) {
                            const uint64_t alo = kmajor_desc<KB>(sAlo(s) + koff), wlo = kmajor_desc<KB>(sWlo(s) + koff);
                            mma_bf16_desc(acc, whi, alo, idesc, 1u);
                            mma_bf16_desc(acc, wlo, ahi, idesc, 1u);
                        }
                    }
                    mma_commit(empty_bar(s));
                }
                if (ok) mma_commit(accf_bar(a));
            }
        }
        mma_commit(done_bar);      // tracks every MMA issued above, also on the error path
    } else if (warp >= 2) {
        // ---------------- epilogue warps ----------------
        const int q = warp & 3;    // TMEM lane quarter this warp may access
        const int h0 = (warp - 2) / 4 * (TN / 2);          // its islands of the tile: h0 .. h0 + TN / 2
        constexpr int NC = TN / 32;                        // in pieces of 16
        pdl_wait();                // C may still be read by the kernel before
        int i = 0;
        bool go = true;
        for (int qi = q0; qi < q1 && go; ++qi) {
            const int t = items[qi];
            const int g = find_group(G, ng, t);
            const GemmGroupDev& gg = G[g];
            int b0, r0, sl;
            item_origin(gg, t - gg.tile_begin, b0, r0, sl);
            const int row = r0 + q * 32 + lane;             // operator row = column of C
            const int nv = min(gg.nb, gg.M - b0) - h0;      // islands of this tile from h0 on
            float sum[NC][16];
            for (int u = 0; u < gg.segs; ++u, ++i) {
                const int a = i & 1;
                const bool have = mbar_wait(accf_bar(a), (i >> 1) & 1, err, 15, true, wait_ns);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                go = __shfl_sync(0xffffffffu, (have && *(volatile int*)err == 0) ? 1 : 0, 0) != 0;
                if (!go) break;
                const uint32_t lane_addr = tmem + (uint32_t)(a * TN + h0) + ((uint32_t)(q * 32) << 16);
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (16 * c < nv) tmem_sum16(lane_addr + 16u * c, u > 0, sum[c]);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(acce_bar(a));
            }
            if (!go || row >= gg.N) continue;
            float* dst = gg.C + (size_t)sl * gg.plane + (size_t)(b0 + h0) * gg.ldc + row;
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (16 * c < nv)                            // (one island: 16 guarded stores, not all)
#pragma unroll
                    for (int v = 0; v < 16; ++v)
                        if (16 * c + v < nv) dst[(size_t)(16 * c + v) * gg.ldc] = sum[c][v];
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        mbar_drain(done_bar, 0, err, 16);     // every MMA has completed before TMEM is released
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TN) : "memory");
    }
}

template <int P, int TN, int KB>
int launch_grouped(cudaStream_t s, const GroupedGemm& gg, int* err, bool pdl) {
    static bool configured = false;
    if (!configured) {
        BPM_CK(cudaFuncSetAttribute(k_gemm_grouped<P, TN, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    GCfg<P, TN, KB>::smem));
        configured = true;
    }
    BPM_CK(launch_pdl(k_gemm_grouped<P, TN, KB>, dim3(gg.grid), dim3(kGThreads), GCfg<P, TN, KB>::smem, s, pdl,
                      gg.d_groups, gg.n_groups, gg.d_sched, err, gg.wait_ns ? gg.wait_ns : kWaitNs));
    return BPM_OK;
}

}  // namespace

int gemm_slices(int K, int sm_count) {
    const int tiles = (K + tc::TM - 1) / tc::TM, kb = K / tc::TK;
    // slices of at least three k-blocks, at most four (the consumers read every plane), no more items than SMs
    const int want = std::max(1, std::min({4, sm_count / tiles, (kb + 2) / 3}));
    const int per = (kb + want - 1) / want;
    return (kb + per - 1) / per;
}

namespace {

// Time of an MMA of nb islands relative to a 256-wide one's 256: N / 2 cycles of tensor work, or the
// 128 operator rows and nb island rows of 32 B that it reads from shared memory at 128 B a cycle
int mma_cost(int nb) { return std::max(nb, 64 + nb / 2); }

// Islands per tile of a group of M islands when no tile may exceed cap: even tiles, a multiple of 16
int even_tile(int M, int cap) {
    const int t = (M + cap - 1) / cap;
    return (((M + t - 1) / t) + 15) / 16 * 16;
}

// Islands per tile at most (256 .. 16): the cap with the least of
//   - the time of the busiest SM: waves of items x cost of an item (k-steps x MMA cost, an item's fixed cost
//     as 12 k-steps), and
//   - ten times the launch's own use of the chip, the rows its items read (128 + islands each) as if spread
//     over every SM: what it takes from the stage kernels, other chains and other batches beside it.
// Wide tiles win ties.  The second term decides where narrow tiles would read the operator again for each.
// Without it (the tile that is fastest alone) 200 islands of 1547 nodes took 148 items of 64: an interval
// 4.25 ms alone but 3.80 with three batches in turn on as many streams (each a pass), against 4.22 and 2.13 so;
// 512 islands 5.26 and 4.26 against 5.79 and 3.24; nine hundred of 481 nodes 0.64 and 0.52 against 0.73
// and 0.35; 1318 of 209 nodes 0.41 and 0.29 against 0.46 and 0.23.
// share > 1: the product runs beside share - 1 others on as many streams and takes no whole waves (an SM
// takes the others' work next).
int tile_cap(const std::vector<GemmOperands>& ops, int tile_n, int sm_count, int share) {
    int best = tile_n;
    double best_t = 1e300;
    for (int cap : {256, 208, 160, 128, 96, 64, 48, 32, 16}) {
        if (cap > tile_n) continue;
        long long items = 0;
        double sum = 0, top = 0, rows = 0;
        for (const GemmOperands& o : ops) {
            const int nb = even_tile(o.M, cap);
            const long long it = (long long)((o.M + nb - 1) / nb) * ((o.N + tc::TM - 1) / tc::TM) * o.planes;
            const double steps = o.K / 16.0 / o.planes + 12.0, c = mma_cost(nb) * steps;
            items += it;
            sum += it * c;
            rows += it * steps * (128 + nb) / 1.5;          // in the MMA's units at 256 islands
            top = std::max(top, c);
        }
        const double waves = (double)items * share / sm_count;
        const double busy = std::max(top, (share > 1 ? waves : std::ceil(waves)) * sum / (double)items);
        const double t = busy + 10.0 * rows / sm_count;
        if (t < best_t * 0.98) {
            best_t = t;
            best = cap;
        }
    }
    return best;
}

// Offsets [grid + 1] of each CTA's items, then the items: longest first (list order among equals), each
// to the CTA with the least cost so far (the lowest index among equals); an item costs the MMAs of its
// slice and a fixed part (see tile_cap)
std::vector<int> deal_items(const std::vector<GemmGroupDev>& h, int items, int grid) {
    struct Item {
        double cost;
        int it;
    };
    std::vector<Item> list;
    list.reserve(items);
    for (const GemmGroupDev& g : h)
        for (int k = 0; k < g.tiles_m * g.tiles_n * g.splits; ++k) {
            const int lo = (k % g.splits) * g.slice_k, hi = std::min(g.K, lo + g.segs * g.slice_k);
            list.push_back(Item{mma_cost(g.nb) * ((hi - lo) / 16.0 + 12.0), g.tile_begin + k});
        }
    std::stable_sort(list.begin(), list.end(), [](const Item& x, const Item& y) { return x.cost > y.cost; });
    std::vector<std::vector<int>> of(grid);
    std::priority_queue<std::pair<double, int>, std::vector<std::pair<double, int>>, std::greater<>> load;
    for (int c = 0; c < grid; ++c) load.push({0.0, c});
    for (const Item& x : list) {
        const auto [l, c] = load.top();
        load.pop();
        of[c].push_back(x.it);
        load.push({l + x.cost, c});
    }
    std::vector<int> out(1, 0);
    for (const auto& v : of) out.push_back(out.back() + (int)v.size());
    for (const auto& v : of) out.insert(out.end(), v.begin(), v.end());
    return out;
}

}  // namespace

int grouped_gemm_setup(GroupedGemm* gg, const std::vector<GemmOperands>& ops, int tile_n, int products, int raster,
                       int k_block, int sm_count, int pair, int share) {
    if (pair && tile_n != 256) {
        set_error("the CTA-pair GEMM computes 256 x 256 tiles (tile_n 256)");
        return BPM_ERR_ARG;
    }
    if (k_block != 64 && k_block != 32) {
        set_error("grouped GEMM k-block must be 64 or 32");
        return BPM_ERR_ARG;
    }
    if (tile_n != 128 && tile_n != 256) {
        set_error("grouped GEMM tile width must be 128 or 256");
        return BPM_ERR_ARG;
    }
    if (raster != BPM_RASTER_AUTO && raster != BPM_RASTER_M && raster != BPM_RASTER_N) {
        set_error("unknown GEMM raster %d", raster);
        return BPM_ERR_ARG;
    }
    std::vector<GemmGroupDev> h(ops.size());
    int tiles = 0, nb_max = 16;
    const int cap = tile_cap(ops, tile_n, sm_count, share);
    for (const GemmOperands& o : ops)
        if (o.M > 0) nb_max = std::max(nb_max, even_tile(o.M, cap));
    // Tiles of up to 128 islands leave room for three or four stages of 64-deep k-blocks, which read 128 bytes
    // of a row at a time and take half the barriers: an interval of one island of 1547 nodes 1256 -> 1139 us,
    // of 60 islands 1655 -> 1522, of eight uneven variants of 14 islands 24.2 -> 23.7 ms.  Wider tiles hold one such
    // stage only (1024 islands 6.64 ms at 32, 7.00 at 64).
    if (!pair && nb_max <= 128) k_block = 64;
    for (size_t g = 0; g < ops.size(); ++g) {
        const GemmOperands& o = ops[g];
        if (o.rows % tc::TM || o.K % tc::TK || o.N % 16 || o.M <= 0 || o.M > o.rows || o.N <= 0 || o.slices < 1 ||
            (o.planes != 1 && o.planes != o.slices)) {
            set_error("grouped GEMM group %zu: rows %% 128, K %% 64, N %% 16 required (M=%d rows=%d N=%d K=%d)", g,
                      o.M, o.rows, o.N, o.K);
            return BPM_ERR_ARG;
        }
        std::memset(&h[g], 0, sizeof(GemmGroupDev));
        const int nb = even_tile(o.M, cap);
        // a CTA of a pair stages 128 of the tile's 256 rows of either operand
        const int a_box = pair ? tc::TM : nb;
        BPM_TRY(make_bf16_tensor_map(&h[g].ahi, o.Ahi, o.K, o.rows, a_box, k_block));
        BPM_TRY(make_bf16_tensor_map(&h[g].whi, o.Whi, o.K, o.N, tc::TM, k_block));
        if (products == 3) {
            BPM_TRY(make_bf16_tensor_map(&h[g].alo, o.Alo, o.K, o.rows, a_box, k_block));
            BPM_TRY(make_bf16_tensor_map(&h[g].wlo, o.Wlo, o.K, o.N, tc::TM, k_block));
        } else {
            h[g].alo = h[g].ahi;
            h[g].wlo = h[g].whi;
        }
        h[g].C = o.C;
        h[g].M = pair ? o.rows : o.M;
        h[g].N = o.N;
        h[g].K = o.K;
        h[g].ldc = o.N;
        h[g].nb = nb;
        h[g].splits = pair ? 1 : o.planes;
        h[g].segs = o.slices / h[g].splits;
        h[g].slice_k = (o.K / tc::TK + o.slices - 1) / o.slices * tc::TK;
        h[g].plane = o.plane;
        h[g].tiles_m = pair ? (o.rows + 2 * tc::TM - 1) / (2 * tc::TM) : (o.M + nb - 1) / nb;
        h[g].tiles_n = (o.N + (pair ? 2 : 1) * tc::TM - 1) / ((pair ? 2 : 1) * tc::TM);
        h[g].tile_begin = tiles;
        // AUTO: N-major when the operator has more rows than the batch operand, so that the
        // larger operand is streamed once per launch and the smaller one re-read from L2
        const bool auto_n = o.N > o.M;
        h[g].n_major = raster == BPM_RASTER_N || (raster == BPM_RASTER_AUTO && auto_n) ? 1 : 0;
        tiles += h[g].tiles_m * h[g].tiles_n * h[g].splits;
    }
    grouped_gemm_free(gg);
    const int grid = std::max(1, std::min(tiles, sm_count));
    const std::vector<int> sched = pair ? std::vector<int>() : deal_items(h, tiles, grid);
    const size_t gbytes = h.size() * sizeof(GemmGroupDev), sbytes = sched.size() * sizeof(int);
    std::vector<char> host(gbytes + sbytes);
    std::memcpy(host.data(), h.data(), gbytes);
    if (sbytes) std::memcpy(host.data() + gbytes, sched.data(), sbytes);
    BPM_CK(cudaMalloc(&gg->d_groups, host.size()));
    BPM_CK(cudaMemcpy(gg->d_groups, host.data(), host.size(), cudaMemcpyHostToDevice));
    gg->d_sched = reinterpret_cast<int*>(reinterpret_cast<char*>(gg->d_groups) + gbytes);
    gg->grid = grid;
    gg->n_groups = (int)h.size();
    gg->total_tiles = tiles;
    gg->tile_n = nb_max <= 64 ? 64 : nb_max <= 128 ? 128 : 256;
    gg->products = products;
    gg->k_block = k_block;
    gg->pair = pair;
    return BPM_OK;
}

void grouped_gemm_free(GroupedGemm* gg) {
    if (gg->d_groups) cudaFree(gg->d_groups);
    gg->d_groups = nullptr;
    gg->d_sched = nullptr;
    gg->n_groups = gg->total_tiles = 0;
}

int grouped_gemm_launch(cudaStream_t s, GroupedGemm& gg, int sm_count, int* err, bool pdl) {
    if (!gg.d_groups) {
        set_error("grouped GEMM not set up");
        return BPM_ERR_STATE;
    }
    if (gg.pair) return grouped_gemm_pair_launch(s, gg, sm_count, err);
    const bool split = gg.products == 3;
    if (gg.tile_n == 64) return split ? launch_grouped<3, 64, 64>(s, gg, err, pdl)
                                      : launch_grouped<1, 64, 64>(s, gg, err, pdl);
    if (gg.tile_n == 128) return split ? launch_grouped<3, 128, 64>(s, gg, err, pdl)
                                       : launch_grouped<1, 128, 64>(s, gg, err, pdl);
    if (gg.k_block == 64) return split ? launch_grouped<3, 256, 64>(s, gg, err, pdl)
                                       : launch_grouped<1, 256, 64>(s, gg, err, pdl);
    return split ? launch_grouped<3, 256, 32>(s, gg, err, pdl)
                 : launch_grouped<1, 256, 32>(s, gg, err, pdl);
}

}  // namespace bpm
