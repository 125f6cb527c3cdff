// Rank-r shrink t = s A_k x on the tensor cores (the inner product of the low-rank delta of Eq. 5),
// split along the hidden dimension over a thread-block cluster.
//
// The shrink has few output tiles (one of 128 rows x 3 blocks q / k / v of the adapter's padded rank per (row tile,
// adapter) pair) but a long contraction (the hidden dimension), so each pair is given to a cluster of 8 or 4 blocks.
// Block c of the cluster contracts hidden columns of its own K range with tcgen05.mma into tensor memory, copies its fp32
// partial tile into its shared memory, and after a cluster barrier reduces its share of the tile's columns over all
// blocks' shared memory (distributed shared memory loads) in the fixed order 0, 1, ....  The order does not depend on
// timing, so the result is run-to-run deterministic.
// Bound by what a block takes in (operands by TMA, 20 bytes / ns of other blocks' shared memory) and by the rounds of clusters:
// only the padded rank's rows of A are loaded, multiplied and reduced, and where more pairs are possible than clusters
// of 8 fit on the device (15), clusters are of 4 (33 fit).  48 requests over four adapters of rank 8 .. 64, 24 pairs at
// hidden 4096: 32 -> 18 us against 192 rows of A for each and 8 blocks.
#include <algorithm>

#include "alora_internal.h"
#include "tc_common.cuh"

namespace alora {

constexpr int kShrinkMaxSplits = 8;     // blocks per cluster = K ranges per row tile
constexpr int kShrinkBM = 128;          // rows per tile
constexpr int kShrinkBN = 192;          // 3 blocks x 64 rows of A stored per adapter
constexpr int kShrinkBK = 64;
constexpr int kShrinkStages = 4;
constexpr int kShrinkThreads = 192;     // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue / reduction

struct ShrinkArgs {
    const TilePair *pairs;
    const int32_t *n_pairs;
    const int32_t *row_adapter;   // [T] applied adapter per row
    const AdapterDev *adapters;
    __nv_bfloat16 *t;   // [pair][t_parts][128][192]
    int t_parts, T, splits;
    int K;              // hidden
    int32_t *status;
};

struct ShrinkSmem {
    static constexpr int kABytes = kShrinkBM * kShrinkBK * 2;
    static constexpr int kBBytes = kShrinkBN * kShrinkBK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kRingBytes = kShrinkStages * kStageBytes;        // 160 KB; reused as the fp32 partial tile
    static constexpr int kPartialBytes = kShrinkBN * kShrinkBM * 4;       // [192 columns][128 rows] fp32
    static constexpr int kBarOffset = kRingBytes;
    static constexpr int kTotal = kBarOffset + 256 + 1024;
    static_assert(kPartialBytes <= kRingBytes, "partial tile must fit in the ring");
};

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float ld_dsmem_f32(uint32_t local_addr, uint32_t rank) {
    uint32_t remote;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local_addr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}

__global__ void __launch_bounds__(kShrinkThreads, 1)
shrink_tcgen05_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ RankMaps tmA,
                      const ShrinkArgs a) {
    using S = ShrinkSmem;
    tc::grid_dep_launch();
    tc::grid_dep_wait();   // the pairs and the row -> adapter map come from the metadata kernel, x from the kernel before
    // the whole cluster takes the same decision: blockIdx.y selects the pair
    if ((int)blockIdx.y >= *a.n_pairs) return;
    const TilePair pair = a.pairs[blockIdx.y];
    const int rpad = a.adapters[pair.adapter].rpad, cols = 3 * rpad;
    if (cols == 0) return;   // not registered on this layer (a finding of the metadata step): its t is not used

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_al = smem_raw + (smem_base - tc::smem_u32(smem_raw));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_al + S::kBarOffset);
    const uint32_t bar0 = smem_base + S::kBarOffset;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kShrinkStages + s); };
    const uint32_t acc_bar = bar0 + 8u * (2 * kShrinkStages);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(bars + 2 * kShrinkStages + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 2 * kShrinkStages + 2);
    float *partial = reinterpret_cast<float *>(smem_al);  // [192][128], aliases the ring once the MMAs are done

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kTmemCols = 256;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kShrinkStages; ++s) { tc::mbar_init(full_bar(s), 1); tc::mbar_init(empty_bar(s), 1); }
        tc::mbar_init(acc_bar, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
        tc::fence_proxy_async();
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32((const void *)tmem_slot), kTmemCols);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    // this block's K range, in 64-column blocks
    const uint32_t crank = cluster_ctarank();
    const int kb_all = (a.K + kShrinkBK - 1) / kShrinkBK;
    const int kb_per = (kb_all + a.splits - 1) / a.splits;
    const int kb0 = (int)crank * kb_per;
    const int nkb = max(0, min(kb_per, kb_all - kb0));

    if (warp == 0) {
        if (lane == 0) {
            tc::tma_prefetch_desc(&tmX); tc::tma_prefetch_desc(&tmA.box[rpad / 16 - 1]);
            bool ok = true;
            int kc = 0;
            for (; kc < nkb; ++kc) {
                const int s = kc % kShrinkStages;
                if (!tc::mbar_wait(empty_bar(s), ((kc / kShrinkStages) & 1) ^ 1, abort_flag)) { ok = false; break; }
                const uint32_t sa = smem_base + s * S::kStageBytes, sb = sa + S::kABytes;
                tc::mbar_arrive_expect_tx(full_bar(s), S::kABytes + cols * kShrinkBK * 2);
                tc::tma_load_2d(sa, &tmX, full_bar(s), (kb0 + kc) * kShrinkBK, pair.tile * kShrinkBM);
                for (int blk = 0; blk < 3; ++blk)
                    tc::tma_load_2d(sb + blk * rpad * kShrinkBK * 2, &tmA.box[rpad / 16 - 1], full_bar(s), (kb0 + kc) * kShrinkBK,
                                    pair.adapter * kShrinkBN + blk * kRankPadMax);
            }
            if (!ok) {
                // copies already in flight must land before the shared memory is reused or released
                for (int i = max(0, kc - kShrinkStages); i < kc; ++i) {
                    const long long t0 = clock64();
                    while (!tc::mbar_try_wait(full_bar(i % kShrinkStages), (i / kShrinkStages) & 1) &&
                           clock64() - t0 < tc::kWaitCycleLimit) {}
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && nkb > 0) {
            const uint32_t idesc = tc::idesc_bf16_f32(kShrinkBM, cols);
            for (int kc = 0; kc < nkb; ++kc) {
                const int s = kc % kShrinkStages;
                if (!tc::mbar_wait(full_bar(s), (kc / kShrinkStages) & 1, abort_flag)) break;
                tc::tc_fence_after();
                const uint32_t sa = smem_base + s * S::kStageBytes, sb = sa + S::kABytes;
                const uint64_t da = tc::smem_desc_k_sw128(sa), db = tc::smem_desc_k_sw128(sb);
                for (int k = 0; k < kShrinkBK / 16; ++k)
                    tc::mma_bf16(tmem_base, da + 2 * k, db + 2 * k, idesc, (kc | k) != 0 ? 1u : 0u);
                tc::mma_commit(empty_bar(s));
            }
            tc::mma_commit(acc_bar);  // arrives once every MMA issued above has completed (also after a failed wait)
        }
    } else {
        // epilogue warps: this block's partial tile -> shared memory, column-major so that the 32 rows of
        // a warp are 32 consecutive words
        const int q = warp & 3;
        const int r = q * 32 + lane;
        bool have = nkb > 0;
        if (have) have = tc::mbar_wait(acc_bar, 0, abort_flag);
        tc::tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < cols; c += 32) {   // (16 columns of a last half are not read by anyone)
            uint32_t v[32];
            if (have) {
                tc::tmem_ld_32x32(tmem_base + c + ((uint32_t)(q * 32) << 16), v);
                tc::tmem_ld_wait();
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = 0u;
            }
#pragma unroll
            for (int e = 0; e < 32; ++e) partial[(c + e) * kShrinkBM + r] = __uint_as_float(v[e]);
        }
        tc::tc_fence_before();
    }

    __syncthreads();
    cluster_sync_all();  // every block's partial tile is in its shared memory

    if (warp >= 2) {
        const int q = warp & 3;
        const int r = q * 32 + lane;
        const float scale = a.adapters[pair.adapter].scale;
        const int row = pair.tile * kShrinkBM + r;
        const bool use = row < a.T && a.row_adapter[row] == pair.adapter;
        for (int u = (int)crank * (cols / 8) / a.splits; u < ((int)crank + 1) * (cols / 8) / a.splits; ++u) {   // 8 columns
            float part[kShrinkMaxSplits][8], acc[8];
#pragma unroll
            for (int src = 0; src < kShrinkMaxSplits; ++src)
                if (src < a.splits) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) part[src][j] = ld_dsmem_f32(tc::smem_u32(partial + (u * 8 + j) * kShrinkBM + r), (uint32_t)src);
                }
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = 0.f;
#pragma unroll
            for (int src = 0; src < kShrinkMaxSplits; ++src)   // fixed order: deterministic sum
                if (src < a.splits) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[j] += part[src][j];
                }
            const int blk = u * 8 / rpad;
            __nv_bfloat16 *orow = a.t + ((size_t)blockIdx.y * a.t_parts * kShrinkBM + r) * kShrinkBN + blk * kRankPadMax + u * 8 - blk * rpad;
            tc::store_t8(acc, scale, use, orow, a.t_parts, kShrinkBM * kShrinkBN);
        }
    }

    cluster_sync_all();  // no block may release its shared memory while another still reads it
    if (threadIdx.x == 0 && *abort_flag) report(a.status, ALORA_ERR_TIMEOUT);
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem_base, kTmemCols);
    }
}

// t = s A x of the (row tile, adapter) pairs of the current batch, of which there are at most max_pairs.  Returns false
// if the launch could not be set up.
bool launch_shrink_tc(alora_ctx *ctx, const CUtensorMap &tmX, const RankMaps &tmA, const AdapterDev *adapters,
                      int T, int K, int max_pairs, int t_parts, cudaStream_t s) {
    static bool attr_set[64] = {};
    const int dev = ctx->cfg.device;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        if (cudaFuncSetAttribute(shrink_tcgen05_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 ShrinkSmem::kTotal) != cudaSuccess)
            return false;
        attr_set[dev] = true;
    }
    ShrinkArgs a{ctx->d_pairs, ctx->d_counts + 2, ctx->d_row_adapter, adapters, (__nv_bfloat16 *)ctx->d_t, t_parts, T,
                 max_pairs <= ctx->few_clusters[8] ? 8 : 4, K, ctx->d_status};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(a.splits, std::max(1, max_pairs)); cfg.blockDim = dim3(kShrinkThreads);
    cfg.dynamicSmemBytes = ShrinkSmem::kTotal; cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)a.splits; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, shrink_tcgen05_kernel, tmX, tmA, a) == cudaSuccess;
}

}  // namespace alora
