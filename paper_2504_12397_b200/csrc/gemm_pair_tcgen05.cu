// Dense contractions of many rows with the aLoRA delta fused in: the gated q/k/v projection (Eq. 2 / Eq. 5) with 256 x 192
// output tiles, and the o_proj / MLP matrices of the layer stack with 256 x 256 tiles (residual in the epilogue; with
// adapters on the MLP block the same gated delta).
//
// Same computation and the same work list as gemm_tcgen05.cu's tile route (dense row tiles of 128 rows and the
// (row tile, adapter) pairs that occur; t = s A_k x from leading "shrink items" of the same launch; a tile appends
// t B_k^T of each of its adapters to its K loop; optional KV append in the epilogue), with another tile shape: a block
// owns TWO row tiles that share the W tile.  256 x 192: 56 KB of operands per 64-wide K block for 8 x 96 tensor-pipe
// cycles instead of 48 KB for 4 x 128, i.e. 1.3 x the flops per operand byte (one SM cannot fill its shared memory fast
// enough for the 128 x 256 tile), and 192-wide column tiles so that 2048 rows x 6144 columns make 256 tiles: two rounds
// over 148 blocks at 86 %.  256 x 256: 64 KB for 8 x 128 cycles, 1.5 x the flops per byte.
// The two row tiles accumulate in the two halves of tensor memory (not double-buffered; the next item's loads run
// under the epilogue and its MMAs start on a half as soon as that half has been drained).
//
// The MLP deltas as further K blocks cost next to nothing: 2048 rows of 8 x (8192 + 256) through two adapted layers took
// 174 us a layer for them when the shrink and the update of the finished gate / up / down rows were kernels of their own.
//
// A 192-wide column tile can straddle the q | k | v boundaries of the fused row.  The expand step therefore takes
// one K block per (pair, q/k/v block that the column tile touches): A = that block's 64 (padded-rank) columns
// of t, B = the adapter's B rows of that block through a 3-D tensor map (rank column, row inside the block,
// adapter) whose out-of-range rows read as zero, so the columns of the other block get no contribution.
//
//   warp 0   TMA producer (4 slots of 56 KB or 3 of 64 KB)      warp 1   MMA issuer (whole warp walks, elected lane issues)
//   warps 2-5 / 6-9  epilogue of the first / second row tile: tcgen05.ld one row per thread, bf16, 16-byte stores,
//              KV append, or t for shrink items
// All waits are bounded; on expiry ALORA_ERR_TIMEOUT is recorded and the block leaves normally.
#include <algorithm>

#include "alora_internal.h"
#include "tc_common.cuh"
#include "claim_order.h"

namespace alora {

namespace {
constexpr int kBKp = 64, kThreadsP = 320;          // producer, issuer, 2 x 4 epilogue warps
constexpr int kBNqkv = 192;                        // column tile of the q/k/v projection
constexpr int kTensorRP = 64;                      // the tensor path stores adapters padded to 64 rank columns
constexpr int kHalfAp = 128 * kBKp * 2;            // one row tile's x (or t) block: 16 KB
template <int BN>
struct PairSmem {
    static constexpr int kStages = BN <= 192 ? 4 : 3;
    static constexpr int kBBytes = BN * kBKp * 2;
    static constexpr int kStageBytes = 2 * kHalfAp + kBBytes;
    static constexpr int kBarOff = kStages * kStageBytes;
    static constexpr int kItemRingOff = kBarOff + 256;
    static constexpr int kTotal = kItemRingOff + 128 + 1024;
};

struct PairArgs {
    const TilePair *pairs;          // (row tile, adapter) pairs, nullptr: no adapters in this launch
    const int32_t *pair_off;        // [row tiles + 1] first pair of each row tile
    int tile0;                      // row tile of the batch that holds this launch's first row
    int shrink;                     // the launch has shrink items, one per pair of its row tiles (0: t is there already)
    int t_cols;                     // columns of t: 64 padded rank columns per adapted matrix
    const int32_t *adapters;        // per adapter `ad_stride` words, the first three: padded rank, scale (float), b_odd
    int ad_stride;
    int M, N, K, Nq, Nkv;           // Nq, Nkv: the q/k/v blocks of the fused row
    int blk_cols;                   // other launches: columns per adapted matrix
    __nv_bfloat16 *out;
    int ldo;
    const __nv_bfloat16 *residual;  // optional, same layout as out, may alias it
    const int32_t *row_adapter;     // [M] applied adapter per row (shrink items: which rows of t are kept)
    const int32_t *any_odd;         // not 0: an adapter of the context may have b_odd set
    const __nv_bfloat16 *b_all;     // the launch's B rows of all adapters, [adapter][N][64] (read for rows of those)
    int32_t *t_ready;               // [pair] epilogue warps that have published their part of t
    __nv_bfloat16 *t;               // [pair][128][t_cols]
    // KV append fused into the epilogue (nullptr: off), as in gemm_tcgen05.cu
    __nv_bfloat16 *kv_pool;
    const int32_t *slot_map;
    int kv_hd_shift, kv_heads, kv_page_size, kv_num_pages;
    int32_t *item_counters;         // [2] next unclaimed work item of the launch, blocks that have finished
    int32_t *status;
};

__device__ __forceinline__ int ld_acquire_p(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void tma_load_3d_p(uint32_t smem_dst, const CUtensorMap *map, uint32_t bar, int c0, int c1,
                                              int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_dst), "l"((uint64_t)map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// (none for a B with an Inf or NaN: see TilePair)
__device__ __forceinline__ int rank_steps(const PairArgs &a, int adapter) {
    const int32_t *ad = a.adapters + adapter * a.ad_stride;
    const int rpad = ad[0], odd = ad[2];
    return odd ? 0 : rpad / 16;
}

// One work item: a shrink item (pair p0[0], row tile m[0]) or two row tiles (m[1] = -1: none) x one column tile.
struct PairItem {
    int m[2];
    int p0[2], p1[2];    // pairs of each row tile
    int n0, adapter;
    bool shrink;
};
// kQkv: the column tiles of a row-tile pair are neighbours in the list; else the row tiles of a column tile (the blocks
// that run together share a W tile).
template <int BN, bool kQkv>
__device__ __forceinline__ PairItem decode_pair(const PairArgs &a, int item, int n_shrink, int p_base, int n_m, int n_n) {
    PairItem g;
    g.n0 = 0; g.adapter = -1; g.m[1] = -1;
    g.p0[0] = g.p1[0] = g.p0[1] = g.p1[1] = 0;
    g.shrink = item < n_shrink;
    if (g.shrink) {
        const TilePair p = a.pairs[p_base + item];
        g.m[0] = p.tile - a.tile0;
        g.adapter = p.adapter;
        g.p0[0] = g.p1[0] = g.p0[1] = g.p1[1] = p_base + item;
    } else {
        const int j = item - n_shrink, n_mp = (n_m + 1) / 2;
        g.m[0] = 2 * (kQkv ? j / n_n : j % n_mp);
        g.m[1] = g.m[0] + 1 < n_m ? g.m[0] + 1 : -1;
        g.n0 = (kQkv ? j % n_n : j / n_mp) * BN;
        if (a.pairs) {
            const int32_t *off = a.pair_off + a.tile0 + g.m[0];
            g.p0[0] = off[0];
            g.p1[0] = g.p0[1] = off[1];
            g.p1[1] = g.m[1] >= 0 ? off[2] : g.p0[1];
        }
    }
    return g;
}
// first row of q/k/v block `blk` in the fused row, and one past its last
__device__ __forceinline__ int blk_start(const PairArgs &a, int blk) { return blk == 0 ? 0 : (blk == 1 ? a.Nq : a.Nq + a.Nkv); }
__device__ __forceinline__ int blk_end(const PairArgs &a, int blk) { return blk == 0 ? a.Nq : (blk == 1 ? a.Nq + a.Nkv : a.N); }
// does the column tile at n0 touch block blk?
__device__ __forceinline__ bool touches(const PairArgs &a, int n0, int blk) {
    return n0 < blk_end(a, blk) && n0 + kBNqkv > blk_start(a, blk);
}

template <int BN, bool kQkv>
__global__ void __launch_bounds__(kThreadsP, 1)
gemm_pair_tcgen05_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                         const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmS,
                         const __grid_constant__ CUtensorMap tmB0, const __grid_constant__ CUtensorMap tmB1,
                         const __grid_constant__ CUtensorMap tmB2, const PairArgs a) {
    using S = PairSmem<BN>;
    constexpr int kStagesP = S::kStages, kBBytesP = S::kBBytes, kStageBytesP = S::kStageBytes;
    constexpr int kBarOffP = S::kBarOff, kItemRingOffP = S::kItemRingOff;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_al = smem_raw + (smem_base - tc::smem_u32(smem_raw));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_al + kBarOffP);
    // barrier words: full[stages], empty[stages], acc_full, acc_empty[2] (one per half), drain
    const uint32_t bar0 = smem_base + kBarOffP;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kStagesP + s); };
    const uint32_t accf_bar = bar0 + 8u * (2 * kStagesP);
    auto acce_bar = [&](int h) { return bar0 + 8u * (2 * kStagesP + 1 + h); };
    const uint32_t drain_bar = bar0 + 8u * (2 * kStagesP + 3);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(bars + 2 * kStagesP + 4);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 2 * kStagesP + 5);

    tc::ItemRing ring{smem_base + kItemRingOffP, reinterpret_cast<volatile int *>(smem_al + kItemRingOffP + 16 * tc::kItemSlots)};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        ring.init(9);   // the issuing warp and the eight epilogue warps
        for (int s = 0; s < kStagesP; ++s) { tc::mbar_init(full_bar(s), 1); tc::mbar_init(empty_bar(s), 1); }
        tc::mbar_init(accf_bar, 1);
        tc::mbar_init(acce_bar(0), 4); tc::mbar_init(acce_bar(1), 4);
        tc::mbar_init(drain_bar, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
        tc::fence_proxy_async();
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32((const void *)tmem_slot), 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    tc::grid_dep_launch();
    tc::grid_dep_wait();   // the metadata step's lists, the activations: all written by earlier kernels of the stream

    const int n_m = (a.M + 127) / 128;
    const int n_n = (a.N + BN - 1) / BN;
    const int p_base = a.shrink ? a.pair_off[a.tile0] : 0;
    const int n_shrink = a.shrink ? a.pair_off[a.tile0 + n_m] - p_base : 0;
    const int total = n_shrink + ((n_m + 1) / 2) * n_n;
    const int kb_main = (a.K + kBKp - 1) / kBKp;

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------ TMA producer ------------------------------
            tc::tma_prefetch_desc(&tmX); tc::tma_prefetch_desc(&tmW);
            uint32_t kc = 0;        // ring slots filled so far
            bool ok = true;
            // Order of this block's items.  Shrink items (the head of the list) are claimed from a global counter by
            // the blocks (see below which), one at a time, until none is left; only then does the block walk its
            // projection items, which are dealt out by block index as if the shrink items sat at list positions
            // 0 .. n_shrink-1 (what the first blocks to start normally take).  A projection item that waits for its row
            // tile's t therefore waits for a shrink item that a RUNNING block has claimed, however few blocks are
            // resident; and in the usual case every block keeps the items (and the L2 neighbours) it always had.
            bool shrink_phase = n_shrink > 0;
            int stat = (int)blockIdx.x;
            if (shrink_phase && !claims_at_once((int)blockIdx.x, n_shrink)) {
                // The blocks with the lowest indices have a free place in their list and normally take the shrink items
                // within a microsecond.  The others look on for a short while (about 30 us) and join the claiming
                // only if the shrink items are still not all taken by then (blocks that have not been scheduled).
                const long long t0 = clock64();
                while (ld_acquire_p(a.item_counters) < n_shrink && clock64() - t0 < 60000) {}
                if (ld_acquire_p(a.item_counters) >= n_shrink) shrink_phase = false;
            }
            while (ok) {
                int item = -1;
                if (shrink_phase) {
                    item = atomicAdd(a.item_counters, 1);
                    if (item >= n_shrink) { shrink_phase = false; item = -1; }
                }
                if (!shrink_phase && item < 0) {
                    item = next_dealt_item(stat, n_shrink, total, (int)gridDim.x);
                }
                if (!ring.put(item, abort_flag)) { ok = false; break; }
                if (item < 0) break;
                const PairItem g = decode_pair<BN, kQkv>(a, item, n_shrink, p_base, n_m, n_n);
                const bool two = g.m[1] >= 0;
                for (int kb = 0; kb < kb_main && ok; ++kb, ++kc) {
                    const int s = kc % kStagesP;
                    if (!tc::mbar_wait(empty_bar(s), ((kc / kStagesP) & 1) ^ 1, abort_flag)) { ok = false; break; }
                    const uint32_t sa = smem_base + s * kStageBytesP, sb = sa + 2 * kHalfAp;
                    tc::mbar_arrive_expect_tx(full_bar(s), (two ? 2 : 1) * kHalfAp + (g.shrink ? a.t_cols * kBKp * 2 : kBBytesP));
                    tc::tma_load_2d(sa, &tmX, full_bar(s), kb * kBKp, g.m[0] * 128);
                    if (two) tc::tma_load_2d(sa + kHalfAp, &tmX, full_bar(s), kb * kBKp, g.m[1] * 128);
                    if (g.shrink) tc::tma_load_2d(sb, &tmS, full_bar(s), kb * kBKp, g.adapter * a.t_cols);
                    else tc::tma_load_2d(sb, &tmW, full_bar(s), kb * kBKp, g.n0);
                }
                if (g.shrink) continue;
                // expand: per pair of the row tiles, one K block per adapted matrix (q / k / v block) the column tile touches
                for (int h = 0; h < 2 && ok && !g.shrink; ++h) {
                    int next_ad = g.p0[h] < g.p1[h] ? a.pairs[g.p0[h]].adapter : -1;
                    for (int p = g.p0[h]; p < g.p1[h] && ok; ++p) {
                        const int adapter = next_ad;
                        if (p + 1 < g.p1[h]) next_ad = a.pairs[p + 1].adapter;   // (in flight while this pair is waited for)
                        if (n_shrink > 0) {
                            // t of this pair is written by a shrink item (earlier in the list, so claimed by a running
                            // block): wait until its four epilogue warps have published, then order the TMA read after it
                            const long long t0 = clock64();
                            while (ld_acquire_p(a.t_ready + p) < 4) {
                                if (*abort_flag || clock64() - t0 > tc::kWaitCycleLimit) { *abort_flag = 1; ok = false; break; }
                            }
                            if (!ok) break;
                            asm volatile("fence.proxy.async.global;" ::: "memory");
                        }
                        for (int blk = 0; blk < (kQkv ? 3 : 1) && ok; ++blk) {
                            if (kQkv && !touches(a, g.n0, blk)) continue;
                            const int s = kc % kStagesP;
                            if (!tc::mbar_wait(empty_bar(s), ((kc / kStagesP) & 1) ^ 1, abort_flag)) { ok = false; break; }
                            const uint32_t sa = smem_base + s * kStageBytesP, sb = sa + 2 * kHalfAp;
                            tc::mbar_arrive_expect_tx(full_bar(s), kHalfAp + kBBytesP);
                            const int t_blk = kQkv ? blk : g.n0 / a.blk_cols;
                            tc::tma_load_2d(sa + h * kHalfAp, &tmT, full_bar(s), t_blk * kTensorRP, p * 128);
                            if (kQkv) tma_load_3d_p(sb, blk == 0 ? &tmB0 : (blk == 1 ? &tmB1 : &tmB2), full_bar(s), 0,
                                                    g.n0 - blk_start(a, blk), adapter);
                            else tc::tma_load_2d(sb, &tmB0, full_bar(s), 0, adapter * a.N + g.n0);
                            ++kc;
                        }
                    }
                }
            }
            if (!ok) {
                // give copies already in flight time to land before the block's shared memory is released
                const uint32_t first = kc > (uint32_t)kStagesP ? kc - kStagesP : 0;
                for (uint32_t i = first; i < kc; ++i) {
                    const long long t0 = clock64();
                    while (!tc::mbar_try_wait(full_bar(i % kStagesP), (i / kStagesP) & 1) &&
                           clock64() - t0 < tc::kWaitCycleLimit) {}
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        const bool leader = tc::elect_one();
        auto wait_all = [&](uint32_t bar, uint32_t parity) {
            return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, abort_flag));
        };
        constexpr uint32_t idesc_main = tc::idesc_bf16_f32(128, BN);
        const uint32_t idesc_shrink = tc::idesc_bf16_f32(128, a.t_cols);
        uint32_t kc = 0, it = 0;
        bool ok = true;
        for (;; ++it) {
            const int item = ring.take(abort_flag);
            if (item < 0) { ok = item == -1; break; }
            const PairItem g = decode_pair<BN, kQkv>(a, item, n_shrink, p_base, n_m, n_n);
            const bool two = g.m[1] >= 0;
            // MMA steps of the row tiles' adapters, one per lane, loaded while the main loop runs
            const int my_steps = g.p0[0] + lane < g.p1[1] ? rank_steps(a, a.pairs[g.p0[0] + lane].adapter) : 0;
            const uint32_t idesc = g.shrink ? idesc_shrink : idesc_main;
            for (int kb = 0; kb < kb_main && ok; ++kb, ++kc) {
                const int s = kc % kStagesP;
                if (!wait_all(full_bar(s), (kc / kStagesP) & 1)) { ok = false; break; }
                tc::tc_fence_after();
                const uint32_t sa = smem_base + s * kStageBytesP;
                const uint64_t db = tc::smem_desc_k_sw128(sa + 2 * kHalfAp);
                const uint64_t da0 = tc::smem_desc_k_sw128(sa), da1 = tc::smem_desc_k_sw128(sa + kHalfAp);
                // a half's accumulator must have been drained by the previous item's epilogue before its first MMA
                if (kb == 0 && !wait_all(acce_bar(0), (it & 1) ^ 1)) { ok = false; break; }
                if (leader) {
#pragma unroll
                    for (int k = 0; k < kBKp / 16; ++k)
                        tc::mma_bf16(tmem_base, da0 + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
                }
                if (kb == 0 && !wait_all(acce_bar(1), (it & 1) ^ 1)) { ok = false; break; }
                if (leader) {
                    if (two) {
#pragma unroll
                        for (int k = 0; k < kBKp / 16; ++k)
                            tc::mma_bf16(tmem_base + 256, da1 + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
                    }
                    tc::mma_commit(empty_bar(s));  // slot reusable once these MMAs have read it
                }
            }
            if (!ok) break;
            for (int h = 0; h < 2 && ok; ++h) {
                for (int p = g.p0[h]; p < g.p1[h] && ok; ++p) {
                    const int at = p - g.p0[0];   // (the pairs of the two row tiles follow one another)
                    const int steps = at < 32 ? __shfl_sync(0xffffffffu, my_steps, at) : rank_steps(a, a.pairs[p].adapter);
                    for (int blk = 0; blk < (kQkv ? 3 : 1) && ok; ++blk) {
                        if (kQkv && !touches(a, g.n0, blk)) continue;
                        const int s = kc % kStagesP;
                        if (!wait_all(full_bar(s), (kc / kStagesP) & 1)) { ok = false; break; }
                        tc::tc_fence_after();
                        const uint32_t sa = smem_base + s * kStageBytesP;
                        const uint64_t db = tc::smem_desc_k_sw128(sa + 2 * kHalfAp);
                        const uint64_t da = tc::smem_desc_k_sw128(sa + h * kHalfAp);
                        if (leader) {
                            for (int k = 0; k < steps; ++k) tc::mma_bf16(tmem_base + h * 256, da + 2 * k, db + 2 * k, idesc, 1u);
                            tc::mma_commit(empty_bar(s));
                        }
                        ++kc;
                    }
                }
            }
            if (!ok) break;
            if (leader) tc::mma_commit(accf_bar);      // accumulators complete
        }
        if (!ok && leader) {
            tc::mma_commit(drain_bar);                 // wait (bounded) for tensor-core work still in flight
            const long long t0 = clock64();
            while (!tc::mbar_try_wait(drain_bar, 0) && clock64() - t0 < tc::kWaitCycleLimit) {}
        }
    } else {
        // ------------------------------ epilogue (warps 2..5: first row tile, warps 6..9: second) ------------------------------
        const int q = warp & 3;           // tensor-memory lane quarter this warp may read
        const int my_h = (warp - 2) >> 2; // the half of tensor memory (row tile of the pair) this warp drains
        const bool any_odd = a.pairs != nullptr && *a.any_odd != 0;
        uint32_t it = 0;
        bool ok = true;
        for (;; ++it) {
            const int item = ring.take(abort_flag);
            if (item < 0) break;
            const PairItem g = decode_pair<BN, kQkv>(a, item, n_shrink, p_base, n_m, n_n);
            if (!tc::mbar_wait(accf_bar, it & 1, abort_flag)) { ok = false; break; }
            tc::tc_fence_after();
            const int r = q * 32 + lane;
            if (g.shrink && my_h == 1) {   // a shrink item has one row tile only
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(acce_bar(1));
                continue;
            }
            if (g.shrink) {
                // t = s A x of this pair, zero in the rows that do not use the adapter
                const int row = g.m[0] * 128 + r;
                const bool use = row < a.M && a.row_adapter[row] == g.adapter;
                const float scale = __int_as_float(a.adapters[g.adapter * a.ad_stride + 1]);
                __nv_bfloat16 *trow = a.t + ((size_t)g.p0[0] * 128 + r) * a.t_cols;
                const int rpad = a.adapters[g.adapter * a.ad_stride];
#pragma unroll 1
                for (int c = 0; c < a.t_cols; c += 32) {
                    if ((c & (kTensorRP - 1)) >= rpad) continue;   // (columns that no MMA step reads)
                    uint32_t v[32];
                    tc::tmem_ld_32x32(tmem_base + c + ((uint32_t)(q * 32) << 16), v);
                    tc::tmem_ld_wait();
                    tc::store_t_warp(reinterpret_cast<float(&)[32]>(v), scale, use, trow + c, a.t_cols, 1, 0);
                }
                tc::tc_fence_before();
                // publish: the rows are read by other blocks through TMA (async proxy)
                asm volatile("fence.proxy.async.global;" ::: "memory");
                __threadfence();
                __syncwarp();
                if (lane == 0) {
                    atomicAdd(a.t_ready + g.p0[0], 1);
                    tc::mbar_arrive(acce_bar(0));
                }
                continue;
            }
            {
                const int h = my_h;
                if (g.m[h] >= 0) {
                    const int row = g.m[h] * 128 + r;
                    const bool row_ok = row < a.M;
                    __nv_bfloat16 *orow = a.out + (size_t)row * a.ldo + g.n0;
                    const __nv_bfloat16 *rrow = a.residual ? a.residual + (size_t)row * a.ldo + g.n0 : nullptr;
                    // fused KV append: where this row's k / v columns go in the page pool
                    int kv_page = -1, kv_row = 0;
                    if (kQkv && a.kv_pool != nullptr && row_ok && g.n0 + BN > a.Nq) {
                        const int slot = a.slot_map[row];
                        if (slot >= 0) {
                            kv_page = slot / a.kv_page_size;
                            kv_row = slot % a.kv_page_size;
                            if (kv_page >= a.kv_num_pages) { report(a.status, ALORA_ERR_PAGE_RANGE); kv_page = -1; }
                        }
                    }
                    const uint32_t acc_addr = tmem_base + h * 256 + ((uint32_t)(q * 32) << 16);
                    auto put8 = [&](int c, float (&f)[8]) {   // columns c .. c + 7 of the tile
                        if (!kQkv && rrow) {
                            const uint4 rv = *reinterpret_cast<const uint4 *>(rrow + c);
                            const uint32_t rw[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const __nv_bfloat162 b2 = *reinterpret_cast<const __nv_bfloat162 *>(&rw[e]);
                                f[2 * e] += __low2float(b2);
                                f[2 * e + 1] += __high2float(b2);
                            }
                        }
                        uint4 o;
                        o.x = tc::pack_bf16(f[0], f[1]); o.y = tc::pack_bf16(f[2], f[3]);
                        o.z = tc::pack_bf16(f[4], f[5]); o.w = tc::pack_bf16(f[6], f[7]);
                        *reinterpret_cast<uint4 *>(orow + c) = o;
                        if (!kQkv) return;
                        const int kcol = g.n0 + c - a.Nq;   // column inside [k | v]
                        if (kv_page >= 0 && kcol >= 0) {
                            const int plane = kcol >= a.Nkv ? 1 : 0, c2 = kcol - plane * a.Nkv;
                            const int head = c2 >> a.kv_hd_shift, dd = c2 & ((1 << a.kv_hd_shift) - 1);
                            __nv_bfloat16 *dst = a.kv_pool +
                                ((((size_t)kv_page * 2 + plane) * a.kv_heads + head) * a.kv_page_size + kv_row << a.kv_hd_shift) + dd;
                            *reinterpret_cast<uint4 *>(dst) = o;
                        }
                    };
                    bool own_pass = false;   // the row's adapter has a B with an Inf or NaN
                    if (any_odd && row_ok && g.p0[h] < g.p1[h]) {
                        const int k = a.row_adapter[row];
                        own_pass = k >= 0 && a.adapters[k * a.ad_stride + 2] != 0;
                    }
#pragma unroll 1
                    for (int c = 0; c < BN; c += 32) {
                        uint32_t v[32];
                        tc::tmem_ld_32x32(acc_addr + c, v);
                        tc::tmem_ld_wait();
                        if (row_ok && !own_pass) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                if (g.n0 + c + 8 * j >= a.N) break;
                                put8(c + 8 * j, reinterpret_cast<float(&)[8]>(v[8 * j]));
                            }
                        }
                    }
                    if (__any_sync(0xffffffffu, own_pass)) {
                        tc::OddRow odd;
                        if (own_pass) {
                            const int k = a.row_adapter[row];
                            int p = g.p0[h];
                            while (p + 1 < g.p1[h] && a.pairs[p].adapter != k) ++p;
                            if (a.shrink) ld_acquire_p(a.t_ready + p);   // (complete since the tile's K blocks were loaded; orders the reads)
                            odd.t = a.t + ((size_t)p * 128 + r) * a.t_cols;
                            odd.b = a.b_all + (size_t)k * a.N * kTensorRP;
                            odd.n = a.adapters[k * a.ad_stride];
                        }
#pragma unroll 1
                        for (int c = 0; c < BN && g.n0 + c < a.N; c += 8) {
                            uint32_t v[8];
                            tc::tmem_ld_32x8(acc_addr + c, v);
                            tc::tmem_ld_wait();
                            if (!own_pass) continue;
                            const int col = g.n0 + c;
                            odd.add8(reinterpret_cast<float(&)[8]>(v), col, !kQkv ? col / a.blk_cols : col < a.Nq ? 0 : (col < a.Nq + a.Nkv ? 1 : 2));
                            put8(c, reinterpret_cast<float(&)[8]>(v));
                        }
                    }
                }
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(acce_bar(h));   // this half may be overwritten
            }
        }
    }

    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) report(a.status, ALORA_ERR_TIMEOUT);
    if (threadIdx.x == 0) tc::item_counter_release(a.item_counters, a.t_ready + p_base, n_shrink);
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem_base, 512);
    }
}
}  // namespace

bool make_tensor_map_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld,
                          uint32_t box_rows);  // gemm_tcgen05.cu
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn tensor_map_encoder();  // gemm_tcgen05.cu

// The per-layer tensor maps of this kernel: W in boxes of 192 rows, and for each of the q / k / v blocks the B
// rows of all adapters as (rank column, row inside the block, adapter).
bool build_pair_maps(alora_ctx *ctx, int layer) {
    const Dims &d = ctx->d;
    TcLayerMaps &lm = ctx->tc_maps[layer];
    const LayerWeights &lw = ctx->layers[layer];
    bool ok = true;
    if (lw.wqkv) ok &= make_tensor_map_bf16(&lm.wqkv192, lw.wqkv, d.N, d.H, d.H, kBNqkv);
    EncodeTiledFn enc = tensor_map_encoder();
    if (!enc) return false;
    const size_t na = (size_t)std::max(1, ctx->cfg.max_adapters);
    const int starts[3] = {0, d.Nq, d.Nq + d.Nkv}, rows[3] = {d.Nq, d.Nkv, d.Nkv};
    for (int blk = 0; blk < 3; ++blk) {
        cuuint64_t dims[3] = {(cuuint64_t)kTensorRP, (cuuint64_t)rows[blk], (cuuint64_t)na};
        cuuint64_t strides[2] = {(cuuint64_t)kTensorRP * 2, (cuuint64_t)d.N * kTensorRP * 2};
        cuuint32_t box[3] = {(cuuint32_t)kTensorRP, (cuuint32_t)kBNqkv, 1};
        cuuint32_t es[3] = {1, 1, 1};
        void *base = (char *)ctx->tc_b_all[layer] + (size_t)starts[blk] * kTensorRP * 2;
        ok &= enc(&lm.b_blk[blk], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    return ok;
}

template <int BN, bool kQkv>
static bool pair_kernel_ready(alora_ctx *ctx) {
    static bool attr_set[64] = {};   // one per instantiation
    const int dev = ctx->cfg.device;
    if (dev < 0 || dev >= 64 || attr_set[dev]) return true;
    attr_set[dev] = cudaFuncSetAttribute(gemm_pair_tcgen05_kernel<BN, kQkv>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         PairSmem<BN>::kTotal) == cudaSuccess;
    return attr_set[dev];
}

bool launch_shrink_tc(alora_ctx *ctx, const CUtensorMap &tmX, const RankMaps &tmA, const AdapterDev *adapters,
                      int T, int K, int max_pairs, int t_parts, cudaStream_t s);  // shrink_tcgen05.cu
bool shrink_apart(const alora_ctx *ctx, int T, int R, int items);                  // gemm_tcgen05.cu

// Returns the kernels launched, 0 when the batch is better served by the 128-row kernel (nothing launched) or
// -1 on error.  Only for batches of more than kSplitTTokens rows (one summand of t; the decision must not depend on the
// mode, so that rows with a closed gate come out bit-identical to the base-only projection of the same batch).
int launch_project_pair_tc(alora_ctx *ctx, int layer, const void *hidden, int T, int R, void *qkv, cudaStream_t s,
                           void *kv_pool, int num_pages) {
    const Dims &d = ctx->d;
    if (T <= kSplitTTokens || d.H % 8 != 0 || d.N % 8 != 0 || d.Nq % 8 != 0 || d.Nkv % 8 != 0) return 0;
    const int G = ctx->sm_count;
    const int n_n = (d.N + kBNqkv - 1) / kBNqkv, n_n256 = (d.N + 255) / 256;
    const int items = ((T + 255) / 256) * n_n, items128 = ((T + 127) / 128) * n_n256;
    const double eff = (double)items / ((double)((items + G - 1) / G) * G);
    const double eff128 = (double)items128 / ((double)((items128 + G - 1) / G) * G);
    if (eff * 1.25 < eff128) return 0;
    const TcLayerMaps &lm = ctx->tc_maps[layer];
    CUtensorMap tmX, tmT;
    if (!make_tensor_map_bf16(&tmX, hidden, T, d.H, d.H, 128)) return -1;
    if (!make_tensor_map_bf16(&tmT, ctx->d_t, (uint64_t)ctx->t_slots * 128, 3 * kTensorRP, 3 * kTensorRP, 128)) return -1;
    if (!pair_kernel_ready<kBNqkv, true>(ctx)) return -1;
    PairArgs g{};
    g.M = T; g.N = d.N; g.K = d.H; g.Nq = d.Nq; g.Nkv = d.Nkv;
    g.out = (__nv_bfloat16 *)qkv; g.ldo = d.N;
    const AdapterDev *ads = ctx->d_adapters + (size_t)layer * ctx->cfg.max_adapters;
    g.adapters = &ads->rpad;   // (address arithmetic only: padded rank and scale of an AdapterDev are neighbours)
    g.ad_stride = sizeof(AdapterDev) / 4; g.t_cols = 3 * kTensorRP;
    const bool have_adapters = ctx->layer_has_adapter[layer] != 0;
    const bool apart = have_adapters && shrink_apart(ctx, T, R, items);
    const int max_pairs = have_adapters ? pair_bound(ctx, T, R) : 0;
    if (have_adapters) {
        g.pairs = ctx->d_pairs; g.pair_off = ctx->d_pair_off; g.t = (__nv_bfloat16 *)ctx->d_t;
        g.row_adapter = ctx->d_row_adapter; g.any_odd = ctx->d_counts + kOddAdapters;
        g.b_all = (const __nv_bfloat16 *)ctx->tc_b_all[layer];
    }
    if (have_adapters && !apart) { g.shrink = 1; g.t_ready = ctx->d_t_ready; }
    g.item_counters = ctx->d_counts + 10;
    if (kv_pool != nullptr) {
        int shift = 0;
        while ((1 << shift) < d.hd) ++shift;
        g.kv_pool = (__nv_bfloat16 *)kv_pool; g.slot_map = ctx->d_slot; g.kv_hd_shift = shift; g.kv_heads = d.Hkv;
        g.kv_page_size = d.page; g.kv_num_pages = num_pages;
    }
    g.status = ctx->d_status;
    const int grid = std::max(1, std::min(G, items + (apart ? 0 : max_pairs)));
    if (apart && !launch_shrink_tc(ctx, tmX, lm.a_rank, ads, T, d.H, max_pairs, 1, s)) return -1;
    if (launch_kernel(gemm_pair_tcgen05_kernel<kBNqkv, true>, dim3(grid), dim3(kThreadsP), PairSmem<kBNqkv>::kTotal, s, true, tmX,
                      lm.wqkv192, tmT, lm.a_all, lm.b_blk[0], lm.b_blk[1], lm.b_blk[2], g) != cudaSuccess)
        return -1;
    return apart ? 2 : 1;
}

// Plain dense projection y = x W^T (+ residual) with many rows, optionally with a gated low-rank delta: 256 x 256 tiles.
// Returns 1 (launched), 0 (shape better served by the 128-row kernel: not launched) or -1 (error).
int launch_linear256_tc(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y,
                        const void *residual, const LinearDelta *delta, cudaStream_t s) {
    constexpr int BN = 256;
    const int n_n = (N + BN - 1) / BN, G = ctx->sm_count;
    const int items = ((T + 255) / 256) * n_n, items128 = ((T + 127) / 128) * n_n;
    // Rounds over the blocks x cycles of a tile's K block: 1230 here (0.83 of the tensor pipe), 790 for the 128 x 256 tile.  That
    // kernel walks the column tiles of a row tile first, so a W that L2 does not hold is streamed from HBM (3400 bytes a cycle)
    // in every round.  Dense matrices of two 8B layers, us, 128-row tiles for all / for o_proj and down only: 384 rows 427 / 388,
    // 640 rows 650 / 577, 896 rows 803 / 687; this kernel for all / for gate and up only: 1152 rows 820 / 703, 1280 rows 862 / 937.
    const long long rounds128 = (items128 + G - 1) / G;
    const long long w_cycles = (long long)N * K * 2 > (64ll << 20) ? (n_n >= G ? (T + 127) / 128 : rounds128) * N * (2 * kBKp) / 3400 : 0;
    const long long here = (long long)((items + G - 1) / G) * 1230, other = std::max(rounds128 * 790, w_cycles);
    if (T <= 256 || K % 8 != 0 || N % 8 != 0 || here > other) return 0;
    CUtensorMap tmX, tmW, tmT, tmA, tmB;
    if (!make_tensor_map_bf16(&tmX, x, T, K, K, 128)) return -1;
    if (!make_tensor_map_bf16(&tmW, W, N, K, K, BN)) return -1;
    tmT = tmX; tmA = tmW; tmB = tmW;
    PairArgs g{};
    g.M = T; g.N = N; g.K = K; g.Nq = N; g.Nkv = 0; g.blk_cols = N; g.t_cols = kTensorRP;
    g.out = (__nv_bfloat16 *)y; g.residual = (const __nv_bfloat16 *)residual; g.ldo = N;
    g.item_counters = ctx->d_counts + 10; g.status = ctx->d_status;
    if (delta != nullptr) {
        const uint64_t na = (uint64_t)std::max(1, ctx->cfg.max_adapters);
        g.t_cols = delta->n_blk * kTensorRP; g.blk_cols = N / delta->n_blk;
        if (!make_tensor_map_bf16(&tmT, delta->t, (uint64_t)ctx->max_pairs * 128, g.t_cols, g.t_cols, 128)) return -1;
        if (!make_tensor_map_bf16(&tmA, delta->A, na * g.t_cols, K, K, g.t_cols)) return -1;
        if (!make_tensor_map_bf16(&tmB, delta->B, na * N, kTensorRP, kTensorRP, BN)) return -1;
        g.pairs = ctx->d_pairs; g.pair_off = ctx->d_pair_off; g.tile0 = delta->tile0; g.shrink = 1;
        g.adapters = &delta->table->rpad; g.ad_stride = sizeof(MlpAdapterDev) / 4;
        g.row_adapter = delta->row_adapter; g.t_ready = ctx->d_t_ready; g.t = (__nv_bfloat16 *)delta->t;
        g.any_odd = ctx->d_counts + kOddAdapters; g.b_all = (const __nv_bfloat16 *)delta->B;
    }
    if (!pair_kernel_ready<BN, false>(ctx)) return -1;
    const int grid = std::max(1, std::min(G, items + (delta != nullptr ? ctx->max_pairs : 0)));
    if (launch_kernel(gemm_pair_tcgen05_kernel<BN, false>, dim3(grid), dim3(kThreadsP), PairSmem<BN>::kTotal, s, true, tmX, tmW,
                      tmT, tmA, tmB, tmB, tmB, g) != cudaSuccess)
        return -1;
    return 1;
}

}  // namespace alora
