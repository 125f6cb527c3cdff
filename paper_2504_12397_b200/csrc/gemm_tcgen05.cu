// bf16 dense contraction on the 5th-generation tensor cores: out[rows][N] = act[rows][K] . W[N][K]^T
// with the aLoRA delta fused in.
//
// One persistent block per SM, three roles:
//   warp 0 (one lane)  TMA producer: streams 128 x 64 activation tiles and BN x 64 weight tiles
//                      (128-byte swizzle) through a 4-deep shared-memory ring;
//   warp 1 (one lane)  MMA issuer: tcgen05.mma 128 x BN x 16 steps into one of two fp32 accumulators in
//                      tensor memory, releasing ring slots and publishing accumulators via
//                      tcgen05.commit;
//   warps 2-5          epilogue: tcgen05.ld the accumulator (one row per thread), optional residual
//                      add / scale, round to bf16, 16-byte row-predicated stores.  The second
//                      accumulator lets the next tile's main loop overlap this epilogue.
//
// Row tiles are dense.  For every adapter that some row of the tile uses (the (row tile, adapter) pairs of the
// batch-metadata step) the main K loop (the base term W x of Eq. 5) is followed by further K blocks whose operands are
// t = s A x and the adapter's B rows of this column tile, i.e. the delta s B (A x) is accumulated by the same
// tensor-core instruction stream.  The rows of t that do not use the adapter (another adapter, or a closed gate) are
// zero, so those rows of the accumulator are added zeros: a row whose gate is closed keeps the bits of a base-only
// call (Prop. 1).  (Cutting the row tiles at every change of adapter instead left most tiles of a batch of short
// requests nearly empty, and a per-row delta beside dense tiles took 190 us for 742 rows.)
//
// Where t = s A x comes from.  With 256-wide column tiles the shrink can be part of this kernel: the first
// work items of the launch are one "shrink item" per pair, whose B operand is the adapter's
// 192 A rows (q, k, v blocks, rank padded to 64) and whose epilogue writes t and then raises a per-pair
// ready counter in global memory.  A projection item waits (bounded) for the counters of its row tile's pairs
// before it loads their t; shrink items are claimed first (claim_order.h).  With 128-wide column tiles, and where the
// shrink items would add a round over the blocks, the shrink is a cluster split-K kernel before (shrink_tcgen05.cu).
// No split-K, no atomics in the arithmetic: results are run-to-run deterministic.
//
// Every wait is bounded (tc::mbar_wait); on expiry the block records ALORA_ERR_TIMEOUT, drains its
// outstanding copies and tensor-core work with bounded waits, frees its tensor memory and returns.
#include "alora_internal.h"
#include "tc_common.cuh"
#include "claim_order.h"

namespace alora {

constexpr int kBM = 128;      // rows per tile (UMMA M)
constexpr int kBK = 64;       // K elements per ring slot (one 128-byte swizzle row)
constexpr int kGemmThreads = 192;
constexpr int kTensorRP = 64; // the tensor path stores adapters padded to 64 rank columns

struct GemmArgs {
    // Bytes one copy of the activation tile brings (0: the full 128-row tile).  A batch of at most 64 rows uses a
    // 64-row box: the other half of the tile in shared memory is never filled, the accumulator rows it feeds are
    // never read, and the shared-memory fill of a stage, which bounds this shape, drops by a third.
    int a_tile_bytes;
    const TilePair *pairs;          // (row tile, adapter) pairs of the batch, nullptr: no adapters in this launch
    const int32_t *pair_off;        // [row tiles + 1] first pair of each row tile
    int tile0;                      // row tile of the batch that holds this launch's first row
    int shrink;                     // the launch has shrink items, one per pair of its row tiles (0: t is there already)
    int t_cols;                     // columns of t: 64 padded rank columns per adapted matrix
    const int32_t *adapters;        // per adapter `ad_stride` words, the first three: padded rank, scale (float), b_odd
    int ad_stride;
    int M, N, K;
    __nv_bfloat16 *out;
    int ldo;
    const __nv_bfloat16 *residual;  // optional, same layout as out, may alias it
    int Nq, Nkv;                    // block boundaries of the fused output row (expand; gate | up: Nq = Nkv = half)
    int total_adapter_rows;         // rows per adapter in the B_all map (= N of the layer)
    const int32_t *row_adapter;     // [M] applied adapter per row (shrink items: which rows of t are kept)
    const int32_t *any_odd;         // not 0: an adapter of the context may have b_odd set
    const __nv_bfloat16 *b_all;     // the launch's B rows of all adapters, [adapter][N][64] (read for rows of those)
    int32_t *t_ready;               // [pair] epilogue warps that have published their part of t
    __nv_bfloat16 *t;               // [pair][t_parts][128][t_cols]
    int t_parts;                    // t is the sum of this many bf16 values (1 or 3)
    // KV append fused into the epilogue (nullptr: off): columns Nq .. N of row t also go to the paged cache,
    // pool[page][plane][head][row in page][:] with page * page_size + row = slot_map[t] (-1: token rejected, skipped)
    __nv_bfloat16 *kv_pool;
    const int32_t *slot_map;
    int kv_hd_shift, kv_heads, kv_page_size, kv_num_pages;
    int32_t *item_counters;         // [2] next unclaimed work item of the launch, blocks that have finished
    int32_t *status;
};

template <int BN>
struct GemmSmem {
    // ring depth: 4 slots of 32 .. 48 KB for the wide tiles; the 64-wide tile of the skinny (few rows, weight
    // streaming) case gets 8 slots of 24 KB so that enough bytes are in flight per SM
    static constexpr int kStages = BN <= 64 ? 8 : 4;
    static constexpr int kABytes = kBM * kBK * 2;
    static constexpr int kBBytes = BN * kBK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kSummandsPerSlot = kBBytes >= kABytes ? 2 : 1;   // t blocks in a slot without B
    static constexpr int kBarOffset = kStages * kStageBytes;
    static constexpr int kItemRingOffset = kBarOffset + 256;
    static constexpr int kTotal = kItemRingOffset + 128 + 1024;  // barriers, item ring, slack for 1024-byte alignment
};

// (none for a B with an Inf or NaN: see TilePair)
__device__ __forceinline__ int rank_steps(const GemmArgs &a, int adapter) {
    const int32_t *ad = a.adapters + adapter * a.ad_stride;
    const int rpad = ad[0], odd = ad[2];
    return odd ? 0 : rpad / 16;
}

// Work item `item` of a launch: shrink items first (one per pair), then the projection's
// (row tile, column tile) pairs.
struct GemmItem {
    int m;            // row-tile index
    int n0;           // first output column (projection items)
    int p0, p1;       // projection items: the row tile's pairs; shrink items: p0 = p1 = its pair
    int adapter;      // shrink items
    bool shrink;
};
__device__ __forceinline__ GemmItem decode_item(const GemmArgs &a, int item, int n_shrink, int p_base, int n_n, int BN) {
    GemmItem g;
    g.n0 = 0; g.p0 = 0; g.p1 = 0; g.adapter = -1;
    g.shrink = item < n_shrink;
    if (g.shrink) {
        const TilePair p = a.pairs[p_base + item];
        g.m = p.tile - a.tile0;
        g.adapter = p.adapter;
        g.p0 = g.p1 = p_base + item;
    } else {
        const int j = item - n_shrink;
        g.m = j / n_n;
        g.n0 = (j % n_n) * BN;
        if (a.pairs) { g.p0 = a.pair_off[a.tile0 + g.m]; g.p1 = a.pair_off[a.tile0 + g.m + 1]; }
    }
    return g;
}

__device__ __forceinline__ int ld_acquire(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

template <int BN>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_tcgen05_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmL,
                    const __grid_constant__ CUtensorMap tmS, const GemmArgs a) {
    using S = GemmSmem<BN>;
    constexpr int kStages = S::kStages;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_al = smem_raw + (smem_base - tc::smem_u32(smem_raw));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_al + S::kBarOffset);
    // barrier words: full[kStages], empty[kStages], acc_full[2], acc_empty[2], drain
    const uint32_t bar0 = smem_base + S::kBarOffset;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
    auto accf_bar = [&](int i) { return bar0 + 8u * (2 * kStages + i); };
    auto acce_bar = [&](int i) { return bar0 + 8u * (2 * kStages + 2 + i); };
    const uint32_t drain_bar = bar0 + 8u * (2 * kStages + 4);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(bars + 2 * kStages + 5);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 2 * kStages + 6);
    tc::ItemRing ring{smem_base + S::kItemRingOffset,
                      reinterpret_cast<volatile int *>(smem_al + S::kItemRingOffset + 16 * tc::kItemSlots)};

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kTmemCols = (2 * BN <= 256) ? 256 : 512;

    if (threadIdx.x == 0) {
        ring.init(5);   // the issuing warp and the four epilogue warps
        for (int s = 0; s < kStages; ++s) { tc::mbar_init(full_bar(s), 1); tc::mbar_init(empty_bar(s), 1); }
        for (int i = 0; i < 2; ++i) { tc::mbar_init(accf_bar(i), 1); tc::mbar_init(acce_bar(i), 4); }
        tc::mbar_init(drain_bar, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
        tc::fence_proxy_async();
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32((const void *)tmem_slot), kTmemCols);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    tc::grid_dep_launch();
    tc::grid_dep_wait();   // the metadata step's lists, the activations: all written by earlier kernels of the stream

    const int n_m = (a.M + kBM - 1) / kBM;
    const int n_n = (a.N + BN - 1) / BN;
    const int p_base = (BN == 256 && a.shrink) ? a.pair_off[a.tile0] : 0;
    const int n_shrink = (BN == 256 && a.shrink) ? a.pair_off[a.tile0 + n_m] - p_base : 0;
    const int total = n_shrink + n_m * n_n;
    const int kb_main = (a.K + kBK - 1) / kBK;
    const int t_slots = a.t_parts > 1 ? 1 + (a.t_parts - 1) / S::kSummandsPerSlot : 1;   // ring slots of a pair

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------ TMA producer ------------------------------
            tc::tma_prefetch_desc(&tmA); tc::tma_prefetch_desc(&tmB);
            if (a.pairs != nullptr) { tc::tma_prefetch_desc(&tmT); tc::tma_prefetch_desc(&tmL); }
            const uint32_t a_bytes = a.a_tile_bytes ? (uint32_t)a.a_tile_bytes : (uint32_t)S::kABytes;
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
                while (ld_acquire(a.item_counters) < n_shrink && clock64() - t0 < 60000) {}
                if (ld_acquire(a.item_counters) >= n_shrink) shrink_phase = false;
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
                const GemmItem g = decode_item(a, item, n_shrink, p_base, n_n, BN);
                const int row0 = g.m * kBM, n0 = g.n0;
                for (int kb = 0; kb < kb_main; ++kb, ++kc) {
                    const int s = kc % kStages;
                    if (!tc::mbar_wait(empty_bar(s), ((kc / kStages) & 1) ^ 1, abort_flag)) { ok = false; break; }
                    const uint32_t sa = smem_base + s * S::kStageBytes, sb = sa + S::kABytes;
                    tc::mbar_arrive_expect_tx(full_bar(s), a_bytes + (g.shrink ? a.t_cols * kBK * 2 : S::kBBytes));
                    tc::tma_load_2d(sa, &tmA, full_bar(s), kb * kBK, row0);
                    if (g.shrink) tc::tma_load_2d(sb, &tmS, full_bar(s), kb * kBK, g.adapter * a.t_cols);
                    else tc::tma_load_2d(sb, &tmB, full_bar(s), kb * kBK, n0);
                }
                // expand: per adapter of the row tile a ring slot with the first summand of t and B, and one with the
                // other two summands, which meet the same B
                int next_ad = g.p0 < g.p1 ? a.pairs[g.p0].adapter : -1;
                for (int p = g.p0; p < g.p1 && ok; ++p) {
                    const int adapter = next_ad;
                    if (p + 1 < g.p1) next_ad = a.pairs[p + 1].adapter;   // (in flight while this pair is waited for)
                    if (n_shrink > 0) {
                        // t of this pair is written by a shrink item, which comes earlier in the list and has
                        // therefore been claimed by a running block: wait until its four epilogue warps have
                        // published, then order the TMA read after their writes
                        const long long t0 = clock64();
                        while (ld_acquire(a.t_ready + p) < 4) {
                            if (*abort_flag || clock64() - t0 > tc::kWaitCycleLimit) { *abort_flag = 1; ok = false; break; }
                        }
                        if (!ok) break;
                        fence_proxy_async_global();
                    }
                    const int blk = n0 < a.Nq ? 0 : (n0 < a.Nq + a.Nkv ? 1 : 2);
                    for (int slot = 0; slot < t_slots; ++slot, ++kc) {
                        const int s = kc % kStages;
                        if (!tc::mbar_wait(empty_bar(s), ((kc / kStages) & 1) ^ 1, abort_flag)) { ok = false; break; }
                        const uint32_t sa = smem_base + s * S::kStageBytes, sb = sa + S::kABytes;
                        const int part = slot * (slot > 0 ? S::kSummandsPerSlot : 1) - (slot > 0 ? S::kSummandsPerSlot - 1 : 0);
                        const bool two = slot > 0 && S::kSummandsPerSlot == 2;
                        tc::mbar_arrive_expect_tx(full_bar(s), slot == 0 ? S::kStageBytes : (two ? 2 : 1) * S::kABytes);
                        tc::tma_load_2d(sa, &tmT, full_bar(s), blk * kTensorRP, (p * a.t_parts + part) * kBM);
                        if (slot == 0) tc::tma_load_2d(sb, &tmL, full_bar(s), 0, adapter * a.total_adapter_rows + n0);
                        else if (two) tc::tma_load_2d(sb, &tmT, full_bar(s), blk * kTensorRP, (p * a.t_parts + part + 1) * kBM);
                    }
                }
            }
            if (!ok) {
                // give copies already in flight time to land before the block's shared memory is released
                const uint32_t first = kc > (uint32_t)kStages ? kc - kStages : 0;
                for (uint32_t i = first; i < kc; ++i) {
                    const long long t0 = clock64();
                    while (!tc::mbar_try_wait(full_bar(i % kStages), (i / kStages) & 1) &&
                           clock64() - t0 < tc::kWaitCycleLimit) {}
                }
            }
        }
    } else if (warp == 1) {
        {
            // ------------------------------ MMA issuer ------------------------------
            // The whole warp walks the schedule (uniform control flow keeps descriptors and loop state in uniform
            // registers, which is what lets the issue rate reach the tensor pipe's); one elected lane issues the
            // tensor-core instructions and their commits.
            const bool leader = tc::elect_one();
            auto wait_all = [&](uint32_t bar, uint32_t parity) {
                return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, abort_flag));
            };
            constexpr uint32_t idesc_main = tc::idesc_bf16_f32(kBM, BN);
            const uint32_t idesc_shrink = tc::idesc_bf16_f32(kBM, a.t_cols);
            uint32_t kc = 0, it = 0;
            bool ok = true;
            while (ok) {
                const int item = ring.take(abort_flag);
                if (item < 0) { ok = item == -1; break; }
                const GemmItem g = decode_item(a, item, n_shrink, p_base, n_n, BN);
                // MMA steps of the row tile's adapters, one per lane, loaded while the main loop runs
                const int my_steps = g.p0 + lane < g.p1 ? rank_steps(a, a.pairs[g.p0 + lane].adapter) : 0;
                const uint32_t idesc = g.shrink ? idesc_shrink : idesc_main;
                const uint32_t acc = it & 1;
                if (!wait_all(acce_bar(acc), ((it >> 1) & 1) ^ 1)) { ok = false; break; }
                tc::tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int kb = 0; kb < kb_main; ++kb, ++kc) {
                    const int s = kc % kStages;
                    if (!wait_all(full_bar(s), (kc / kStages) & 1)) { ok = false; break; }
                    tc::tc_fence_after();
                    const uint32_t sa = smem_base + s * S::kStageBytes, sb = sa + S::kABytes;
                    const uint64_t da = tc::smem_desc_k_sw128(sa), db = tc::smem_desc_k_sw128(sb);
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k)
                            tc::mma_bf16(d_tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
                        tc::mma_commit(empty_bar(s));  // slot reusable once these MMAs have read it
                    }
                }
                for (int p = g.p0; p < g.p1 && ok; ++p) {
                    const int at = p - g.p0;
                    const int steps = at < 32 ? __shfl_sync(0xffffffffu, my_steps, at) : rank_steps(a, a.pairs[p].adapter);
                    uint64_t db = 0;
                    for (int slot = 0; slot < t_slots; ++slot) {
                        const int s = (kc + slot) % kStages;
                        if (!wait_all(full_bar(s), ((kc + slot) / kStages) & 1)) { ok = false; break; }
                        tc::tc_fence_after();
                        const uint32_t sa = smem_base + s * S::kStageBytes, sb = sa + S::kABytes;
                        const uint64_t da = tc::smem_desc_k_sw128(sa), db2 = tc::smem_desc_k_sw128(sb);
                        if (slot == 0) db = db2;
                        if (leader) {
                            for (int k = 0; k < steps; ++k) tc::mma_bf16(d_tmem, da + 2 * k, db + 2 * k, idesc, 1u);
                            if (slot > 0 && S::kSummandsPerSlot == 2)   // (the third summand lies where B lies in the first slot)
                                for (int k = 0; k < steps; ++k) tc::mma_bf16(d_tmem, db2 + 2 * k, db + 2 * k, idesc, 1u);
                        }
                    }
                    if (!ok) break;
                    for (int slot = 0; slot < t_slots; ++slot, ++kc)   // B is read up to the last summand
                        if (leader) tc::mma_commit(empty_bar(kc % kStages));
                }
                if (!ok) break;
                if (leader) tc::mma_commit(accf_bar(acc));      // accumulator complete
                ++it;
            }
            if (!ok && leader) {
                tc::mma_commit(drain_bar);          // wait (bounded) for tensor-core work still in flight
                const long long t0 = clock64();
                while (!tc::mbar_try_wait(drain_bar, 0) && clock64() - t0 < tc::kWaitCycleLimit) {}
            }
        }
    } else {
        // ------------------------------ epilogue (warps 2..5) ------------------------------
        const int q = warp & 3;  // tensor-memory lane quarter this warp may read
        const bool any_odd = a.pairs != nullptr && *a.any_odd != 0;
        uint32_t it = 0;
        bool ok = true;
        while (ok) {
            const int item = ring.take(abort_flag);
            if (item < 0) break;
            const GemmItem g = decode_item(a, item, n_shrink, p_base, n_n, BN);
            const int n0 = g.n0, row = g.m * kBM + q * 32 + lane;   // this thread's row
            const uint32_t acc = it & 1;
            if (!tc::mbar_wait(accf_bar(acc), (it >> 1) & 1, abort_flag)) { ok = false; break; }
            tc::tc_fence_after();
            const bool row_ok = row < a.M;
            if (g.shrink) {
                // t = s A x of this pair, zero in the rows that do not use the adapter
                const float scale = __int_as_float(a.adapters[g.adapter * a.ad_stride + 1]);
                const bool use = row_ok && a.row_adapter[row] == g.adapter;
                __nv_bfloat16 *trow = a.t + ((size_t)g.p0 * a.t_parts * kBM + q * 32 + lane) * a.t_cols;
                const int rpad = a.adapters[g.adapter * a.ad_stride];
#pragma unroll 1
                for (int c = 0; c < a.t_cols && c < BN; c += 32) {
                    if ((c & (kTensorRP - 1)) >= rpad) continue;   // (columns that no MMA step reads)
                    uint32_t v[32];
                    tc::tmem_ld_32x32(tmem_base + acc * BN + c + ((uint32_t)(q * 32) << 16), v);
                    tc::tmem_ld_wait();
                    tc::store_t_warp(reinterpret_cast<float(&)[32]>(v), scale, use, trow + c, a.t_cols, a.t_parts, kBM * a.t_cols);
                }
                tc::tc_fence_before();
                // publish: the rows are read by other blocks through TMA (async proxy)
                fence_proxy_async_global();
                __threadfence();
                __syncwarp();
                if (lane == 0) {
                    atomicAdd(a.t_ready + g.p0, 1);
                    tc::mbar_arrive(acce_bar(acc));
                }
                ++it;
                continue;
            }
            __nv_bfloat16 *orow = a.out + (size_t)row * a.ldo + n0;
            const __nv_bfloat16 *rrow = a.residual ? a.residual + (size_t)row * a.ldo + n0 : nullptr;
            // fused KV append: where this row's k / v columns go in the page pool
            int kv_page = -1, kv_row = 0;
            if (a.kv_pool != nullptr && row_ok && n0 + BN > a.Nq) {
                const int slot = a.slot_map[row];
                if (slot >= 0) {
                    kv_page = slot / a.kv_page_size;
                    kv_row = slot % a.kv_page_size;
                    if (kv_page >= a.kv_num_pages) { report(a.status, ALORA_ERR_PAGE_RANGE); kv_page = -1; }
                }
            }
            const uint32_t acc_addr = tmem_base + acc * BN + ((uint32_t)(q * 32) << 16);
            auto put8 = [&](int c, float (&f)[8]) {   // columns c .. c + 7 of the tile
                if (rrow) {
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
                const int kc = n0 + c - a.Nq;   // column inside [k | v]
                if (kv_page >= 0 && kc >= 0) {
                    const int plane = kc >= a.Nkv ? 1 : 0, c2 = kc - plane * a.Nkv;
                    const int head = c2 >> a.kv_hd_shift, dd = c2 & ((1 << a.kv_hd_shift) - 1);
                    __nv_bfloat16 *dst = a.kv_pool +
                        ((((size_t)kv_page * 2 + plane) * a.kv_heads + head) * a.kv_page_size + kv_row << a.kv_hd_shift) + dd;
                    *reinterpret_cast<uint4 *>(dst) = o;
                }
            };
            bool own_pass = false;   // the row's adapter has a B with an Inf or NaN
            if (any_odd && row_ok && g.p0 < g.p1) {
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
                        if (n0 + c + 8 * j >= a.N) break;
                        put8(c + 8 * j, reinterpret_cast<float(&)[8]>(v[8 * j]));
                    }
                }
            }
            if (__any_sync(0xffffffffu, own_pass)) {
                tc::OddRow odd;
                if (own_pass) {
                    const int k = a.row_adapter[row];
                    int p = g.p0;
                    while (p + 1 < g.p1 && a.pairs[p].adapter != k) ++p;
                    if (a.shrink) ld_acquire(a.t_ready + p);   // (complete since the tile's K blocks were loaded; orders the reads)
                    odd.t = a.t + ((size_t)p * a.t_parts * kBM + q * 32 + lane) * a.t_cols;
                    odd.b = a.b_all + (size_t)k * a.N * kTensorRP;
                    odd.n = a.adapters[k * a.ad_stride];
                    odd.parts = a.t_parts; odd.part_stride = kBM * a.t_cols;
                }
                const int blk = n0 < a.Nq ? 0 : (n0 < a.Nq + a.Nkv ? 1 : 2);
#pragma unroll 1
                for (int c = 0; c < BN && n0 + c < a.N; c += 8) {
                    uint32_t v[8];
                    tc::tmem_ld_32x8(acc_addr + c, v);
                    tc::tmem_ld_wait();
                    if (!own_pass) continue;
                    odd.add8(reinterpret_cast<float(&)[8]>(v), n0 + c, blk);
                    put8(c, reinterpret_cast<float(&)[8]>(v));
                }
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(acce_bar(acc));  // accumulator may be overwritten
            ++it;
        }
    }

    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) report(a.status, ALORA_ERR_TIMEOUT);
    if (threadIdx.x == 0) tc::item_counter_release(a.item_counters, a.t_ready + p_base, n_shrink);
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ---- host side -------------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn tensor_map_encoder() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

// Row-major bf16 matrix [rows][cols] (row pitch ld elements) viewed in boxes of 64 columns x box_rows
// rows, 128-byte swizzle, out-of-range elements read as zero.
bool make_tensor_map_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld,
                          uint32_t box_rows) {
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn || !base || rows == 0 || cols == 0) return false;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) || (ld * 2) % 16 != 0 || box_rows == 0 || box_rows > 256) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)kBK, box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN>
static bool launch_gemm_bn(alora_ctx *ctx, const CUtensorMap &tmA, const CUtensorMap &tmB, const CUtensorMap &tmT,
                           const CUtensorMap &tmL, const CUtensorMap &tmS, const GemmArgs &args, int max_items,
                           cudaStream_t s) {
    static bool attr_set[64] = {};  // one per instantiation
    const int dev = ctx->cfg.device;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        if (cudaFuncSetAttribute(gemm_tcgen05_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 GemmSmem<BN>::kTotal) != cudaSuccess)
            return false;
        attr_set[dev] = true;
    }
    const int grid = std::max(1, std::min(ctx->sm_count, max_items));
    if (launch_kernel(gemm_tcgen05_kernel<BN>, dim3(grid), dim3(kGemmThreads), GemmSmem<BN>::kTotal, s, true, tmA, tmB, tmT, tmL,
                      tmS, args) != cudaSuccess)
        return false;
    return true;
}

bool launch_shrink_tc(alora_ctx *ctx, const CUtensorMap &tmX, const RankMaps &tmA, const AdapterDev *adapters,
                      int T, int K, int max_pairs, int t_parts, cudaStream_t s);  // shrink_tcgen05.cu

// Picks the column-tile width of the q/k/v projection: 256 when the block boundaries allow it, else 128; 64 for batches of
// at most 128 rows, where the kernel streams the weights once and more, narrower tiles put more SMs to work.
static int pick_bn(int N, int Nq, int Nkv, int T) {
    if (T <= kBM && N >= 64 * 48 && Nq % 64 == 0 && Nkv % 64 == 0) return 64;
    if (Nq % 256 == 0 && Nkv % 256 == 0) return 256;
    if (Nq % 128 == 0 && Nkv % 128 == 0) return 128;
    return 0;
}

// q/k/v projection of one layer on the tensor cores: shrink (t = s A x of the (row tile, adapter) pairs), then the
// base GEMM with the expand step fused.  Returns kernels launched, or -1 when the shape is unsupported.
int launch_project_duo_tc(alora_ctx *ctx, int layer, const void *hidden, int T, int R, void *qkv, cudaStream_t s,
                           void *kv_pool, int num_pages);  // gemm_duo_tcgen05.cu

// Whether the shrink of a launch of `items` projection items is a kernel of its own.  As leading items of the projection
// it is free unless it makes another round over the blocks of a launch of one or two rounds (a round is 24 .. 31 us at
// hidden 4096, a kernel for a few pairs 8 us); a kernel for many pairs takes rounds of its own.  The number of pairs is
// an upper bound from the row and request counts, so that the choice does not depend on the mode.
bool shrink_apart(const alora_ctx *ctx, int T, int R, int items) {
    const int G = ctx->sm_count, n = pair_bound(ctx, T, R);
    const int rounds = (items + G - 1) / G;
    return rounds <= 2 && (items + n + G - 1) / G > rounds && n * 8 <= 4 * G;
}

bool skinny_route(const alora_ctx *ctx, int T, int N, int K, bool lora, int Nq, int Nkv);   // gemm_skinny_tcgen05.cu: at most 128
                                  // rows, more adapters than the one-launch kernel takes
int launch_skinny_tc(alora_ctx *ctx, const void *x, const CUtensorMap &tmW, const CUtensorMap *tmA16,
                     const AdapterDev *adapters, const void *b_all, int T, int K, int N, int Nq, int Nkv, void *out,
                     void *kv_pool, int num_pages, int layer, cudaStream_t s);

bool few_cluster_route(const alora_ctx *ctx, int T, int R, int N, int K, bool lora, int Nq, int Nkv);   // gemm_few_cluster.cu
int launch_few_cluster(alora_ctx *ctx, const void *x, const void *W, const RankMaps *tmA, const FewRowMeta *meta,
                       const void *b_all, int T, int R, int K, int N, int Nq, int Nkv, void *out, const void *residual, void *kv_pool,
                       int num_pages, bool x_early, cudaStream_t s, bool glu = false);

// More than 128 rows take the one-launch route only in a context without adapters on the MLP block: those need the (row tile,
// adapter) pairs, which that route's metadata step does not build, and a call in which none of them applies has to take the
// route of the others (rows without a delta keep their bits).
static bool few_cluster_rows(const alora_ctx *ctx, int T) {
    if (T > kFewRowMax)
        for (int n : ctx->mlp_n_adapters) if (n > 0) return false;
    return true;
}
static bool project_few_cluster(const alora_ctx *ctx, int layer, int T, int R) {
    const Dims &d = ctx->d;
    if (!few_cluster_rows(ctx, T)) return false;
    return few_cluster_route(ctx, T, R, d.N, d.H, ctx->layer_has_adapter[layer] != 0, d.Nq, d.Nkv);
}

// Whether the q/k/v projection of a batch of T rows on this layer takes the few-row route (the batch-metadata step
// then prepares that route's adapter facts instead of row tiles).
bool project_is_few_row(const alora_ctx *ctx, int layer, int T, int R) {
    if (ctx->cfg.dtype != ALORA_DTYPE_BF16 || layer < 0 || layer >= ctx->cfg.n_layers) return false;
    const Dims &d = ctx->d;
    return project_few_cluster(ctx, layer, T, R) || skinny_route(ctx, T, d.N, d.H, ctx->layer_has_adapter[layer] != 0, d.Nq, d.Nkv);
}

int launch_project_tc(alora_ctx *ctx, int layer, const void *hidden, int T, int R, void *qkv, cudaStream_t s, void *kv_pool,
                      int num_pages) {
    if (T == 0) return 0;
    const Dims &d = ctx->d;
    const bool have_adapters = ctx->layer_has_adapter[layer];
    if (project_few_cluster(ctx, layer, T, R)) {
        ProfScope prof(ctx, KK_PROJECT, s);
        return launch_few_cluster(ctx, hidden, ctx->layers[layer].wqkv, &ctx->tc_maps[layer].a_rank,
                                  have_adapters ? ctx->d_skinny_meta + (size_t)layer * ctx->few_tiles : nullptr, ctx->tc_b_all[layer], T, R,
                                  d.H, d.N, d.Nq, d.Nkv, qkv, nullptr, kv_pool, num_pages, ctx->x_before_facts, s);
    }
    if (skinny_route(ctx, T, d.N, d.H, have_adapters, d.Nq, d.Nkv)) {
        ProfScope prof(ctx, KK_PROJECT, s);
        const TcLayerMaps &lm = ctx->tc_maps[layer];
        const AdapterDev *ads = ctx->d_adapters + (size_t)layer * ctx->cfg.max_adapters;
        return launch_skinny_tc(ctx, hidden, lm.wqkv[1], have_adapters ? &lm.a_rank.box[0] : nullptr,
                                have_adapters ? ads : nullptr, ctx->tc_b_all[layer], T, d.H, d.N, d.Nq, d.Nkv, qkv,
                                kv_pool, num_pages, layer, s);
    }
    {   // many rows: pairs of SMs (bracketed for the profile there, once the route is decided)
        const int r = launch_project_duo_tc(ctx, layer, hidden, T, R, qkv, s, kv_pool, num_pages);
        if (r != 0) return r;
    }
    const int BN = pick_bn(d.N, d.Nq, d.Nkv, T);
    if (BN == 0 || d.H % 8 != 0) return -1;
    CUtensorMap tmX, tmTt, tmX64;
    if (!make_tensor_map_bf16(&tmX, hidden, T, d.H, d.H, kBM)) return -1;
    const bool half_box = T <= kBM / 2;   // see GemmArgs::a_tile_bytes
    if (half_box && !make_tensor_map_bf16(&tmX64, hidden, T, d.H, d.H, kBM / 2)) return -1;
    if (!make_tensor_map_bf16(&tmTt, ctx->d_t, (uint64_t)ctx->t_slots * kBM, 3 * kTensorRP, 3 * kTensorRP, kBM)) return -1;
    const TcLayerMaps &lm = ctx->tc_maps[layer];
    const AdapterDev *ads = ctx->d_adapters + (size_t)layer * ctx->cfg.max_adapters;
    const int t_parts = T <= kSplitTTokens ? 3 : 1, max_pairs = have_adapters ? pair_bound(ctx, T, R) : 0;
    const int proj_items = ((T + kBM - 1) / kBM) * ((d.N + BN - 1) / BN);
    const bool fuse_shrink = have_adapters && BN == 256 && !shrink_apart(ctx, T, R, proj_items);
    int n = 0;
    if (have_adapters && !fuse_shrink) {
        ProfScope prof(ctx, KK_SHRINK, s);
        if (!launch_shrink_tc(ctx, tmX, lm.a_rank, ads, T, d.H, max_pairs, t_parts, s)) return -1;
        ++n;
    }
    {
        ProfScope prof(ctx, KK_PROJECT, s);
        GemmArgs g{};
        g.a_tile_bytes = half_box ? (kBM / 2) * kBK * 2 : 0;
        const CUtensorMap &tmXg = half_box ? tmX64 : tmX;
        g.M = T; g.N = d.N; g.K = d.H;
        g.out = (__nv_bfloat16 *)qkv; g.ldo = d.N; g.residual = nullptr;
        g.adapters = &ads->rpad;   // (address arithmetic only: padded rank and scale of an AdapterDev are neighbours)
        g.ad_stride = sizeof(AdapterDev) / 4; g.t_cols = 3 * kTensorRP;
        g.Nq = d.Nq; g.Nkv = d.Nkv; g.total_adapter_rows = d.N; g.status = ctx->d_status;
        g.item_counters = ctx->d_counts + 10;
        if (have_adapters) {
            g.pairs = ctx->d_pairs; g.pair_off = ctx->d_pair_off; g.t = (__nv_bfloat16 *)ctx->d_t; g.t_parts = t_parts;
            g.row_adapter = ctx->d_row_adapter; g.any_odd = ctx->d_counts + kOddAdapters;
            g.b_all = (const __nv_bfloat16 *)ctx->tc_b_all[layer];
        }
        if (kv_pool != nullptr) {
            int shift = 0;
            while ((1 << shift) < d.hd) ++shift;
            g.kv_pool = (__nv_bfloat16 *)kv_pool; g.slot_map = ctx->d_slot; g.kv_hd_shift = shift; g.kv_heads = d.Hkv;
            g.kv_page_size = d.page; g.kv_num_pages = num_pages;
        }
        if (fuse_shrink) { g.shrink = 1; g.t_ready = ctx->d_t_ready; }
        const int items = proj_items + (fuse_shrink ? max_pairs : 0);
        const bool ok = BN == 256
                            ? launch_gemm_bn<256>(ctx, tmXg, lm.wqkv[1], tmTt, lm.b_all_bn[1], lm.a_all, g, items, s)
                            : BN == 128
                                  ? launch_gemm_bn<128>(ctx, tmXg, lm.wqkv[0], tmTt, lm.b_all_bn[0], lm.a_all, g, items, s)
                                  : launch_gemm_bn<64>(ctx, tmXg, lm.wqkv[2], tmTt, lm.b_all_bn[2], lm.a_all, g, items, s);
        if (!ok) return -1;
        ++n;
    }
    return n;
}

int launch_linear_duo_tc(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y,
                         const void *residual, const LinearDelta *delta, bool glu, cudaStream_t s);  // gemm_duo_tcgen05.cu

// Dense projection y = x W^T (+ residual) for o_proj and the MLP matrices, with the gated delta of the MLP adapters where
// `delta` is given (more than kFewRowMax rows: a smaller batch may be on the few-row route, which builds no pairs).
int launch_linear_tc(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y,
                     const void *residual, const LinearDelta *delta, cudaStream_t s) {
    if (T == 0) return 0;
    if (K % 8 != 0 || N % 8 != 0) return -1;
    if (delta != nullptr && (T <= kFewRowMax || (N / delta->n_blk) % 256 != 0)) return -1;
    if (delta == nullptr && few_cluster_rows(ctx, T) && few_cluster_route(ctx, T, 0, N, K, false, N, 0)) {
        ProfScope prof(ctx, KK_LINEAR, s);
        return launch_few_cluster(ctx, x, W, nullptr, nullptr, nullptr, T, 0, K, N, N, 0, y, residual, nullptr, 0, false, s);
    }
    {
        const int r = launch_linear_duo_tc(ctx, x, W, T, K, N, y, residual, delta, false, s);   // many rows: pairs of SMs
        if (r != 0) return r;
    }
    ProfScope prof(ctx, KK_LINEAR, s);
    const int BN = N % 256 == 0 || N > 1024 ? 256 : 128;
    CUtensorMap tmX, tmW;
    if (!make_tensor_map_bf16(&tmX, x, T, K, K, kBM)) return -1;
    if (!make_tensor_map_bf16(&tmW, W, N, K, K, BN)) return -1;
    GemmArgs g{};
    g.M = T; g.N = N; g.K = K; g.out = (__nv_bfloat16 *)y; g.ldo = N;
    g.residual = (const __nv_bfloat16 *)residual; g.Nq = N; g.Nkv = 0; g.t_cols = kTensorRP;
    g.total_adapter_rows = N; g.status = ctx->d_status; g.item_counters = ctx->d_counts + 10;
    CUtensorMap tmT = tmX, tmA = tmW, tmB = tmW;
    if (delta != nullptr) {
        const uint64_t na = (uint64_t)std::max(1, ctx->cfg.max_adapters);
        g.t_cols = delta->n_blk * kTensorRP; g.t_parts = 1;
        if (delta->n_blk == 2) g.Nq = g.Nkv = N / 2;
        if (!make_tensor_map_bf16(&tmT, delta->t, (uint64_t)ctx->max_pairs * kBM, g.t_cols, g.t_cols, kBM)) return -1;
        if (!make_tensor_map_bf16(&tmA, delta->A, na * g.t_cols, K, K, g.t_cols)) return -1;
        if (!make_tensor_map_bf16(&tmB, delta->B, na * N, kTensorRP, kTensorRP, BN)) return -1;
        g.pairs = ctx->d_pairs; g.pair_off = ctx->d_pair_off; g.tile0 = delta->tile0; g.shrink = 1;
        g.adapters = &delta->table->rpad; g.ad_stride = sizeof(MlpAdapterDev) / 4;
        g.row_adapter = delta->row_adapter; g.t_ready = ctx->d_t_ready; g.t = (__nv_bfloat16 *)delta->t;
        g.any_odd = ctx->d_counts + kOddAdapters; g.b_all = (const __nv_bfloat16 *)delta->B;
    }
    const int items = ((T + kBM - 1) / kBM) * ((N + BN - 1) / BN) + (delta != nullptr ? ctx->max_pairs : 0);
    const bool ok = BN == 256 ? launch_gemm_bn<256>(ctx, tmX, tmW, tmT, tmB, tmA, g, items, s)
                              : launch_gemm_bn<128>(ctx, tmX, tmW, tmX, tmW, tmW, g, items, s);
    return ok ? 1 : -1;
}

// Gate and up projection with SwiGLU in the epilogue, for the batches of the few-row kernel and of the pairs of SMs; 0: nothing
// launched.  Not for few rows where the context has adapters on the MLP block: their expand step wants the rounded gate and up rows,
// and a call in which none of them applies has to take the route of the others.
// (So a stack call of few rows rounds gate and up before SwiGLU in such a context, and does not in one without these adapters.)
int launch_glu_tc(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y, cudaStream_t s, const LinearDelta *delta) {
    if (T == 0 || N % 16 != 0) return 0;
    if (delta == nullptr && few_cluster_rows(ctx, T) && few_cluster_route(ctx, T, 0, N, K, false, N, 0)) {
        for (int n : ctx->mlp_n_adapters) if (n > 0) return 0;
        ProfScope prof(ctx, KK_LINEAR, s);
        return launch_few_cluster(ctx, x, W, nullptr, nullptr, nullptr, T, 0, K, N, N, 0, y, nullptr, nullptr, 0, false, s, true);
    }
    return launch_linear_duo_tc(ctx, x, W, T, K, N, y, nullptr, delta, true, s);
}

int duo_project_tile(const alora_ctx *ctx, int layer, int T, int R);                       // gemm_duo_tcgen05.cu
int duo_linear_tile(const alora_ctx *ctx, int T, int K, int N, bool glu, bool adapted);

// The column tile of the kernel on pairs of SMs for one matrix of a layer (0 q/k/v, 1 o_proj, 2 gate / up with SwiGLU, 3 down), 0 where
// another kernel serves it: the order of the launchers above.
int pair_tile(const alora_ctx *ctx, int layer, int matrix, int T, int R, bool adapted) {
    const Dims &d = ctx->d;
    if (T == 0) return 0;
    if (matrix == 0) {
        if (project_few_cluster(ctx, layer, T, R) || skinny_route(ctx, T, d.N, d.H, ctx->layer_has_adapter[layer], d.Nq, d.Nkv)) return 0;
        return duo_project_tile(ctx, layer, T, R);
    }
    const int K = matrix == 1 ? d.Nq : matrix == 2 ? d.H : d.I, N = matrix == 2 ? 2 * d.I : d.H;
    if (!adapted && few_cluster_rows(ctx, T) && few_cluster_route(ctx, T, 0, N, K, false, N, 0)) return 0;
    return duo_linear_tile(ctx, T, K, N, matrix == 2, adapted);
}

// Tensor maps that depend only on registered weights; (re)built when weights or adapters are set.
bool build_layer_maps(alora_ctx *ctx, int layer) {
    const Dims &d = ctx->d;
    TcLayerMaps &lm = ctx->tc_maps[layer];
    const LayerWeights &lw = ctx->layers[layer];
    bool ok = true;
    if (lw.wqkv) {
        ok &= make_tensor_map_bf16(&lm.wqkv[0], lw.wqkv, d.N, d.H, d.H, 128);
        ok &= make_tensor_map_bf16(&lm.wqkv[1], lw.wqkv, d.N, d.H, d.H, 256);
        ok &= make_tensor_map_bf16(&lm.wqkv[2], lw.wqkv, d.N, d.H, d.H, 64);
    }
    const size_t na = (size_t)std::max(1, ctx->cfg.max_adapters);
    ok &= make_tensor_map_bf16(&lm.a_all, ctx->tc_a_all[layer], na * 3 * kTensorRP, d.H, d.H, 3 * kTensorRP);
    for (int i = 0; i < 4; ++i) ok &= make_tensor_map_bf16(&lm.a_rank.box[i], ctx->tc_a_all[layer], na * 3 * kTensorRP, d.H, d.H, 16 * (i + 1));
    ok &= make_tensor_map_bf16(&lm.b_all_bn[0], ctx->tc_b_all[layer], na * d.N, kTensorRP, kTensorRP, 128);
    ok &= make_tensor_map_bf16(&lm.b_all_bn[1], ctx->tc_b_all[layer], na * d.N, kTensorRP, kTensorRP, 256);
    ok &= make_tensor_map_bf16(&lm.b_all_bn[2], ctx->tc_b_all[layer], na * d.N, kTensorRP, kTensorRP, 64);
    return ok;
}

}  // namespace alora
