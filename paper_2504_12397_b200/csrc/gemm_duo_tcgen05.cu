// Dense contractions of many rows on pairs of SMs (tcgen05.mma.cta_group::2) with the aLoRA delta fused in: the gated q/k/v
// projection (Eq. 2 / Eq. 5), and the o_proj / MLP matrices of the layer stack (residual in the epilogue; gate and up
// projection with SwiGLU in the epilogue; with adapters on the MLP block the same gated delta).
//
// A cluster of two blocks owns FOUR row tiles of 128 rows (a "quad") x one column tile of `bn` columns: block r of the cluster
// holds the rows of tiles r and 2 + r and half of the W tile, the even block issues the MMAs for both (256 rows x bn), and
// each block's half of every product lies in its own tensor memory.  What bounds such a kernel on this chip is the shared
// memory: 128 bytes a cycle for what TMA brings in and what the tensor cores read.  Per 64-wide K block of 256 x 256
// outputs an SM on its own needs 64 KB in + 96 KB read = 1250 cycles for 1024 of tensor work (1230 measured); here it is
// 48 + 64 KB, below the tensor time.  32768 x 6144 x 4096 at the power limit: 1420 us on single SMs, 1270 here.
//
// Adapters: for every quad the adapters that occur in it (d_quads, from the batch-metadata step).  t = s A_k x of a
// quad comes from leading "shrink items" of the same launch (rows that do not use the adapter are zero); a column tile
// appends t B_k^T of each of its quad's adapters to its K loop, one K block per adapted matrix (q / k / v, gate / up) that it
// touches; B rows outside the matrix read as zero.  An adapter whose B holds an Inf or NaN is left out of the products
// and added by the epilogue to its own rows (tc::OddRow).
//
//   warp 0   TMA producer (4 slots of 48 KB); that of the even block also hands the work items out
//   warp 1   MMA issuer (even block; the whole warp walks, an elected lane issues)
//   warps 2-9  epilogue: tcgen05.ld one row per thread, bf16, through shared memory and TMA to the output, the new k and v
//            rows to the page pool, or t for shrink items
// The two row tiles of a block accumulate in the two halves of tensor memory; the epilogue takes a half into registers while the
// tensor cores still or already work on the other, and finishes it underneath the next item.
// All waits are bounded; on expiry ALORA_ERR_TIMEOUT is recorded and the blocks leave normally.
#include <algorithm>

#include "alora_internal.h"
#include "tc_common.cuh"
#include "claim_order.h"

namespace alora {

namespace {
constexpr int kBKd = 64, kThreadsD = 320;          // producer, issuer, 2 x 4 epilogue warps
constexpr int kTensorRP = 64;                      // the tensor path stores adapters padded to 64 rank columns
constexpr int kTileBytesD = 128 * kBKd * 2;        // one row tile's x (or t) block: 16 KB
constexpr int kMaxBn = 256;
struct DuoSmem {
    static constexpr int kStages = 4;
    static constexpr int kStageBytes = 2 * kTileBytesD + kMaxBn / 2 * kBKd * 2;   // 48 KB
    static constexpr int kOutOff = kStages * kStageBytes;     // per epilogue warp two buffers of 32 rows x 32 bf16 columns
    static constexpr int kOutBytes = 32 * 64;
    static constexpr int kBarOff = kOutOff + 8 * 2 * kOutBytes;
    static constexpr int kTotal = kBarOff + 512 + 1024;
};
enum DuoMode { kDuoQkv = 0, kDuoLinear = 1, kDuoGlu = 2 };

struct DuoArgs {
    const TilePair *quads;          // (quad, adapter) entries, nullptr: no adapters in this launch
    const int32_t *quad_off;        // [quads + 1] first entry of each quad
    int quad0;                      // quad of the batch that holds this launch's first row
    int t_cols;                     // columns of t: 64 padded rank columns per adapted matrix
    const int32_t *adapters;        // per adapter `ad_stride` words, the first three: padded rank, scale (float), b_odd
    int ad_stride;
    int M, N, K, Nq, Nkv;           // N: rows of W; Nq, Nkv: the q/k/v blocks of the fused row
    int bn;                         // column tile (a multiple of 32; kDuoGlu: bn / 2 gate and the same bn / 2 up columns)
    int n_out;                      // output columns (kDuoGlu: N / 2)
    int b_rows;                     // rows of the B map (an out-of-range row reads as zero)
    __nv_bfloat16 *out;
    int ldo;
    const __nv_bfloat16 *residual;  // optional, same layout as out, may alias it
    const int32_t *row_adapter;     // [M] applied adapter per row (shrink items: which rows of t are kept)
    const int32_t *any_odd;         // not 0: an adapter of the context may have b_odd set
    const __nv_bfloat16 *b_all;     // the launch's B rows of all adapters, [adapter][N][64] (read for rows of those)
    int32_t *t_ready;               // [entry] epilogue warps that have published their part of t
    __nv_bfloat16 *t;               // [entry][kParts][512][t_cols]
    // KV append fused into the epilogue (nullptr: off): the k and v columns then go to the page pool only
    __nv_bfloat16 *kv_pool;
    const int32_t *slot_map;
    int kv_hd_shift, kv_heads, kv_page_size, kv_num_pages;
    int32_t *item_counters;         // [2] next unclaimed work item of the launch, blocks that have finished
    int32_t *status;
};

__device__ __forceinline__ int ld_acquire_d(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// ---- two-block forms of the operations in tc_common.cuh.  `bar` of the loads is a cluster address (the even block's barrier).
__device__ __forceinline__ uint32_t cluster_rank_d() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_d() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
    if (try_wait_cluster(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (try_wait_cluster(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > tc::kWaitCycleLimit) { *abort_flag = 1; return false; }
    }
}
__device__ __forceinline__ void tma2_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"((uint64_t)map), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma2_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"((uint64_t)map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void mma2_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrives on the barrier at this address in both blocks once all MMAs issued so far by this thread have completed
__device__ __forceinline__ void mma2_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];\n\tcp.async.bulk.commit_group;"
                 ::"l"((uint64_t)map), "r"(src), "r"(c0), "r"(c1) : "memory");
}

// (none for a B with an Inf or NaN: see TilePair)
__device__ __forceinline__ int rank_steps(const DuoArgs &a, int adapter) {
    const int32_t *ad = a.adapters + adapter * a.ad_stride;
    const int rpad = ad[0], odd = ad[2];
    return odd ? 0 : rpad / 16;
}

// One work item: a shrink item of (quad, adapter) entry e0 (all of its rows, or one half), or a quad x a column tile with the
// quad's entries e0 .. e1.
struct DuoItem {
    int quad, e0, e1, n0, adapter;
    int h0, halves;   // first half of the quad (256 rows: tiles 2 h0 and 2 h0 + 1), and how many
    bool shrink;
    __device__ __forceinline__ int tile(int h, uint32_t crank) const { return 4 * quad + 2 * (h0 + h) + (int)crank; }
};
// kDuoQkv: the column tiles of a quad are neighbours in the list; else the quads of a column tile (the clusters that
// run together share a W tile), beginning with another one in every column: a last quad of one or two row tiles takes half as
// long, and would always fall to the same clusters.
template <int kMode>
__device__ __forceinline__ DuoItem decode_duo(const DuoArgs &a, int item, int n_shrink, int split, int e_base, int n_m, int n_q, int n_n) {
    DuoItem g;
    g.n0 = 0; g.adapter = -1; g.e0 = g.e1 = 0;
    g.shrink = item < n_shrink;
    if (g.shrink) {
        g.e0 = g.e1 = e_base + item / split;
        const TilePair p = a.quads[g.e0];
        g.quad = p.tile - a.quad0;
        g.adapter = p.adapter;
    } else {
        const int j = item - n_shrink;
        g.quad = kMode == kDuoQkv ? j / n_n : (j % n_q + j / n_q) % n_q;
        g.n0 = (kMode == kDuoQkv ? j % n_n : j / n_q) * (kMode == kDuoGlu ? a.bn / 2 : a.bn);
        if (a.quads) {
            g.e0 = a.quad_off[a.quad0 + g.quad];
            g.e1 = a.quad_off[a.quad0 + g.quad + 1];
        }
    }
    const int all = n_m - 4 * g.quad > 2 ? 2 : 1;
    g.h0 = g.shrink && split == 2 ? item & 1 : 0;
    g.halves = g.shrink && split == 2 ? (g.h0 < all ? 1 : 0) : all;
    return g;
}
// first row of q/k/v block `blk` in the fused row, and one past its last
__device__ __forceinline__ int blk_start(const DuoArgs &a, int blk) { return blk == 0 ? 0 : (blk == 1 ? a.Nq : a.Nq + a.Nkv); }
__device__ __forceinline__ int blk_end(const DuoArgs &a, int blk) { return blk == 0 ? a.Nq : (blk == 1 ? a.Nq + a.Nkv : a.N); }
// K blocks that an entry of the quad takes: one per adapted matrix; does the column tile at n0 touch matrix blk?
template <int kMode>
__device__ __forceinline__ bool touches(const DuoArgs &a, int n0, int blk) {
    return kMode != kDuoQkv || (n0 < blk_end(a, blk) && n0 + a.bn > blk_start(a, blk));
}

template <int kMode, int kParts>   // kParts: bf16 summands of t
__global__ void __launch_bounds__(kThreadsD, 1)
gemm_duo_tcgen05_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                        const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmS,
                        const __grid_constant__ CUtensorMap tmB0, const __grid_constant__ CUtensorMap tmB1,
                        const __grid_constant__ CUtensorMap tmB2, const __grid_constant__ CUtensorMap tmO, const DuoArgs a) {
    using S = DuoSmem;
    constexpr int kBlks = kMode == kDuoQkv ? 3 : (kMode == kDuoGlu ? 2 : 1);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_al = smem_raw + (smem_base - tc::smem_u32(smem_raw));
    const uint32_t bar0 = smem_base + S::kBarOff;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };                       // even block: both blocks' copies have landed
    auto empty_bar = [&](int s) { return bar0 + 8u * (S::kStages + s); };       // each block: its slot has been read
    auto accf_bar = [&](int h) { return bar0 + 8u * (2 * S::kStages + h); };       // each block: accumulators of half h complete
    auto acce_bar = [&](int h) { return bar0 + 8u * (2 * S::kStages + 2 + h); };   // even block: both blocks have drained half h
    const uint32_t drain_bar = bar0 + 8u * (2 * S::kStages + 4);
    // item ring: the even block's producer publishes to both blocks; consumers release in the even block
    const uint32_t ring0 = bar0 + 8u * (2 * S::kStages + 5);
    auto ring_full = [&](int s) { return ring0 + 8u * s; };
    auto ring_empty = [&](int s) { return ring0 + 8u * (tc::kItemSlots + s); };
    const uint32_t slots_addr = ring0 + 16u * tc::kItemSlots;
    volatile int *slots = reinterpret_cast<volatile int *>(smem_al + (slots_addr - smem_base));
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem_al + S::kBarOff + 384);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem_al + S::kBarOff + 392);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t crank = cluster_rank_d();
    const bool even = crank == 0;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S::kStages; ++s) { tc::mbar_init(full_bar(s), 1); tc::mbar_init(empty_bar(s), 1); }
        for (int h = 0; h < 2; ++h) { tc::mbar_init(accf_bar(h), 1); tc::mbar_init(acce_bar(h), 16); }
        tc::mbar_init(drain_bar, 1);
        // consumers of an item: issuing warp and eight epilogue warps here, producer and eight epilogue warps in the odd block
        for (int s = 0; s < tc::kItemSlots; ++s) { tc::mbar_init(ring_full(s), 1); tc::mbar_init(ring_empty(s), 18); }
        *abort_flag = 0;
        tc::fence_barrier_init();
        tc::fence_proxy_async();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32((const void *)tmem_slot)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc::tc_fence_before();
    __syncthreads();
    cluster_sync_d();   // the other block's barriers are ready
    tc::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    tc::grid_dep_launch();
    tc::grid_dep_wait();   // the metadata step's lists, the activations: all written by earlier kernels of the stream

    const int n_m = (a.M + 127) / 128, n_q = (n_m + 3) / 4;
    const int out_bn = kMode == kDuoGlu ? a.bn / 2 : a.bn;
    const int n_n = (a.n_out + out_bn - 1) / out_bn;
    const int e_base = a.quads ? a.quad_off[a.quad0] : 0;
    const int n_entries = a.quads ? a.quad_off[a.quad0 + n_q] - e_base : 0;
    const int kb_main = (a.K + kBKd - 1) / kBKd;
    const int cluster = (int)blockIdx.x / 2, n_clusters = (int)gridDim.x / 2;
    // t of a quad is needed at the end of the first round's items: shrink items of 256 rows are there earlier (t of 2048 rows
    // x 192 columns came 9 k cycles after the first column tiles wanted it, with items of 512 rows), if they bring no further round
    const int rounds = (n_q * n_n + n_entries + n_clusters - 1) / n_clusters;
    const int split = n_q * n_n + 2 * n_entries <= rounds * n_clusters ? 2 : 1;
    const int n_shrink = n_entries * split, total = n_shrink + n_q * n_n;
    const uint32_t peer_slots = map_to(slots_addr, 1);

    uint32_t n_taken = 0;   // items that went through this role
    // a consumer (a whole warp, or the odd block's producer thread): the next item, -1 at the end of the list, -2 when a
    // wait expired
    auto release = [&](int s) {
        if (even) tc::mbar_arrive(ring_empty(s));
        else arrive_cluster(map_to(ring_empty(s), 0));
    };
    auto take_warp = [&]() {
        const int s = n_taken % tc::kItemSlots;
        const bool got = __all_sync(0xffffffffu, wait_cluster(ring_full(s), (n_taken / tc::kItemSlots) & 1, abort_flag));
        const int item = got ? slots[s] : -2;
        __syncwarp();
        if (got && lane == 0) release(s);
        ++n_taken;
        return item;
    };

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------ TMA producer ------------------------------
            tc::tma_prefetch_desc(&tmX); tc::tma_prefetch_desc(&tmW);
            uint32_t kc = 0;        // ring slots filled so far
            bool ok = true;
            // Order of the cluster's items: shrink items (the head of the list) are claimed from a global counter, projection
            // items dealt by cluster index (claim_order.h), so that a column tile that waits for its quad's t waits for
            // a shrink item that a RUNNING cluster has claimed.
            bool shrink_phase = even && n_shrink > 0;
            int stat = cluster;
            if (shrink_phase && !claims_at_once(cluster, n_shrink)) {
                const long long t0 = clock64();
                while (ld_acquire_d(a.item_counters) < n_shrink && clock64() - t0 < 60000) {}
                if (ld_acquire_d(a.item_counters) >= n_shrink) shrink_phase = false;
            }
            const int half_bn = a.bn / 2;
            while (ok) {
                int item = -1;
                const int rs = n_taken % tc::kItemSlots;
                const uint32_t rph = (n_taken / tc::kItemSlots) & 1;
                if (even) {
                    if (shrink_phase) {
                        item = atomicAdd(a.item_counters, 1);
                        if (item >= n_shrink) { shrink_phase = false; item = -1; }
                    }
                    if (!shrink_phase && item < 0) item = next_dealt_item(stat, n_shrink, total, n_clusters);
                    if (!wait_cluster(ring_empty(rs), rph ^ 1, abort_flag)) { ok = false; break; }
                    slots[rs] = item;
                    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(peer_slots + 4u * rs), "r"(item) : "memory");
                    tc::mbar_arrive(ring_full(rs));
                    arrive_cluster(map_to(ring_full(rs), 1));
                } else {
                    if (!wait_cluster(ring_full(rs), rph, abort_flag)) { ok = false; break; }
                    item = slots[rs];
                    release(rs);
                }
                ++n_taken;
                if (item < 0) break;
                const DuoItem g = decode_duo<kMode>(a, item, n_shrink, split, e_base, n_m, n_q, n_n);
                // this block's half of B: rows of the W tile (kDuoGlu: the even block takes the gate, the odd one the up rows),
                // or of the adapter's A
                const int w_row = kMode == kDuoGlu ? g.n0 + (int)crank * (a.N / 2) : g.n0 + (int)crank * half_bn;
                const uint32_t b_bytes = (uint32_t)(g.shrink ? a.t_cols / 2 : half_bn) * kBKd * 2;
                const uint32_t all_bytes = 2u * (g.halves * kTileBytesD + b_bytes);
                auto begin_slot = [&](uint32_t bytes, uint32_t &sa, uint32_t &fb) {
                    const int s = kc % S::kStages;
                    if (!wait_cluster(empty_bar(s), ((kc / S::kStages) & 1) ^ 1, abort_flag)) return false;
                    sa = smem_base + s * S::kStageBytes;
                    if (even) tc::mbar_arrive_expect_tx(full_bar(s), bytes);
                    fb = map_to(full_bar(s), 0);
                    ++kc;
                    return true;
                };
                uint32_t sa, fb;
                for (int kb = 0; kb < kb_main && g.halves > 0; ++kb) {
                    if (!begin_slot(all_bytes, sa, fb)) { ok = false; break; }
                    for (int h = 0; h < g.halves; ++h) tma2_load_2d(sa + h * kTileBytesD, &tmX, fb, kb * kBKd, g.tile(h, crank) * 128);
                    if (g.shrink) tma2_load_2d(sa + 2 * kTileBytesD, &tmS, fb, kb * kBKd, g.adapter * a.t_cols + (int)crank * (a.t_cols / 2));
                    else tma2_load_2d(sa + 2 * kTileBytesD, &tmW, fb, kb * kBKd, w_row);
                }
                if (!ok) break;
                if (g.shrink) continue;
                // expand: per adapter of the quad, one K block per adapted matrix that the column tile touches
                int next_ad = g.e0 < g.e1 ? a.quads[g.e0].adapter : -1;
                for (int e = g.e0; e < g.e1 && ok; ++e) {
                    const int adapter = next_ad;
                    if (e + 1 < g.e1) next_ad = a.quads[e + 1].adapter;   // (in flight while this entry is waited for)
                    // t of this entry is written by shrink items (claimed by running clusters): wait until their sixteen
                    // epilogue warps have published, then order the TMA reads after it
                    const long long t0 = clock64();
                    while (ld_acquire_d(a.t_ready + e) < 16 * split) {
                        if (*abort_flag || clock64() - t0 > tc::kWaitCycleLimit) { *abort_flag = 1; ok = false; break; }
                    }
                    if (!ok) break;
                    asm volatile("fence.proxy.async.global;" ::: "memory");
                    for (int blk = 0; blk < kBlks; ++blk) {
                        if (!touches<kMode>(a, g.n0, blk)) continue;
                        for (int p = 0; p < kParts; ++p) {   // (the summands of t meet the same B tile)
                        if (!begin_slot(all_bytes, sa, fb)) { ok = false; break; }
                        for (int h = 0; h < g.halves; ++h)
                            tma2_load_2d(sa + h * kTileBytesD, &tmT, fb, blk * kTensorRP, (4 * (e * kParts + p) + 2 * h + (int)crank) * 128);
                        if (kMode == kDuoQkv)
                            tma2_load_3d(sa + 2 * kTileBytesD, blk == 0 ? &tmB0 : (blk == 1 ? &tmB1 : &tmB2), fb, 0,
                                         g.n0 + (int)crank * half_bn - blk_start(a, blk), adapter);
                        else if (kMode == kDuoGlu)   // (the half of the other matrix reads as zero)
                            tma2_load_2d(sa + 2 * kTileBytesD, &tmB0, fb, 0, blk == (int)crank ? adapter * a.N + w_row : a.b_rows);
                        else
                            tma2_load_2d(sa + 2 * kTileBytesD, &tmB0, fb, 0, adapter * a.N + w_row);
                        }
                        if (!ok) break;
                    }
                }
            }
            // The copies of this block have landed and its slots have been read before its shared memory is released.
            const long long t0 = clock64();
            for (uint32_t i = kc > (uint32_t)S::kStages ? kc - S::kStages : 0; i < kc; ++i)
                while (!try_wait_cluster(empty_bar(i % S::kStages), (i / S::kStages) & 1) && clock64() - t0 < tc::kWaitCycleLimit)
                    if (!ok && even && try_wait_cluster(full_bar(i % S::kStages), (i / S::kStages) & 1)) break;   // (landed, never to be read)
        }
    } else if (warp == 1) {
        if (even) {
            // ------------------------------ MMA issuer ------------------------------
            const bool leader = tc::elect_one();
            auto wait_all = [&](uint32_t bar, uint32_t parity) {
                return __all_sync(0xffffffffu, wait_cluster(bar, parity, abort_flag));
            };
            const uint32_t idesc_main = tc::idesc_bf16_f32(256, a.bn), idesc_shrink = tc::idesc_bf16_f32(256, a.t_cols);
            uint32_t kc = 0, it = 0;
            bool ok = true;
            for (;; ++it) {
                const int item = take_warp();
                if (item < 0) { ok = item == -1; break; }
                const DuoItem g = decode_duo<kMode>(a, item, n_shrink, split, e_base, n_m, n_q, n_n);
                // MMA steps of the quad's adapters, one per lane, loaded while the main loop runs
                const int my_steps = g.e0 + lane < g.e1 ? rank_steps(a, a.quads[g.e0 + lane].adapter) : 0;
                const uint32_t idesc = g.shrink ? idesc_shrink : idesc_main;
                const bool two = g.halves == 2;
                // K blocks [kb0, kb0 + n): the first half's MMAs, then the second half's
                auto step = [&](int kb0, int n, bool first, bool last) {
                    for (int i = 0; i < n; ++i) {
                        const uint32_t s = (kc + i) % S::kStages;
                        if (!wait_all(full_bar(s), ((kc + i) / S::kStages) & 1)) return false;
                        // a half's accumulator must have been drained by the previous item's epilogue before its first MMA
                        if (first && i == 0 && !wait_all(acce_bar(0), (it & 1) ^ 1)) return false;
                        tc::tc_fence_after();
                        const uint32_t sa = smem_base + s * S::kStageBytes;
                        const uint64_t da = tc::smem_desc_k_sw128(sa), db = tc::smem_desc_k_sw128(sa + 2 * kTileBytesD);
                        if (leader) {
#pragma unroll
                            for (int k = 0; k < kBKd / 16; ++k)
                                mma2_bf16(tmem_base, da + 2 * k, db + 2 * k, idesc, (kb0 | i | k) != 0 ? 1u : 0u);
                        }
                    }
                    if (leader && last) mma2_commit(accf_bar(0));
                    if (first) {
                        if (!wait_all(acce_bar(1), (it & 1) ^ 1)) return false;
                        tc::tc_fence_after();
                    }
                    for (int i = 0; i < n; ++i, ++kc) {
                        const uint32_t sa = smem_base + (kc % S::kStages) * S::kStageBytes;
                        const uint64_t da = tc::smem_desc_k_sw128(sa + kTileBytesD), db = tc::smem_desc_k_sw128(sa + 2 * kTileBytesD);
                        if (leader) {
                            if (two) {
#pragma unroll
                                for (int k = 0; k < kBKd / 16; ++k)
                                    mma2_bf16(tmem_base + 256, da + 2 * k, db + 2 * k, idesc, (kb0 | i | k) != 0 ? 1u : 0u);
                            }
                            mma2_commit(empty_bar(kc % S::kStages));  // slot reusable in both blocks once these MMAs have read it
                        }
                    }
                    if (leader && last) mma2_commit(accf_bar(1));
                    return true;
                };
                // The first and the last K blocks of an item are taken kEdge at a time, so that the tensor cores have work on one
                // half while the epilogue still drains, or already drains, the other.
                constexpr int kEdge = 2;
                const bool expand = g.e0 < g.e1;
                if (g.halves == 0) {   // (a shrink item without rows)
                    ok = wait_all(acce_bar(0), (it & 1) ^ 1) && wait_all(acce_bar(1), (it & 1) ^ 1);
                    if (leader) { mma2_commit(accf_bar(0)); mma2_commit(accf_bar(1)); }
                    if (!ok) break;
                    continue;
                }
                const int head = min(kEdge, kb_main), tail = min(kEdge, kb_main - head);
                ok = step(0, head, true, tail == 0 && !expand);
                for (int kb = head; ok && kb < kb_main - tail; ++kb) ok = step(kb, 1, false, false);
                if (ok && tail > 0) ok = step(kb_main - tail, tail, false, !expand);
                if (!ok) break;
                for (int e = g.e0; e < g.e1 && ok; ++e) {
                    const int at = e - g.e0;
                    const int steps = at < 32 ? __shfl_sync(0xffffffffu, my_steps, at) : rank_steps(a, a.quads[e].adapter);
                    for (int bp = 0; bp < kBlks * kParts; ++bp) {
                        if (!touches<kMode>(a, g.n0, bp / kParts)) continue;
                        const int s = kc % S::kStages;
                        if (!wait_all(full_bar(s), (kc / S::kStages) & 1)) { ok = false; break; }
                        tc::tc_fence_after();
                        const uint32_t sa = smem_base + s * S::kStageBytes;
                        const uint64_t db = tc::smem_desc_k_sw128(sa + 2 * kTileBytesD);
                        if (leader) {
                            for (int h = 0; h < g.halves; ++h) {
                                const uint64_t da = tc::smem_desc_k_sw128(sa + h * kTileBytesD);
                                for (int k = 0; k < steps; ++k) mma2_bf16(tmem_base + h * 256, da + 2 * k, db + 2 * k, idesc, 1u);
                            }
                            mma2_commit(empty_bar(s));
                        }
                        ++kc;
                    }
                }
                if (!ok) break;
                if (leader && expand) { mma2_commit(accf_bar(0)); mma2_commit(accf_bar(1)); }
            }
            if (!ok && leader) {
                mma2_commit(drain_bar);                 // wait (bounded) for tensor-core work still in flight
                const long long t0 = clock64();
                while (!tc::mbar_try_wait(drain_bar, 0) && clock64() - t0 < tc::kWaitCycleLimit) {}
            }
        }
    } else {
        // ------------------------------ epilogue: warps 2..5 the first columns of a tile, warps 6..9 the others ------------------------------
        const int q = warp & 3;           // tensor-memory lane quarter this warp may read
        const int part = (warp - 2) >> 2;
        const int r = q * 32 + lane, ql = lane & 3;
        const bool any_odd = a.quads != nullptr && *a.any_odd != 0;
        auto drained = [&](int h) {   // this half may be overwritten
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (even) tc::mbar_arrive(acce_bar(h));
                else arrive_cluster(map_to(acce_bar(h), 0));
            }
        };
        const uint32_t out_buf = smem_base + S::kOutOff + (warp - 2) * 2 * S::kOutBytes;
        uint8_t *out_row = smem_al + S::kOutOff + (warp - 2) * 2 * S::kOutBytes + lane * 64;
        uint32_t it = 0, n_out_bufs = 0;
        bool ok = true;
        for (; ok; ++it) {
            const int item = take_warp();
            if (item < 0) break;
            const DuoItem g = decode_duo<kMode>(a, item, n_shrink, split, e_base, n_m, n_q, n_n);
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                if (!__all_sync(0xffffffffu, wait_cluster(accf_bar(h), it & 1, abort_flag))) { ok = false; break; }
                tc::tc_fence_after();
                if (h >= g.halves) { drained(h); continue; }
                const int row = g.tile(h, crank) * 128 + r;
                const bool row_ok = row < a.M;
                const uint32_t acc_addr = tmem_base + h * 256 + ((uint32_t)(q * 32) << 16);
                if (g.shrink) {
                    // t = s A x of this entry, zero in the rows that do not use the adapter
                    const bool use = row_ok && a.row_adapter[row] == g.adapter;
                    const float scale = __int_as_float(a.adapters[g.adapter * a.ad_stride + 1]);
                    const int rpad = a.adapters[g.adapter * a.ad_stride];
                    __nv_bfloat16 *trow = a.t + ((size_t)(4 * g.e0 * kParts + 2 * (g.h0 + h) + (int)crank) * 128 + r) * a.t_cols;
#pragma unroll 1
                    for (int c = part * 32; c < a.t_cols; c += 64) {
                        if ((c & (kTensorRP - 1)) >= rpad) continue;   // (columns that no MMA step reads)
                        uint32_t v[32];
                        tc::tmem_ld_32x32(acc_addr + c, v);
                        tc::tmem_ld_wait();
                        tc::store_t_warp(reinterpret_cast<float(&)[32]>(v), scale, use, trow + c, a.t_cols, kParts, kQuadRows * a.t_cols);
                    }
                    // (published below: the rows are read by other blocks through TMA)
                    asm volatile("fence.proxy.async.global;" ::: "memory");
                    __threadfence();
                    drained(h);
                    continue;
                }
                bool own_pass = false;   // the row's adapter has a B with an Inf or NaN
                if (any_odd && row_ok && g.e0 < g.e1) {
                    const int k = a.row_adapter[row];
                    own_pass = k >= 0 && a.adapters[k * a.ad_stride + 2] != 0;
                }
                // fused KV append: where this row's k / v columns go in the page pool (element offset of head 0, dim 0 in the
                // page; -1: nowhere)
                long long kv_at = -1;
                if (kMode == kDuoQkv && a.kv_pool != nullptr && row_ok && g.n0 + a.bn > a.Nq) {
                    const int slot = a.slot_map[row];
                    if (slot >= 0) {
                        const int page = slot / a.kv_page_size;
                        if (page >= a.kv_num_pages) report(a.status, ALORA_ERR_PAGE_RANGE);
                        else kv_at = ((long long)page * 2 * a.kv_heads * a.kv_page_size + slot % a.kv_page_size) << a.kv_hd_shift;
                    }
                }
                const size_t row4 = (size_t)(row & ~3);
                auto kv_put = [&](long long at, int col, uint4 o) {   // columns col .. col + 7 of the fused row
                    const int kcol = col - a.Nq;
                    if (at < 0) return;
                    const int plane = kcol >= a.Nkv ? 1 : 0, c2 = kcol - plane * a.Nkv;
                    const int head = c2 >> a.kv_hd_shift, dd = c2 & ((1 << a.kv_hd_shift) - 1);
                    *reinterpret_cast<uint4 *>(a.kv_pool + at + (((size_t)plane * a.kv_heads + head) * a.kv_page_size << a.kv_hd_shift) + dd) = o;
                };
                auto add_res8 = [&](float (&f)[8], uint4 rv) {
                    const uint32_t rw[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const __nv_bfloat162 b2 = *reinterpret_cast<const __nv_bfloat162 *>(&rw[e]);
                        f[2 * e] += __low2float(b2);
                        f[2 * e + 1] += __high2float(b2);
                    }
                };
                auto pack8 = [&](const float (&f)[8]) {
                    return make_uint4(tc::pack_bf16(f[0], f[1]), tc::pack_bf16(f[2], f[3]), tc::pack_bf16(f[4], f[5]), tc::pack_bf16(f[6], f[7]));
                };
                // 8 columns of this lane's own row
                auto put_own8 = [&](int col, float (&f)[8]) {
                    if (kMode == kDuoLinear && a.residual) add_res8(f, *reinterpret_cast<const uint4 *>(a.residual + (size_t)row * a.ldo + col));
                    const uint4 o = pack8(f);
                    if (kMode == kDuoQkv && a.kv_pool != nullptr && col >= a.Nq) kv_put(kv_at, col, o);
                    else *reinterpret_cast<uint4 *>(a.out + (size_t)row * a.ldo + col) = o;
                };
                const bool any_own = __any_sync(0xffffffffu, own_pass);
                const int c_mid = (out_bn / 2 + 31) & ~31, c0 = part == 0 ? 0 : c_mid, n_cols = (part == 0 ? c_mid : out_bn) - c0;
                if (any_own) {   // rows whose adapter has a B with an Inf or NaN get their delta here; 8 columns at a time
                    tc::OddRow odd;
                    if (own_pass) {
                        const int k = a.row_adapter[row];
                        int e = g.e0;
                        while (e + 1 < g.e1 && a.quads[e].adapter != k) ++e;
                        ld_acquire_d(a.t_ready + e);   // (complete since the tile's K blocks were loaded; orders the reads)
                        odd.t = a.t + ((size_t)(4 * e * kParts + 2 * (g.h0 + h) + (int)crank) * 128 + r) * a.t_cols;
                        odd.parts = kParts; odd.part_stride = kQuadRows * a.t_cols;
                        odd.b = a.b_all + (size_t)k * a.N * kTensorRP;
                        odd.n = a.adapters[k * a.ad_stride];
                    }
#pragma unroll 1
                    for (int c = 0; c < n_cols && g.n0 + c0 + c < a.n_out; c += 8) {
                        const int col = g.n0 + c0 + c;
                        uint32_t v[8], w[8];
                        tc::tmem_ld_32x8(acc_addr + c0 + c, v);
                        if (kMode == kDuoGlu) tc::tmem_ld_32x8(acc_addr + out_bn + c0 + c, w);
                        tc::tmem_ld_wait();
                        if (own_pass) {
                            odd.add8(reinterpret_cast<float(&)[8]>(v), col, kMode != kDuoQkv || col < a.Nq ? 0 : (col < a.Nq + a.Nkv ? 1 : 2));
                            if (kMode == kDuoGlu) odd.add8(reinterpret_cast<float(&)[8]>(w), a.N / 2 + col, 1);
                        }
                        if (kMode == kDuoGlu) {
#pragma unroll
                            for (int e = 0; e < 8; e += 2)
                                tc::silu_mul2(reinterpret_cast<float &>(v[e]), reinterpret_cast<float &>(v[e + 1]), __uint_as_float(w[e]), __uint_as_float(w[e + 1]));
                        }
                        if (row_ok) put_own8(col, reinterpret_cast<float(&)[8]>(v));
                    }
                    drained(h);
                    continue;
                }
                // Chunks of 32 columns: in registers, packed, and only the last ones not yet packed when the half is given
                // free for the next item; the rest runs underneath its MMAs.  (With the stores in between a half was taken
                // up for 4 k cycles, with SwiGLU for 8 k, at 57 k for its MMAs.)
                const bool res = kMode == kDuoLinear && a.residual != nullptr;
                // this lane's row of the chunk at column `col`, rounded
                auto pack32 = [&](int col, float (&f)[32], uint4 (&u)[4]) {
                    const int cu = col + ql * 8;   // the columns of the quad's four rows that this lane reads
                    if (res) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            u[j] = (row & ~3) + j < a.M && cu < a.n_out ? *reinterpret_cast<const uint4 *>(a.residual + (row4 + j) * a.ldo + cu) : make_uint4(0, 0, 0, 0);
                        tc::quad_transpose(u, ql);
#pragma unroll
                        for (int x = 0; x < 4; ++x) add_res8(reinterpret_cast<float(&)[8]>(f[8 * x]), u[x]);
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) u[x] = pack8(reinterpret_cast<const float(&)[8]>(f[8 * x]));
                };
                auto put32 = [&](int k, uint4 (&u)[4]) {   // chunk k: 32 columns, 16, or none
                    const int col = g.n0 + c0 + 32 * k, left = n_cols - 32 * k;
                    if (left <= 0 || col >= a.n_out) return;
                    if (left < 32) {
                        if (row_ok)
#pragma unroll
                            for (int x = 0; x < 2; ++x)
                                if (col + 8 * x < a.n_out) *reinterpret_cast<uint4 *>(a.out + (size_t)row * a.ldo + col + 8 * x) = u[x];
                    } else if (kMode == kDuoQkv && a.kv_pool != nullptr && col >= a.Nq) {
                        tc::quad_transpose(u, ql);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const long long at = __shfl_sync(0xffffffffu, kv_at, (lane & ~3) + j);   // (-1 for rows beyond the end)
                            if (col + ql * 8 < a.n_out) kv_put(at, col + ql * 8, u[j]);
                        }
                    } else {
                        // through shared memory and TMA, which cuts rows and columns off at the matrix's end
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                        __syncwarp();
                        const int b = n_out_bufs++ & 1;
#pragma unroll
                        for (int x = 0; x < 4; ++x)   // 64-byte swizzle
                            *reinterpret_cast<uint4 *>(out_row + b * S::kOutBytes + ((x ^ ((lane >> 1) & 3)) << 4)) = u[x];
                        tc::fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) tma_store_2d(&tmO, out_buf + b * S::kOutBytes, col, row);
                    }
                };
                constexpr int kFirst = kMode == kDuoGlu ? 1 : 2;   // chunks of a step: 64 columns of tensor memory
                uint4 held[kFirst][4];
#pragma unroll
                for (int st = 0; st < 2; ++st) {
                    uint32_t v[64];   // kDuoGlu: gate, up
                    if (32 * kFirst * st < n_cols) {
                        const uint32_t at = acc_addr + c0 + 32 * kFirst * st;
                        tc::tmem_ld_32x32(at, reinterpret_cast<uint32_t(&)[32]>(v[0]));
                        if (kMode == kDuoGlu) tc::tmem_ld_32x32(at + out_bn, reinterpret_cast<uint32_t(&)[32]>(v[32]));
                        else if (32 * kFirst * st + 32 < n_cols) tc::tmem_ld_32x32(at + 32, reinterpret_cast<uint32_t(&)[32]>(v[32]));
                        tc::tmem_ld_wait();
                    }
                    if (st == 1) {
                        drained(h);
                        if (!res)
#pragma unroll
                            for (int k = 0; k < kFirst; ++k) put32(k, held[k]);
                    }
                    if (kMode == kDuoGlu) {
#pragma unroll
                        for (int e = 0; e < 32; e += 2)
                            tc::silu_mul2(reinterpret_cast<float &>(v[e]), reinterpret_cast<float &>(v[e + 1]), __uint_as_float(v[32 + e]), __uint_as_float(v[33 + e]));
                    }
#pragma unroll
                    for (int k = 0; k < kFirst; ++k) {
                        const int c = 32 * (kFirst * st + k);
                        if (c >= n_cols) break;
                        pack32(g.n0 + c0 + c, reinterpret_cast<float(&)[32]>(v[32 * k]), held[k]);
                        if (st == 1 || res) put32(kFirst * st + k, held[k]);
                    }
                }
            }
            if (ok && g.shrink && lane == 0) atomicAdd(a.t_ready + g.e0, 1);   // (behind each lane's fence and the warp's sync)
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    tc::tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) report(a.status, ALORA_ERR_TIMEOUT);
    if (threadIdx.x == 0) tc::item_counter_release(a.item_counters, a.t_ready + e_base, n_entries);
    cluster_sync_d();   // no block leaves while the other may still signal it
    if (warp == 1) {
        tc::tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}
}  // namespace

bool make_tensor_map_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld,
                          uint32_t box_rows);  // gemm_tcgen05.cu
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn tensor_map_encoder();  // gemm_tcgen05.cu

// The column tile of a launch with `entries` shrink items: least rounds over the clusters x (K loop + what an epilogue leaves
// uncovered).  A K block takes the tensor time of 512 rows, or 65536 bytes of A and 192 of each W row through the shared memory at
// 128 a cycle.
static int duo_pick_bn(const alora_ctx *ctx, int T, int K, int n_cols, bool glu, int entries, long long *cycles) {
    const int clusters = std::max(1, ctx->sm_count / 2);
    int best = 0;
    for (int bn = kMaxBn; bn >= 128; bn -= 32) {   // (the instruction takes multiples of 32)
        const int out_bn = glu ? bn / 2 : bn, items = ((T + kQuadRows - 1) / kQuadRows) * ((n_cols + out_bn - 1) / out_bn) + entries;
        const long long kblock = std::max(4 * bn, (65536 + 192 * bn) / 128);
        const int rounds = (items + clusters - 1) / clusters;
        // (shrink items of 512 rows end with the first round's column tiles, which then wait for their t)
        const long long c = rounds * ((K + kBKd - 1) / kBKd * kblock + 24 * bn) + (items + entries > rounds * clusters ? 10000 : 0);
        if (best == 0 || c < *cycles) { best = bn; *cycles = c; }
    }
    return best;
}

template <int kMode, int kParts>
static int launch_duo(alora_ctx *ctx, const CUtensorMap &tmX, const CUtensorMap &tmW, const CUtensorMap &tmT, const CUtensorMap &tmS,
                      const CUtensorMap (&tmB)[3], const DuoArgs &g, int max_entries, cudaStream_t s) {
    // the output in boxes of 32 rows x 32 columns, 64-byte swizzle
    CUtensorMap tmO;
    {
        EncodeTiledFn enc = tensor_map_encoder();
        cuuint64_t dims[2] = {(cuuint64_t)g.n_out, (cuuint64_t)g.M};
        cuuint64_t strides[1] = {(cuuint64_t)g.ldo * 2};
        cuuint32_t box[2] = {32, 32}, es[2] = {1, 1};
        if (!enc || enc(&tmO, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, g.out, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return -1;
    }
    static bool attr_set[64] = {};   // one per instantiation
    const int dev = ctx->cfg.device;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        if (cudaFuncSetAttribute(gemm_duo_tcgen05_kernel<kMode, kParts>, cudaFuncAttributeMaxDynamicSharedMemorySize, DuoSmem::kTotal) != cudaSuccess) return -1;
        attr_set[dev] = true;
    }
    const int out_bn = kMode == kDuoGlu ? g.bn / 2 : g.bn;
    const int items = ((g.M + kQuadRows - 1) / kQuadRows) * ((g.n_out + out_bn - 1) / out_bn) + max_entries;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2 * std::max(1, std::min(ctx->sm_count / 2, items))); cfg.blockDim = dim3(kThreadsD);
    cfg.dynamicSmemBytes = DuoSmem::kTotal; cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    ProfScope prof(ctx, kMode == kDuoQkv ? KK_PROJECT : KK_LINEAR, s);
    return cudaLaunchKernelEx(&cfg, gemm_duo_tcgen05_kernel<kMode, kParts>, tmX, tmW, tmT, tmS, tmB[0], tmB[1], tmB[2], tmO, g) == cudaSuccess ? 1 : -1;
}

bool shrink_apart(const alora_ctx *ctx, int T, int R, int items);   // gemm_tcgen05.cu

// The column tile that the q/k/v projection of a batch takes here, 0: it is better served by the 128-row kernel.  The decision must not
// depend on the mode, so that rows with a closed gate come out bit-identical to the base-only projection of the same batch.
int duo_project_tile(const alora_ctx *ctx, int layer, int T, int R) {
    const Dims &d = ctx->d;
    if (T <= kQuadRows || ctx->sm_count < 2 || d.H % 8 != 0 || d.N % 8 != 0 || d.Nq % 32 != 0 || d.Nkv % 32 != 0) return 0;
    const int G = ctx->sm_count;
    // against the 128 x 256 tiles of gemm_tcgen05.cu, 790 cycles a K block
    const bool have_adapters = ctx->layer_has_adapter[layer] != 0;
    long long here = 0;
    const int bn = duo_pick_bn(ctx, T, d.H, d.N, false, have_adapters ? quad_bound(ctx, T, R) : 0, &here);
    const int items128 = ((T + 127) / 128) * ((d.N + 255) / 256);
    const bool apart = have_adapters && shrink_apart(ctx, T, R, items128);
    const int shrink128 = have_adapters && !apart ? pair_bound(ctx, T, R) : 0;
    const long long other = (long long)((items128 + shrink128 + G - 1) / G) * ((d.H + kBKd - 1) / kBKd) * 790;
    // With three summands of t (few rows) what follows the K loop counts: 15 k cycles for each adapter of a quad here, 8 k for each of
    // a row tile there, 30 k for a shrink kernel of its own.  One layer call, us, there / here: 777 rows and one adapter 101 / 87,
    // 1000 rows and two 80 / 66 (the projection alone), 753 rows of 48 requests and four 69 / 81.
    const int n_m = (T + 127) / 128, n_q = (n_m + 3) / 4;
    const bool few = have_adapters && T <= kSplitTTokens;
    const long long late_here = few ? 15000ll * ((quad_bound(ctx, T, R) + n_q - 1) / n_q) : 0;
    const long long late_other = few ? 8000ll * ((pair_bound(ctx, T, R) + n_m - 1) / n_m) + (apart ? 30000 : 0) : 0;
    return here + late_here > other + late_other ? 0 : bn;
}

// q/k/v projection of a batch.  Returns the kernels launched, 0 when the batch is not for this kernel (nothing launched) or -1 on error.
int launch_project_duo_tc(alora_ctx *ctx, int layer, const void *hidden, int T, int R, void *qkv, cudaStream_t s,
                          void *kv_pool, int num_pages) {
    const Dims &d = ctx->d;
    const int bn = duo_project_tile(ctx, layer, T, R), t_parts = T <= kSplitTTokens ? 3 : 1;
    const bool have_adapters = ctx->layer_has_adapter[layer] != 0;
    if (bn == 0) return 0;
    const void *W = ctx->layers[layer].wqkv;
    CUtensorMap tmX, tmW, tmT, tmS, tmB[3];
    if (!make_tensor_map_bf16(&tmX, hidden, T, d.H, d.H, 128)) return -1;
    if (!make_tensor_map_bf16(&tmW, W, d.N, d.H, d.H, bn / 2)) return -1;
    tmT = tmX; tmS = tmW; tmB[0] = tmB[1] = tmB[2] = tmW;
    DuoArgs g{};
    g.M = T; g.N = g.n_out = d.N; g.K = d.H; g.Nq = d.Nq; g.Nkv = d.Nkv; g.bn = bn;
    g.out = (__nv_bfloat16 *)qkv; g.ldo = d.N; g.t_cols = 3 * kTensorRP;
    if (have_adapters) {
        const size_t na = (size_t)std::max(1, ctx->cfg.max_adapters);
        if (!make_tensor_map_bf16(&tmT, ctx->d_t, (uint64_t)ctx->t_slots * 128, 3 * kTensorRP, 3 * kTensorRP, 128)) return -1;
        if (!make_tensor_map_bf16(&tmS, ctx->tc_a_all[layer], na * 3 * kTensorRP, d.H, d.H, 3 * kTensorRP / 2)) return -1;
        EncodeTiledFn enc = tensor_map_encoder();
        const int rows[3] = {d.Nq, d.Nkv, d.Nkv};
        for (int blk = 0, start = 0; blk < 3; start += rows[blk++]) {   // B of one block: (rank column, row inside the block, adapter)
            cuuint64_t dims[3] = {(cuuint64_t)kTensorRP, (cuuint64_t)rows[blk], (cuuint64_t)na};
            cuuint64_t strides[2] = {(cuuint64_t)kTensorRP * 2, (cuuint64_t)d.N * kTensorRP * 2};
            cuuint32_t box[3] = {(cuuint32_t)kTensorRP, (cuuint32_t)bn / 2, 1};
            cuuint32_t es[3] = {1, 1, 1};
            void *base = (char *)ctx->tc_b_all[layer] + (size_t)start * kTensorRP * 2;
            if (!enc || enc(&tmB[blk], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, es,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return -1;
        }
        const AdapterDev *ads = ctx->d_adapters + (size_t)layer * ctx->cfg.max_adapters;
        g.adapters = &ads->rpad;   // (address arithmetic only: padded rank and scale of an AdapterDev are neighbours)
        g.ad_stride = sizeof(AdapterDev) / 4;
        g.quads = ctx->d_quads; g.quad_off = ctx->d_quad_off; g.t = (__nv_bfloat16 *)ctx->d_t; g.t_ready = ctx->d_quad_ready;
        g.row_adapter = ctx->d_row_adapter; g.any_odd = ctx->d_counts + kOddAdapters;
        g.b_all = (const __nv_bfloat16 *)ctx->tc_b_all[layer];
    }
    g.item_counters = ctx->d_counts + 10;
    if (kv_pool != nullptr) {
        int shift = 0;
        while ((1 << shift) < d.hd) ++shift;
        g.kv_pool = (__nv_bfloat16 *)kv_pool; g.slot_map = ctx->d_slot; g.kv_hd_shift = shift; g.kv_heads = d.Hkv;
        g.kv_page_size = d.page; g.kv_num_pages = num_pages;
    }
    g.status = ctx->d_status;
    const int max_items = have_adapters ? 2 * quad_bound(ctx, T, R) : 0;
    return t_parts == 3 ? launch_duo<kDuoQkv, 3>(ctx, tmX, tmW, tmT, tmS, tmB, g, max_items, s)
                        : launch_duo<kDuoQkv, 1>(ctx, tmX, tmW, tmT, tmS, tmB, g, max_items, s);
}

static int duo_max_entries(const alora_ctx *ctx, int T) {
    return std::min(ctx->max_quads, (T + kQuadRows - 1) / kQuadRows * std::max(1, ctx->cfg.max_adapters));
}
// The column tile that a dense projection of T rows takes here, 0: it is better served by the 128-row kernel.  (The choice of the
// kernel must not depend on the mode; that of the tile may, a row's sums are the same in all of them.)
int duo_linear_tile(const alora_ctx *ctx, int T, int K, int N, bool glu, bool adapted) {
    const int G = ctx->sm_count, n_out = glu ? N / 2 : N;
    // Against rounds over the blocks x 790 cycles of the 128 x 256 tile's K block.  That
    // kernel walks the column tiles of a row tile first, so a W that L2 does not hold is streamed from HBM (3400 bytes a cycle)
    // in every round.
    const int n_n = (N + 255) / 256, items128 = ((T + 127) / 128) * n_n;
    const long long rounds128 = (items128 + G - 1) / G;
    const long long w_cycles = (long long)N * K * 2 > (64ll << 20) ? (n_n >= G ? (T + 127) / 128 : rounds128) * N * (2 * kBKd) / 3400 : 0;
    const long long other = std::max(rounds128 * 790, w_cycles) * ((K + kBKd - 1) / kBKd);
    if (T <= 256 || G < 2 || K % 8 != 0 || N % 8 != 0 || (glu && N % 16 != 0)) return 0;
    long long here = 0;
    const int bn = duo_pick_bn(ctx, T, K, n_out, glu, 0, &here);
    if (here > other) return 0;
    return adapted ? duo_pick_bn(ctx, T, K, n_out, glu, duo_max_entries(ctx, T), &here) : bn;
}

// Plain dense projection y = x W^T (+ residual), or with `glu` y = silu(x Wg^T) * (x Wu^T) for W = [Wg; Wu]; optionally with a gated
// low-rank delta.  Returns 1 (launched), 0 (not for this kernel: nothing launched) or -1 (error).
int launch_linear_duo_tc(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y,
                         const void *residual, const LinearDelta *delta, bool glu, cudaStream_t s) {
    const int n_out = glu ? N / 2 : N;
    if (delta != nullptr && (delta->n_blk != (glu ? 2 : 1) || delta->tile0 % 4 != 0)) return 0;
    if (glu && residual != nullptr) return 0;
    const int bn = duo_linear_tile(ctx, T, K, N, glu, delta != nullptr), max_entries = delta == nullptr ? 0 : duo_max_entries(ctx, T);
    if (bn == 0) return 0;
    CUtensorMap tmX, tmW, tmT, tmA, tmB[3];
    if (!make_tensor_map_bf16(&tmX, x, T, K, K, 128)) return -1;
    if (!make_tensor_map_bf16(&tmW, W, N, K, K, bn / 2)) return -1;
    tmT = tmX; tmA = tmW; tmB[0] = tmB[1] = tmB[2] = tmW;
    DuoArgs g{};
    g.M = T; g.N = N; g.K = K; g.Nq = N; g.Nkv = 0; g.bn = bn; g.n_out = n_out; g.t_cols = kTensorRP;
    g.out = (__nv_bfloat16 *)y; g.residual = (const __nv_bfloat16 *)residual; g.ldo = n_out;
    g.item_counters = ctx->d_counts + 10; g.status = ctx->d_status;
    if (delta != nullptr) {
        const uint64_t na = (uint64_t)std::max(1, ctx->cfg.max_adapters);
        g.t_cols = delta->n_blk * kTensorRP; g.b_rows = (int)(na * N);
        if (!make_tensor_map_bf16(&tmT, delta->t, (uint64_t)ctx->max_quads * kQuadRows, g.t_cols, g.t_cols, 128)) return -1;
        if (!make_tensor_map_bf16(&tmA, delta->A, na * g.t_cols, K, K, g.t_cols / 2)) return -1;
        if (!make_tensor_map_bf16(&tmB[0], delta->B, na * N, kTensorRP, kTensorRP, bn / 2)) return -1;
        g.quads = ctx->d_quads; g.quad_off = ctx->d_quad_off; g.quad0 = delta->tile0 / 4;
        g.adapters = &delta->table->rpad; g.ad_stride = sizeof(MlpAdapterDev) / 4;
        g.row_adapter = delta->row_adapter; g.t_ready = ctx->d_quad_ready; g.t = (__nv_bfloat16 *)delta->t;
        g.any_odd = ctx->d_counts + kOddAdapters; g.b_all = (const __nv_bfloat16 *)delta->B;
    }
    return glu ? launch_duo<kDuoGlu, 1>(ctx, tmX, tmW, tmT, tmA, tmB, g, 2 * max_entries, s)
               : launch_duo<kDuoLinear, 1>(ctx, tmX, tmW, tmT, tmA, tmB, g, 2 * max_entries, s);
}

}  // namespace alora
