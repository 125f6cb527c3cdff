// Projection of a batch of few rows (decode steps, short invocation suffixes; up to kFewTiles row tiles of 128) in one
// launch: out = x W^T with the aLoRA delta of Eq. 5 on the rows whose gate is open.
//
// Bound by streaming W out of HBM once, and, at 12 .. 25 us a launch, by everything that does not overlap that stream.
// A thread-block cluster owns a tile of W's columns (and 128 rows of x); its blocks take a slice of K each, as many slices
// as give every SM a block, stream their part of W and x through a TMA ring and accumulate in tensor memory
// (tcgen05.mma 128 x tile x 16).  The partial products then go to each block's shared memory, and after a cluster barrier
// every block adds up its share of the tile's columns over the cluster's shared memory, in slice order, and finishes them:
// delta, residual or SwiGLU, bf16, k / v columns to the cache slots.
// Measured against the two kernels it replaces (the second one read the partials back from L2), hidden 4096: q/k/v of 128
// rows with one adapter 38 -> 26 us, of 64 rows with four 34 -> 24; o_proj of 40 rows 13.7 -> 11.7, gate/up 46 -> 41 (35 us of
// HBM time), down 27.7 -> 24 (18); against 48 tiles of 128 x 256 on the dense route, 194 rows: 52 -> 42 with the metadata.
// What is left of q/k/v's 24: 7 wait for the batch's facts (W is on its way by then), 11 stream (each cluster reads the A rows
// of all adapters present: 208 KB a block on top of 520), 3 to shared memory and barrier, 3 sums, 3 delta and stores.
//
// The rank-r shrink rides along in every cluster: the A rows of the adapters present in the row tile (those of the q / k / v
// block that the column tile lies in, padded to 16) are extra columns of the B operand, so t = A x of the whole tile is
// in the cluster's tensor memory at the end; of each row only its own adapter's part is kept.  x is read once, or, in a layer
// call whose x does not wait for anything, a second time from L2 for A x, so that W x starts 7 us before the batch's facts
// are there (8 x 16 rows 83.2 -> 79.5 us a call, a base prefill of 235 rows 47.6 -> 45.2).  t is fp32 throughout.  Rows without an applied adapter add nothing, so they go through exactly the arithmetic of a base-only call
// (Prop. 1: gated-off rows are bit-identical).  No atomics, fixed summation orders: run-to-run deterministic.
//
// The W tiles of the first ring round are requested before the wait on the preceding kernel (they depend on nothing it
// writes).  All waits are bounded; on expiry ALORA_ERR_TIMEOUT is recorded and the blocks leave through the barriers.
#include <algorithm>

#include "alora_internal.h"
#include "tc_common.cuh"

namespace alora {

namespace {
constexpr int kFcBNMax = 256, kFcBK = 64, kFcThreads = 320, kFcWarps = kFcThreads / 32;   // producer, issuer, 8 epilogue warps
constexpr int kFcMaxStages = 8, kFcMaxChunks = 16, kFcMaxCluster = 8;
constexpr int kFcChunkBytes = 16 * kFcBK * 2;
constexpr int kFcRank = kRankPadMax;      // row pitch of the B slab, and A rows per adapter and block

struct FewArgs {
    int T, N, K, bn, ksplit, n_rt;      // bn: columns of a tile of W; n_rt: row tiles of 128
    int rows_shift;               // log2 of the rows of the x box and of the partial arrays: 16, 32, 64 or 128
    int x_early;                  // x was complete before the kernel before this one began: only its adapter facts are waited for
    int stage_bytes, n_stages, t_off, b_off, bar_off;   // shared-memory layout, see few_plan()
    const FewRowMeta *meta;       // [row tile] adapter facts, nullptr: no adapters in this launch
    const __nv_bfloat16 *b_all;   // the layer's B rows of all adapters, [adapter][N][64]
    int Nq, Nkv;
    const __nv_bfloat16 *residual;
    __nv_bfloat16 *out;
    int ldo;
    int glu;                      // W = [gate; up]: a tile holds bn / 2 rows of each, out = silu(gate) * up
    __nv_bfloat16 *kv_pool;
    const int32_t *slot_map;
    int kv_hd_shift, kv_heads, kv_page_size, kv_num_pages;
    int32_t *status;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void st_cluster4(uint32_t addr, const float4 &v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

// kSecondPass: the A rows take a second pass over x (FewArgs::x_early with adapters)
template <bool kSecondPass>
__global__ void __launch_bounds__(kFcThreads, 1)
gemm_few_cluster_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                        const __grid_constant__ RankMaps tmA, const FewArgs a) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ int kv_slot_s[kFewRowMax], slot_s[kFewRowMax], id_s[kFewRowMax], rpad_s[kFewRowMax], first_chunk[kFewRowMax], b_start[kFewRowMax];
    __shared__ float scale_s[kFewRowMax];
    __shared__ int n_present_s, n_chunk_s, max_rank_s;
    const uint32_t smem_base = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem_al = smem_raw + (smem_base - tc::smem_u32(smem_raw));
    const uint32_t bar0 = smem_base + (uint32_t)a.bar_off;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_al + a.bar_off);
    // barrier words: full[8], empty[8], acc_full, drain, facts; then the tensor-memory address and the abort flag
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kFcMaxStages + s); };
    const uint32_t accf_bar = bar0 + 8u * (2 * kFcMaxStages), drain_bar = accf_bar + 8u, facts_bar = accf_bar + 16u;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(bars + 2 * kFcMaxStages + 3);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bars + 2 * kFcMaxStages + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_stages = a.n_stages, rs = 1 << a.rows_shift;
    const uint32_t x_bytes = (uint32_t)rs * kFcBK * 2, w_bytes = (uint32_t)a.bn * kFcBK * 2;
    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) { tc::mbar_init(full_bar(s), 1); tc::mbar_init(empty_bar(s), 1); }
        tc::mbar_init(accf_bar, 1); tc::mbar_init(drain_bar, 1); tc::mbar_init(facts_bar, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
        tc::fence_proxy_async();
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32((const void *)tmem_slot), 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // this block's tile and K range (the blocks of a cluster are consecutive, and the row tiles of a column tile)
    const int sl = (int)blockIdx.x % a.ksplit, tile = (int)blockIdx.x / a.ksplit / a.n_rt, rt = (int)blockIdx.x / a.ksplit % a.n_rt;
    const int row0 = rt * kFewRowMax, T = min(kFewRowMax, a.T - row0);   // its rows
    const int kb_total = (a.K + kFcBK - 1) / kFcBK, kb_base = kb_total / a.ksplit, kb_rem = kb_total % a.ksplit;
    const int kb0 = sl * kb_base + min(sl, kb_rem), nkb = kb_base + (sl < kb_rem ? 1 : 0);
    tc::grid_dep_launch();
    const int w_ahead = min(nkb, n_stages);
    auto load_w = [&](uint32_t dst, uint32_t bar, int k) {
        if (!a.glu) {
            tc::tma_load_2d(dst, &tmW, bar, k, tile * a.bn);
        } else {
            tc::tma_load_2d(dst, &tmW, bar, k, tile * (a.bn / 2));
            tc::tma_load_2d(dst + w_bytes / 2, &tmW, bar, k, a.N / 2 + tile * (a.bn / 2));
        }
    };
    if (threadIdx.x == 0) {
        tc::tma_prefetch_desc(&tmW);
        for (int s = 0; s < w_ahead; ++s) {
            tc::mbar_expect_tx(full_bar(s), w_bytes);
            load_w(smem_base + s * a.stage_bytes + x_bytes, full_bar(s), (kb0 + s) * kFcBK);
        }
    }
    // x and the adapter facts are written by earlier kernels of the stream.  Where only the facts come from the kernel before,
    // W x does not wait for them, and the A rows take a second pass over x (from L2) once the facts are there.
    constexpr bool second_pass = kSecondPass;
    if (!kSecondPass && !a.x_early) tc::grid_dep_wait();
    const int out_bn = a.glu ? a.bn / 2 : a.bn, n_out = a.glu ? a.N / 2 : a.N, col0 = tile * out_bn;
    const int v0 = sl * (out_bn / 8) / a.ksplit, v1 = (sl + 1) * (out_bn / 8) / a.ksplit;   // this block's share: 8-column vectors
    const int share = (v1 - v0) * 8;
    const int blk = col0 < a.Nq ? 0 : (col0 < a.Nq + a.Nkv ? 1 : 2);
    // over the ring, once the accumulators are complete, column-major with the rows contiguous:
    float *part = reinterpret_cast<float *>(smem_al);                // [bn][rs] partial products, then this share's sums
    float *t_s = reinterpret_cast<float *>(smem_al + a.t_off);       // [ranks][rs] partial t of each row's own adapter, then t
    uint8_t *b_s = smem_al + a.b_off;                                // per adapter present: [share][rpad] bf16

    if (warp == 0) {
        if (lane == 0) {
            // ------------------------------ TMA producer ------------------------------
            tc::tma_prefetch_desc(&tmX);
            bool ok = true;
            int kc = 0, n_chunk = 0, n_present = 0;
            auto facts = [&]() {
                if (!tc::mbar_wait(facts_bar, 0, abort_flag)) return false;
                n_chunk = n_chunk_s; n_present = n_present_s;
                return true;
            };
            auto a_rows = [&](uint32_t dst, int s, int k) {
                for (int p = 0; p < n_present; ++p)
                    tc::tma_load_2d(dst + first_chunk[p] * kFcChunkBytes, &tmA.box[rpad_s[p] / 16 - 1], full_bar(s), k, id_s[p] * 3 * kFcRank + blk * kFcRank);
            };
            if (a.meta != nullptr && !second_pass) ok = facts();
            for (; ok && kc < nkb; ++kc) {
                const int s = kc % n_stages, k = (kb0 + kc) * kFcBK;
                if (!tc::mbar_wait(empty_bar(s), ((kc / n_stages) & 1) ^ 1, abort_flag)) { ok = false; break; }
                const uint32_t sx = smem_base + s * a.stage_bytes, sw = sx + x_bytes;
                if (kc < w_ahead) {   // this stage's W tile is already on its way
                    tc::mbar_arrive_expect_tx(full_bar(s), x_bytes + n_chunk * kFcChunkBytes);
                } else {
                    tc::mbar_arrive_expect_tx(full_bar(s), x_bytes + w_bytes + n_chunk * kFcChunkBytes);
                    load_w(sw, full_bar(s), k);
                }
                tc::tma_load_2d(sx, &tmX, full_bar(s), k, row0);
                a_rows(sw + w_bytes, s, k);
            }
            if (ok && second_pass) ok = facts();
            if (second_pass && n_chunk > 0) {
                for (; ok && kc < 2 * nkb; ++kc) {
                    const int s = kc % n_stages, k = (kb0 + kc - nkb) * kFcBK;
                    if (!tc::mbar_wait(empty_bar(s), ((kc / n_stages) & 1) ^ 1, abort_flag)) { ok = false; break; }
                    const uint32_t sx = smem_base + s * a.stage_bytes;
                    tc::mbar_arrive_expect_tx(full_bar(s), x_bytes + n_chunk * kFcChunkBytes);
                    tc::tma_load_2d(sx, &tmX, full_bar(s), k, row0);
                    a_rows(sx + x_bytes, s, k);
                }
            }
            if (!ok) {
                // copies already in flight must land before the shared memory is reused or released
                for (int i = max(0, kc - n_stages); i < max(kc, w_ahead); ++i) {
                    const long long t0 = clock64();
                    while (!tc::mbar_try_wait(full_bar(i % n_stages), (i / n_stages) & 1) && clock64() - t0 < 20000000LL) {}
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        // the whole warp walks the schedule (uniform control flow), one elected lane issues
        const bool leader = tc::elect_one();
        auto wait_all = [&](uint32_t bar, uint32_t parity) {
            return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, abort_flag));
        };
        // the A chunks are consecutive rows of one B operand (one instruction per k for all of them: 16-column
        // instructions took 0.6 us a stage for 8 chunks)
        const uint32_t idesc_main = tc::idesc_bf16_f32(128, a.bn);
        uint32_t idesc_chunk = 0;
        bool ok = true;
        int n_chunk = 0;
        auto facts = [&]() {
            if (!wait_all(facts_bar, 0)) return false;
            n_chunk = n_chunk_s;
            idesc_chunk = tc::idesc_bf16_f32(128, 16 * max(n_chunk, 1));
            return true;
        };
        if (a.meta != nullptr && !second_pass) ok = facts();
        int kc = 0;
        for (; ok && kc < nkb; ++kc) {
            const int s = kc % n_stages;
            if (!wait_all(full_bar(s), (kc / n_stages) & 1)) { ok = false; break; }
            tc::tc_fence_after();
            const uint32_t sx = smem_base + s * a.stage_bytes, sw = sx + x_bytes, sc = sw + w_bytes;
            const uint64_t dx = tc::smem_desc_k_sw128(sx), dw = tc::smem_desc_k_sw128(sw), dc = tc::smem_desc_k_sw128(sc);
            if (leader) {
#pragma unroll
                for (int k = 0; k < kFcBK / 16; ++k) tc::mma_bf16(tmem_base, dx + 2 * k, dw + 2 * k, idesc_main, (kc | k) != 0 ? 1u : 0u);
                if (n_chunk > 0) {
#pragma unroll
                    for (int k = 0; k < kFcBK / 16; ++k)
                        tc::mma_bf16(tmem_base + kFcBNMax, dx + 2 * k, dc + 2 * k, idesc_chunk, (kc | k) != 0 ? 1u : 0u);
                }
                tc::mma_commit(empty_bar(s));
            }
        }
        if (ok && second_pass) ok = facts();
        if (second_pass && n_chunk > 0) {
            for (; ok && kc < 2 * nkb; ++kc) {
                const int s = kc % n_stages;
                if (!wait_all(full_bar(s), (kc / n_stages) & 1)) { ok = false; break; }
                tc::tc_fence_after();
                const uint32_t sx = smem_base + s * a.stage_bytes;
                const uint64_t dx = tc::smem_desc_k_sw128(sx), dc = tc::smem_desc_k_sw128(sx + x_bytes);
                if (leader) {
#pragma unroll
                    for (int k = 0; k < kFcBK / 16; ++k)
                        tc::mma_bf16(tmem_base + kFcBNMax, dx + 2 * k, dc + 2 * k, idesc_chunk, ((kc - nkb) | k) != 0 ? 1u : 0u);
                    tc::mma_commit(empty_bar(s));
                }
            }
        }
        if (leader) {
            tc::mma_commit(ok ? accf_bar : drain_bar);
            if (!ok) {
                const long long t0 = clock64();
                while (!tc::mbar_try_wait(drain_bar, 0) && clock64() - t0 < 20000000LL) {}
            }
        }
        __syncwarp();
    } else {
        // ------------------------------ epilogue warps: tensor memory -> shared memory ------------------------------
        // (a thread owns a row; arrays are column-major so that a warp's 32 rows are 32 consecutive words.  All MMAs have
        // completed by then, so the ring that the arrays lie over is no longer read.)
        tc::grid_dep_wait();
        {
            const int e = threadIdx.x - 64;
            if (a.kv_pool != nullptr && e < T) kv_slot_s[e] = a.slot_map[row0 + e];
            if (a.meta != nullptr) {
                const FewRowMeta *meta = a.meta + rt;
                if (warp == 2) {
                    // a lane per adapter present (at most kFcMaxChunks: few_plan()): where its A rows lie in a ring stage, in
                    // chunks of 16, and its B rows; the producer and the issuer wait for just this
                    const int n = meta->n_present, id = meta->id[lane], rp = lane < n ? meta->rpad[lane] : 0;
                    int sum = rp / 16, mx = rp;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, sum, off);
                        if (lane >= off) sum += v;
                        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                    }
                    const int first = sum - rp / 16;
                    id_s[lane] = id; rpad_s[lane] = rp; first_chunk[lane] = first;
                    b_start[lane] = first * share * 32 + 16 * lane;   // 16 bytes between the adapters: rows of different ones in different banks
                    if (lane == 31) { n_present_s = n; n_chunk_s = sum; max_rank_s = mx; }
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(facts_bar);
                }
                const int r = e - (kFcThreads - 64 - kFewRowMax);   // (the last 128 threads)
                if (r >= 0) { slot_s[r] = meta->slot_of_row[r]; scale_s[r] = meta->scale[r]; }
            } else if (e == 0) {
                n_present_s = 0; n_chunk_s = 0; max_rank_s = 0;
            }
            epilogue_sync();
        }
        const int n_present = n_present_s, n_chunk = n_chunk_s;
        const int q = warp & 3, half = (warp - 2) >> 2;   // tensor-memory lane quarter; half of the columns
        const int r = q * 32 + lane;
        const bool have = __all_sync(0xffffffffu, tc::mbar_wait(accf_bar, 0, abort_flag));
        // the B rows of this block's columns, for every adapter present (needed only after the sums: their fetch is hidden)
        for (int p = 0; have && p < n_present; ++p) {
            const int vecs = rpad_s[p] / 8;   // 16-byte vectors of a column's B row
            const __nv_bfloat16 *src = a.b_all + ((size_t)id_s[p] * a.N + col0 + v0 * 8) * kFcRank;
            for (int i = threadIdx.x - 64; i < share * vecs; i += kFcThreads - 64)
                cp_async16(tc::smem_u32(b_s + b_start[p]) + 16u * i, src + (size_t)(i / vecs) * kFcRank + (i % vecs) * 8);
        }
        if (have && q * 32 < T) {
            tc::tc_fence_after();
            const uint32_t lane_off = (uint32_t)(q * 32) << 16;
            // (rank columns first: two 16-column loads in flight hide some of their latency)
            const int mine = n_present > 0 && r < T ? slot_s[r] : -1;
            for (int p = half; p < n_present; p += 2) {
                const int first = first_chunk[p] * 16, n = min(rpad_s[p], n_chunk * 16 - first);
                for (int c = 0; c < n; c += 32) {
                    uint32_t v[2][16];
                    tmem_ld_32x16(tmem_base + kFcBNMax + first + c + lane_off, v[0]);
                    if (c + 16 < n) tmem_ld_32x16(tmem_base + kFcBNMax + first + c + 16 + lane_off, v[1]);
                    tc::tmem_ld_wait();
                    if (mine == p) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) t_s[(c + e << a.rows_shift) + r] = __uint_as_float(v[0][e]);
                        if (c + 16 < n) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) t_s[(c + 16 + e << a.rows_shift) + r] = __uint_as_float(v[1][e]);
                        }
                    }
                }
            }
#pragma unroll 1
            for (int c = half * 16; c < a.bn; c += 64) {
                uint32_t v[2][16];
                tmem_ld_32x16(tmem_base + c + lane_off, v[0]);
                if (c + 32 < a.bn) tmem_ld_32x16(tmem_base + c + 32 + lane_off, v[1]);
                tc::tmem_ld_wait();
                if (r < rs) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) part[(c + e << a.rows_shift) + r] = __uint_as_float(v[0][e]);
                    if (c + 32 < a.bn) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) part[(c + 32 + e << a.rows_shift) + r] = __uint_as_float(v[1][e]);
                    }
                }
            }
        }
        tc::tc_fence_before();
    }
    if (warp < 2) tc::grid_dep_wait();   // (they write results from here on too)
    __syncwarp();
    cluster_arrive();
    cluster_wait();   // every slice's partial results are in its block's shared memory

    // ------------------------------ all warps: this block's share of the tile's columns ------------------------------
    const int n_present = n_present_s;
    // 1. the slices' partials, added in slice order, in vectors of four rows.  A block reads another's shared memory at
    //    about 17 bytes a cycle and waits half a microsecond for a load, so each thread keeps those of two vectors in
    //    flight, and t, which every block needs whole, is added up once, in shares, and written to all of them.
    const int rv_shift = a.rows_shift - 2, rvs = 1 << rv_shift, n_rv = (T + 3) / 4;
    auto add_slices = [&](uint32_t base, int first, int last, auto &&put) {   // vectors [first, last) of the array at `base`
        for (int i0 = first + threadIdx.x; i0 < last; i0 += 2 * kFcThreads) {
            float4 p[2][kFcMaxCluster];
            bool on[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = i0 + h * kFcThreads;
                on[h] = i < last && (i & (rvs - 1)) < n_rv;
#pragma unroll
                for (int s = 0; s < kFcMaxCluster; ++s)
                    if (on[h] && s < a.ksplit) p[h][s] = ld_cluster4(map_rank(base + 16u * i, (uint32_t)s));
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!on[h]) continue;
                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int s = 0; s < kFcMaxCluster; ++s)
                    if (s < a.ksplit) { f.x += p[h][s].x; f.y += p[h][s].y; f.z += p[h][s].z; f.w += p[h][s].w; }
                put(i0 + h * kFcThreads, f);
            }
        }
    };
    if (n_present > 0) {
        // (in place in every block: only the block that adds a vector up reads it)
        const uint32_t t_addr = tc::smem_u32(t_s);
        const int c0 = sl * max_rank_s / a.ksplit, c1 = (sl + 1) * max_rank_s / a.ksplit;
        add_slices(t_addr, c0 << rv_shift, c1 << rv_shift, [&](int i, const float4 &f) {
            // (rows and rank columns without an adapter hold anything here; nothing reads them)
            const int r = (i & (rvs - 1)) * 4;
            float sc[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) sc[e] = r + e < T && slot_s[r + e] >= 0 ? scale_s[slot_s[r + e]] : 0.f;
            const float4 t = make_float4(f.x * sc[0], f.y * sc[1], f.z * sc[2], f.w * sc[3]);
            for (int s = 0; s < a.ksplit; ++s) st_cluster4(map_rank(t_addr + 16u * i, (uint32_t)s), t);
        });
    }
    __syncwarp();
    cluster_arrive();
    if (a.ksplit > 1)   // in place: only this block reads its own share of its own partials
        for (int c = 0; c < a.bn; c += out_bn)
            add_slices(tc::smem_u32(part), c + v0 * 8 << rv_shift, c + v1 * 8 << rv_shift,
                       [&](int i, const float4 &f) { *reinterpret_cast<float4 *>(part + 4 * i) = f; });
    cp_async_wait_all();
    __syncwarp();
    cluster_wait();     // t is complete
    __syncthreads();
    cluster_arrive();   // this block reads no other's shared memory any more
    // 2. delta, residual, bf16, stores: a thread takes 8 columns of a row, the lanes of a warp consecutive rows.  (The delta
    //    by 16 x 8 x 16 matrix instructions, an adapter at a time, took as long for one adapter and twice as long for four.)
    for (int u = threadIdx.x; u < (v1 - v0) << a.rows_shift; u += kFcThreads) {
        const int row = u & (rs - 1), v = v0 + (u >> a.rows_shift), col = col0 + v * 8;
        if (col >= n_out || row >= T) continue;
        float f[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = part[((v * 8 + e) << a.rows_shift) + row];
        if (a.glu) {
#pragma unroll
            for (int e = 0; e < 8; e += 2)
                tc::silu_mul2(f[e], f[e + 1], part[((out_bn + v * 8 + e) << a.rows_shift) + row], part[((out_bn + v * 8 + e + 1) << a.rows_shift) + row]);
        }
        const int slot = n_present > 0 ? slot_s[row] : -1;
        if (slot >= 0) {   // only rows with an applied adapter add anything (a gated-off row never sees "+ 0")
            const int vecs = rpad_s[slot] / 8;
            const uint4 *b = reinterpret_cast<const uint4 *>(b_s + b_start[slot]) + (v - v0) * 8 * vecs;
            float d[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) d[e] = 0.f;
#pragma unroll 1
            for (int x = 0; x < vecs; ++x) {   // 8 rank columns per step, the 8 outputs as independent chains
                float t[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) t[i] = t_s[((x * 8 + i) << a.rows_shift) + row];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint4 bv = b[e * vecs + x];
                    const uint32_t w[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        d[e] = fmaf(__uint_as_float(w[i] << 16), t[2 * i], d[e]);
                        d[e] = fmaf(__uint_as_float(w[i] & 0xffff0000u), t[2 * i + 1], d[e]);
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] += d[e];
        }
        if (a.residual) {
            const uint4 rv4 = *reinterpret_cast<const uint4 *>(a.residual + (size_t)(row0 + row) * a.ldo + col);
            const uint32_t rw[4] = {rv4.x, rv4.y, rv4.z, rv4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) { f[2 * e] += __uint_as_float(rw[e] << 16); f[2 * e + 1] += __uint_as_float(rw[e] & 0xffff0000u); }
        }
        const uint4 o = make_uint4(tc::pack_bf16(f[0], f[1]), tc::pack_bf16(f[2], f[3]), tc::pack_bf16(f[4], f[5]), tc::pack_bf16(f[6], f[7]));
        *reinterpret_cast<uint4 *>(a.out + (size_t)(row0 + row) * a.ldo + col) = o;
        const int kc = col - a.Nq;   // column inside [k | v]
        if (a.kv_pool != nullptr && kc >= 0) {
            const int slot_kv = kv_slot_s[row];
            if (slot_kv >= 0) {
                const int page = slot_kv / a.kv_page_size, prow = slot_kv % a.kv_page_size;
                if (page >= a.kv_num_pages) { report(a.status, ALORA_ERR_PAGE_RANGE); continue; }
                const int plane = kc >= a.Nkv ? 1 : 0, c2 = kc - plane * a.Nkv;
                const int head = c2 >> a.kv_hd_shift, dd = c2 & ((1 << a.kv_hd_shift) - 1);
                __nv_bfloat16 *dst = a.kv_pool +
                    ((((size_t)page * 2 + plane) * a.kv_heads + head) * a.kv_page_size + prow << a.kv_hd_shift) + dd;
                *reinterpret_cast<uint4 *>(dst) = o;
            }
        }
    }
    __syncwarp();
    cluster_wait();   // no block may release its shared memory while another still reads it
    if (threadIdx.x == 0 && *abort_flag) report(a.status, ALORA_ERR_TIMEOUT);
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem_base, 512);
    }
}

// 227 KB less the kernel's static part
constexpr int kFcDynMax = 227 * 1024 - 4096;

cudaError_t launch_cluster(dim3 grid, int cluster, size_t smem, cudaStream_t s, const CUtensorMap &x, const CUtensorMap &w,
                           const RankMaps &am, const FewArgs &a) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3(kFcThreads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    return a.x_early && a.meta != nullptr ? cudaLaunchKernelEx(&cfg, gemm_few_cluster_kernel<true>, x, w, am, a)
                                          : cudaLaunchKernelEx(&cfg, gemm_few_cluster_kernel<false>, x, w, am, a);
}
}  // namespace

bool make_tensor_map_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t ld,
                          uint32_t box_rows);   // gemm_tcgen05.cu

// How a projection of T rows is cut and laid out in shared memory; false: it does not take this kernel.  By the shapes
// and by what the context may register, never by the mode (`lora`: the layer has adapters).  The cut depends on N, K and
// T alone, so that rows without a delta come out the same with and without adapters on the layer.
// Tile width and slices: the least streamed per block, (W rows + half the x rows, which come from L2) x K blocks, over the
// widths whose clusters all fit on the device at once.  (hidden 4096 -> 4096, 40 rows: 22 tiles of 192 x 6 slices, 132
// blocks; of 256 columns only 16 x 6 fit.)
static bool few_plan(const alora_ctx *ctx, int T, int R, int N, int K, bool lora, int Nq, int Nkv, bool x_early, FewArgs &a) {
    if (T < 1 || T > kFewRowMax * ctx->few_tiles || N % 8 != 0 || K % 8 != 0 || ctx->few_clusters[1] < 1) return false;
    const int kb_total = (K + kFcBK - 1) / kFcBK;
    a.T = T; a.N = N; a.K = K; a.n_rt = (T + kFewRowMax - 1) / kFewRowMax;
    a.rows_shift = T <= 16 ? 4 : T <= 32 ? 5 : T <= 64 ? 6 : 7;
    const int rs = 1 << a.rows_shift;
    long best = 0;
    a.bn = 0;
    for (int bn = kFcBNMax; bn >= 128; bn -= 16) {
        if (Nkv > 0 && bn < kFcBNMax && (Nq % bn != 0 || Nkv % bn != 0)) continue;   // a tile lies in one of q, k, v
        const int n_tiles = (N + bn - 1) / bn * a.n_rt;
        int ks = std::max(1, std::min(std::min(kFcMaxCluster, kb_total), ctx->sm_count / n_tiles));
        // all clusters at once; with two places to spare where blocks do not pair up, since what still runs of the kernel
        // before breaks up the free SMs (26 clusters of 5 where 26 fit: the last one ran alone, 42 us instead of 25)
        while (ks > 1 && ctx->few_clusters[ks] - (ks % 2 ? 2 : 0) < n_tiles) --ks;
        const long cost = (long)((n_tiles * ks + ctx->sm_count - 1) / ctx->sm_count) * (bn + rs / 2) * ((kb_total + ks - 1) / ks);
        if (a.bn == 0 || cost < best) { best = cost; a.bn = bn; a.ksplit = ks; }
    }
    // several row tiles only where that still splits K: one block per 128 x 256 tile takes 24 us at K = 4096 when there are 48
    // of them and 31 when there are 144 (base prefill of 192 rows: a call 57.5 us on the row tiles, 47.5 here), and with all SMs
    // busy the row tiles' kernel is as fast
    if (a.n_rt > 1 && a.ksplit < 2) return false;
    const int p_cap = lora ? std::min(std::min(ctx->cfg.max_adapters, T), R) : 0, rank = (ctx->cfg.max_rank + 15) / 16 * 16;
    // ... and, with adapters, where the delta is small: a block's share of the columns x rank multiply-adds a row on the CUDA
    // cores, while more row tiles fill the other route's SMs.  Layer calls here / on the row tiles, us, by columns x rank x
    // row tiles: 51 x 64 x 2 44 .. 47 / 49 .. 53; 64 x 32 x 3 48 / 51; 128 x 32 x 2 (hidden 4096) 65.4 / 66.0; 128 x 16 x 4 51.4 / 51.4;
    // 128 x 16 x 5 52 / 51; 64 x 64 x 3 54.2 / 53.3; 128 x 32 x 3 71 / 69; 128 x 64 x 2 74 .. 78 / 66 .. 70; 128 x 64 x 4 66 / 53.
    if (a.n_rt > 1 && lora && a.bn / a.ksplit * rank * a.n_rt > 8192) return false;
    const int chunk_cap = p_cap * (rank / 16);
    if (lora && (Nq % a.bn != 0 || Nkv % a.bn != 0 || ctx->cfg.max_adapters > 1024 || chunk_cap > kFcMaxChunks)) return false;
    // shared memory: the ring, over it later the partial products, t and B; then the barriers
    const int col_bytes = rs * 4, part_bytes = a.bn * col_bytes, t_bytes = lora ? rank * col_bytes : 0;
    const int b_bytes = lora ? (a.bn / 8 + a.ksplit - 1) / a.ksplit * 8 * chunk_cap * 32 + 16 * p_cap : 0;
    // (a second pass over x brings the A rows where W was)
    const int w_bytes = a.bn * kFcBK * 2, a_bytes = chunk_cap * kFcChunkBytes, nkb = (kb_total + a.ksplit - 1) / a.ksplit;
    // (what the second pass costs against the wait it saves, by the bytes of x in a slice: up to 208 KB 0 .. 3 % of the call
    // saved, 1 .. 128 rows, 13 K blocks; 256 KB, 384 rows of a narrow layer 3 .. 5 % lost; 512 KB, 140 .. 384 rows 3 .. 4 % lost)
    a.x_early = x_early && (!lora || (long)rs * kFcBK * 2 * nkb <= 224 * 1024) ? 1 : 0;
    const bool second_pass = a.x_early && lora;
    a.stage_bytes = rs * kFcBK * 2 + (second_pass ? std::max(w_bytes, a_bytes) : w_bytes + a_bytes);
    const int room = kFcDynMax - 1024 - 256;
    a.n_stages = std::min(std::min(kFcMaxStages, second_pass ? 2 * nkb : nkb), room / a.stage_bytes);
    a.t_off = part_bytes; a.b_off = part_bytes + t_bytes;
    a.bar_off = (std::max(a.n_stages * a.stage_bytes, a.b_off + b_bytes) + 15) / 16 * 16;
    return a.n_stages >= 1 && a.bar_off <= room;
}

// What few_plan() asks the device once, at the creation of a context: the clusters of each size that fit at once.
void few_cluster_init(alora_ctx *ctx) {
    for (auto kernel : {gemm_few_cluster_kernel<false>, gemm_few_cluster_kernel<true>}) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFcDynMax) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    }
    for (int c = 1; c <= kFcMaxCluster; ++c) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(c); cfg.blockDim = dim3(kFcThreads); cfg.dynamicSmemBytes = kFcDynMax;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)c; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&ctx->few_clusters[c], gemm_few_cluster_kernel<true>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            ctx->few_clusters[c] = 0;
        }
    }
}

bool few_cluster_route(const alora_ctx *ctx, int T, int R, int N, int K, bool lora, int Nq, int Nkv) {
    FewArgs a{};
    return few_plan(ctx, T, R, N, K, lora, Nq, Nkv, false, a);
}

// Returns kernels launched, or -1.  `glu`: W holds gate and up rows, the output is silu(gate) * up (a kernel for that behind 40
// rows x 28672: 4 us).  `meta`: the batch's adapter facts of the layer (with the layer's A rows as tensor
// maps and its B slab), or nullptr for a plain dense projection.
int launch_few_cluster(alora_ctx *ctx, const void *x, const void *W, const RankMaps *tmA, const FewRowMeta *meta,
                       const void *b_all, int T, int R, int K, int N, int Nq, int Nkv, void *out, const void *residual, void *kv_pool,
                       int num_pages, bool x_early, cudaStream_t s, bool glu) {
    FewArgs a{};
    if (!few_plan(ctx, T, R, N, K, meta != nullptr, Nq, Nkv, x_early, a)) return -1;
    CUtensorMap tmX, tmW;
    if (!make_tensor_map_bf16(&tmX, x, T, K, K, 1 << a.rows_shift) || !make_tensor_map_bf16(&tmW, W, N, K, K, glu ? a.bn / 2 : a.bn)) return -1;
    a.meta = meta; a.b_all = (const __nv_bfloat16 *)b_all; a.Nq = Nq; a.Nkv = Nkv;
    a.residual = (const __nv_bfloat16 *)residual; a.out = (__nv_bfloat16 *)out; a.ldo = glu ? N / 2 : N; a.glu = glu ? 1 : 0; a.status = ctx->d_status;
    if (kv_pool != nullptr) {
        int shift = 0;
        while ((1 << shift) < ctx->d.hd) ++shift;
        a.kv_pool = (__nv_bfloat16 *)kv_pool; a.slot_map = ctx->d_slot; a.kv_hd_shift = shift; a.kv_heads = ctx->d.Hkv;
        a.kv_page_size = ctx->d.page; a.kv_num_pages = num_pages;
    }
    const int n_tiles = (N + a.bn - 1) / a.bn * a.n_rt;
    if (launch_cluster(dim3(n_tiles * a.ksplit), a.ksplit, (size_t)a.bar_off + 256 + 1024, s, tmX, tmW, meta ? *tmA : RankMaps{}, a) != cudaSuccess)
        return -1;
    // the attention work lists of this batch are built now, beside the weight stream (a dependent launch that reads
    // nothing this kernel writes; its blocks wait for this kernel before they exit)
    const BatchArgs *bm = ctx->pending_attn_meta;
    ctx->pending_attn_meta = nullptr;
    const int n = bm == nullptr ? 0 : launch_metadata(ctx, *bm, s, kMetaAttention, /*timed=*/false);
    return n < 0 ? -1 : 1 + n;
}

}  // namespace alora
