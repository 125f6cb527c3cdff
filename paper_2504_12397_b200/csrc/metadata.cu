// Batch metadata: per-token request / applied-adapter / KV-slot arrays and the projection's
// (row tile, adapter) pairs.  Integer work only; every output is compared exactly against the CPU oracle.
#include <algorithm>
#include <climits>
#include "alora_internal.h"
#include "tc_common.cuh"

namespace alora {

constexpr int kMetaSmemInts = 7168;   // 28 KB of builder scratch: batches of up to 511 requests
constexpr int kMetaStageR = 1024;     // per-request inputs of up to this many requests are staged in shared memory

// Request owning flat token t: largest r with query_start_loc[r] <= t (binary search; empty
// requests are skipped because their start equals their successor's).
__device__ __forceinline__ int find_request(const int32_t *qsl, int R, int t) {
    int lo = 0, hi = R;  // invariant: qsl[lo] <= t < qsl[hi]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (qsl[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// Per token: request index, adapter applied to the row (the gate of Eq. 5: position >= activation
// offset; always open in full-LoRA mode, always closed in base mode), and the token slot
// page * page_size + position % page_size.  Findings (inconsistent positions, page id out of
// range, adapter id out of range) go to the status word; the row then gets adapter -1 / slot -1 so that later kernels
// skip it.  The small fp32 layers find the same facts in a kernel of theirs (row_facts() in simt_kernels.cu): a change
// here is one there.  (Whether the adapter is registered on a layer is not looked at here: one that is not has rank 0 there.)
template <typename Hook>
__device__ __forceinline__ int metadata_token(int t, int p,
                                      const int32_t *__restrict__ a_req,
                                      const int32_t *__restrict__ adapter_ids,
                                      const int32_t *__restrict__ qsl, const int32_t *__restrict__ seq_lens,
                                      const int32_t *__restrict__ block_tables, int max_blocks,
                                      int num_pages, int page_size, int max_adapters, int T, int R, int mode,
                                      int32_t *__restrict__ token_req, int32_t *__restrict__ row_adapter,
                                      int32_t *__restrict__ slot_map, int32_t *status, Hook &&with_adapter) {
    if (t >= T) return -1;
    int r = find_request(qsl, R, t);
    // positions of a request are consecutive and end at seq_len - 1
    int expect = seq_lens[r] - (qsl[r + 1] - t);
    bool ok = (p == expect) && p >= 0;
    if (!ok) report(status, ALORA_ERR_BAD_BATCH);
    int k = -1;
    if (mode != ALORA_MODE_BASE && adapter_ids != nullptr) {
        k = adapter_ids[r];
        if (k >= max_adapters || k < -1) { report(status, ALORA_ERR_BAD_BATCH); k = -1; }
        if (k >= 0 && mode == ALORA_MODE_ALORA && p < a_req[r]) k = -1;
    }
    if (token_req) token_req[t] = r;
    k = ok ? k : -1;
    with_adapter(k);
    if (row_adapter) row_adapter[t] = k;
    if (slot_map) {
        int slot = -1;
        if (ok && block_tables != nullptr) {
            int blk = p / page_size;
            if (blk < max_blocks) {
                int page = block_tables[(size_t)r * max_blocks + blk];
                if (page >= 0 && page < num_pages) slot = page * page_size + p % page_size;
                else report(status, ALORA_ERR_PAGE_RANGE);
            } else {
                report(status, ALORA_ERR_BAD_BATCH);
            }
        }
        slot_map[t] = slot;
    }
    return k;
}

// The (row tile, adapter) pairs of the projection: for every tile of kTileRows rows the adapters whose gate is open on
// some row of it, in the order of their first request, each once; or the same for tiles of `tile_rows` rows.  One block; a
// warp per tile, a lane per request.  With `adapters` it also reports a request whose open rows name an adapter that some
// layer of the call has not registered.
__device__ __forceinline__ void metadata_pairs(const int32_t *__restrict__ a_req, const int32_t *__restrict__ adapter_ids,
                                               const int32_t *__restrict__ qsl, const int32_t *__restrict__ seq_lens,
                                               int R, int mode, int max_adapters, int T, int tile_rows, int max_pairs,
                                               TilePair *__restrict__ pairs, int32_t *__restrict__ pair_off,
                                               int32_t *__restrict__ n_pairs, int32_t *scratch /* [3R] */,
                                               const AdapterDev *__restrict__ adapters, int n_layers, int32_t *status) {
    constexpr int kBatch = 128;   // tiles per round
    __shared__ int r_lo[kBatch], r_hi[kBatch], cnt[kBatch], off_s[kBatch];
    __shared__ int total_s;
    int32_t *on0 = scratch, *on1 = scratch + R, *on_k = scratch + 2 * R;   // per request: rows with an open gate, adapter (-1: none)
    bool any = false;
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        const int n_new = qsl[r + 1] - qsl[r];
        int k = (mode == ALORA_MODE_BASE || adapter_ids == nullptr) ? -1 : adapter_ids[r];
        if (k >= max_adapters || k < -1) k = -1;
        int n_off = 0;
        if (k >= 0 && mode == ALORA_MODE_ALORA) {
            const long long d = (long long)a_req[r] - (seq_lens[r] - n_new);
            n_off = d <= 0 ? 0 : (d >= n_new ? n_new : (int)d);
        }
        if (n_off >= n_new) k = -1;
        on0[r] = qsl[r] + n_off; on1[r] = qsl[r + 1]; on_k[r] = k;
        any |= k >= 0;
        if (k >= 0 && adapters != nullptr)
            for (int l = 0; l < n_layers; ++l)
                if (adapters[(size_t)l * max_adapters + k].rank == 0) report(status, ALORA_ERR_NO_WEIGHTS);
    }
    any = __syncthreads_or(any);
    const int n_tiles = (T + tile_rows - 1) / tile_rows;
    if (!any) {   // base model only
        for (int i = threadIdx.x; i <= n_tiles; i += blockDim.x) pair_off[i] = 0;
        if (threadIdx.x == 0 && n_pairs != nullptr) *n_pairs = 0;
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = (int)blockDim.x >> 5;
    // adapters of tile `t` (requests lo .. hi): counted, or written from pairs[at] on; called by whole warps
    auto walk = [&](int t, int lo, int hi, bool write, int at) {
        const int row0 = t * tile_rows, row1 = min(row0 + tile_rows, T);
        int n = 0;
        for (int base = lo; base <= hi; base += 32) {
            const int r = base + lane;
            int k = -1;
            if (r <= hi && on0[r] < row1 && on1[r] > row0) k = on_k[r];
            const unsigned same = __match_any_sync(0xffffffffu, k);   // (every lane takes part)
            bool fresh = k >= 0 && __ffs(same) - 1 == lane;
            for (int q = lo; fresh && q < base; ++q)   // (only a tile with more than 32 requests)
                fresh = !(on_k[q] == k && on0[q] < row1 && on1[q] > row0);
            __syncwarp();
            const unsigned m = __ballot_sync(0xffffffffu, fresh);
            const int slot = at + n + __popc(m & ((1u << lane) - 1u));
            if (write && fresh && slot < max_pairs) { pairs[slot].tile = t; pairs[slot].adapter = k; }
            n += __popc(m);
        }
        return n;
    };
    int carry = 0;
    for (int t0 = 0; t0 < n_tiles; t0 += kBatch) {
        const int nb = min(kBatch, n_tiles - t0);
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
            r_lo[i] = find_request(qsl, R, (t0 + i) * tile_rows);
            r_hi[i] = find_request(qsl, R, min((t0 + i + 1) * tile_rows, T) - 1);
        }
        __syncthreads();
        for (int i = warp; i < nb; i += n_warps) {
            const int n = walk(t0 + i, r_lo[i], r_hi[i], false, 0);
            if (lane == 0) cnt[i] = n;
        }
        __syncthreads();
        if (warp == 0) {
            int acc = carry;
            for (int i = 0; i < nb; i += 32) {
                const int x = i + lane < nb ? cnt[i + lane] : 0;
                int inc = x;
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += v;
                }
                if (i + lane < nb) { off_s[i + lane] = acc + inc - x; pair_off[t0 + i + lane] = min(acc + inc - x, max_pairs); }
                acc += __shfl_sync(0xffffffffu, inc, 31);
            }
            if (lane == 0) total_s = acc;
        }
        __syncthreads();
        carry = total_s;
        for (int i = warp; i < nb; i += n_warps) walk(t0 + i, r_lo[i], r_hi[i], true, off_s[i]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (carry > max_pairs) report(status, ALORA_ERR_CAPACITY);
        pair_off[n_tiles] = min(carry, max_pairs);
        if (n_pairs != nullptr) *n_pairs = min(carry, max_pairs);
    }
}

// Which requests the few-row kernel takes (1 .. returned limit new tokens; the others go to the tensor-core
// kernel).  Normally the limit is small_max.  When the requests with 2 and more new tokens make at least two KV streams
// per SM, they fill the tensor-core kernel's blocks, and the limit is 1: that kernel then reads the cache faster than the
// few-row kernel (64 requests x 4 tokens on 4096 cached ones: 0.82 against 0.67 of the HBM bandwidth), and a few
// requests of 2 .. small_max tokens among longer ones would make a launch of their own behind it (48 requests of 3 .. 29
// tokens: 30 us).  Called by all threads of a block; both list builders take the same decision.
__device__ __forceinline__ int few_row_limit(const int32_t *__restrict__ qsl, int R, int Hkv, int n_sm, int small_max) {
    __shared__ int n_multi;
    if (threadIdx.x == 0) n_multi = 0;
    __syncthreads();
    int mine = 0;
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        const int n_new = qsl[r + 1] - qsl[r];
        mine += n_new >= 2;
    }
    if (mine) atomicAdd(&n_multi, mine);
    __syncthreads();
    const int n = n_multi;
    __syncthreads();   // (the counter may be reused by a second call in this block)
    return (long long)n * Hkv >= 2ll * n_sm ? min(1, small_max) : small_max;
}

// Attention work items of a prefill batch: each request's new tokens are cut into blocks of
// `q_block` tokens; one item per (request, KV head, block), blocks of the same KV stream adjacent so
// that blocks running at the same time share their K/V pages in L2.  Keys 0 .. position of the
// block's last token are visible to the block (causal limit); per-row limits are applied in the kernel.
// Requests are taken longest first (`order`, where the scratch has room for it), a request's last block first: the kernel's blocks
// claim the items in this order and end at about the same time.
// Where items of half the size still fit in one round over the n_blocks blocks of the kernel they are taken instead: a block of
// q_block / 2 tokens takes half as long (both query groups of the kernel work on the same rows, each on half of the keys).
__device__ __forceinline__ void metadata_attn_items(const int32_t *__restrict__ qsl, const int32_t *__restrict__ seq_lens,
                                           int R, int Hkv, int q_block, int small_max, int max_items,
                                           AttnWork *__restrict__ items, int32_t *__restrict__ counts,
                                           int32_t *blk_off /* [R+1] */, int32_t *order /* [2R] or nullptr */, int n_blocks,
                                           int32_t *__restrict__ cta_start, int32_t *status) {
    __shared__ int total;
    small_max = few_row_limit(qsl, R, Hkv, n_blocks, small_max);
    auto blocks_of = [&](int r) {   // (short requests: few-row list)
        const int n_new = qsl[r + 1] - qsl[r];
        return n_new > small_max ? (n_new + q_block - 1) / q_block : 0;
    };
    {
        __shared__ int n_half, n_tiles, longest;
        if (threadIdx.x == 0) n_half = n_tiles = longest = 0;
        __syncthreads();
        for (int r = threadIdx.x; r < R; r += blockDim.x) {
            const int n_new = qsl[r + 1] - qsl[r], n = blocks_of(r);
            if (n == 0) continue;
            atomicAdd(&n_half, (n_new + q_block / 2 - 1) / (q_block / 2));
            const int t = (seq_lens[r] + kAttnKeysPerTile - 1) / kAttnKeysPerTile;
            atomicAdd(&n_tiles, n * t);
            atomicMax(&longest, t);
        }
        __syncthreads();
        // (not where the items are long enough to be cut into runs, see below)
        if (n_half * Hkv <= n_blocks && longest < n_tiles * Hkv / n_blocks + kAttnSpreadMinGain) q_block /= 2;
        __syncthreads();
    }
    if (order != nullptr) {
        int32_t *key = order + R;
        for (int r = threadIdx.x; r < R; r += blockDim.x) key[r] = blocks_of(r) > 0 ? seq_lens[r] : 0;
        __syncthreads();
        for (int r = threadIdx.x; r < R; r += blockDim.x) {
            const int mine = key[r];
            int at = 0;
            for (int q = 0; q < R; ++q) at += key[q] > mine || (key[q] == mine && q < r);
            order[at] = r;
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < R; i += blockDim.x) blk_off[i] = blocks_of(order != nullptr ? order[i] : i);
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int r = 0; r < R; ++r) {
            const int n = blk_off[r];
            blk_off[r] = acc;
            acc += n;
        }
        blk_off[R] = acc;
        int n = acc * Hkv;
        if (n > max_items) { report(status, ALORA_ERR_CAPACITY); n = 0; }
        total = n;
        counts[1] = n;
        counts[15] = counts[16] = 0;   // (the kernel of layer l claims through the one and clears the other for layer l + 1)
    }
    __syncthreads();
    int sum = 0, tmin = INT_MAX, tmax = 0;   // key tiles of this thread's items
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        int lo = 0, hi = R;      // blk_off[lo] * Hkv <= i < blk_off[hi] * Hkv
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (blk_off[mid] * Hkv <= i) lo = mid; else hi = mid;
        }
        const int r = order != nullptr ? order[lo] : lo;
        const int nblk = blk_off[lo + 1] - blk_off[lo];
        const int rem = i - blk_off[lo] * Hkv;
        const int kvh = rem / nblk, blk = nblk - 1 - rem % nblk;
        const int n_new = qsl[r + 1] - qsl[r];
        AttnWork w;
        w.req = r;
        w.q_start = qsl[r] + blk * q_block;
        w.q_count = min(q_block, n_new - blk * q_block);
        w.kv_head = kvh;
        w.kv_start = 0;
        w.kv_end = seq_lens[r] - n_new + blk * q_block + w.q_count;  // last token's position + 1
        w.split = 0;
        w.n_splits = 1;
        items[i] = w;
        const int n = (w.kv_end + kAttnKeysPerTile - 1) / kAttnKeysPerTile;
        sum += n; tmin = min(tmin, n); tmax = max(tmax, n);
    }
    // Work split of the attention kernel over its n_blocks blocks (the launch uses that many whenever a cut is
    // possible).  Normally every item is taken whole.
    // Long batches (at least kAttnCutMinTiles key tiles per block) of items of nearly equal length that make at
    // least kAttnCutMinWaves full rounds: the first n_whole = n_blocks * floor(items / n_blocks) items are taken
    // whole; the key tiles of the remaining items are concatenated and cut into runs of equal length,
    // one per block, so an item can be cut into parts that different blocks work on (a merge kernel adds the
    // parts up).
    //   items[i].split = tiles before item i;  counts[6] = tiles in the concatenation, counts[7] = run length,
    //   counts[8] = n_whole, counts[9] = tiles before item n_whole;
    //   cta_start[c] = the item that holds the first tile of block c's run.
    __shared__ int warp_sum[32], warp_min[32], warp_max[32];
    __shared__ int run_len, run_off, run_first;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        tmin = min(tmin, __shfl_xor_sync(0xffffffffu, tmin, o));
        tmax = max(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    }
    if (lane == 0) { warp_sum[wid] = sum; warp_min[wid] = tmin; warp_max[wid] = tmax; }
    __syncthreads();   // (also: this block's writes to items[] are visible to all of its threads)
    if (threadIdx.x == 0) {
        int acc = 0, mn = INT_MAX, mx = 0;
        for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) {
            acc += warp_sum[w];
            mn = min(mn, warp_min[w]); mx = max(mx, warp_max[w]);
        }
        // cutting pays when most of the work is still done on whole items (whose sibling query blocks share their
        // K/V tiles in L2): items of nearly equal length, at least kAttnCutMinWaves full rounds of whole items
        const bool uniform = mx - mn <= max(1, mx / 16);
        const bool long_batch = acc >= kAttnCutMinTiles * n_blocks && uniform && total >= kAttnCutMinWaves * n_blocks &&
                                total % n_blocks != 0;
        // ... and a batch with fewer items than blocks (a few requests with long contexts) is spread over all blocks
        // when that still leaves every block a run of at least kAttnMinRunTiles key tiles and shortens the longest
        // block's work by more than the merge costs (about the time of kAttnSpreadMinGain key tiles, measured)
        const bool few_items = total > 0 && total < n_blocks && acc >= kAttnMinRunTiles * n_blocks &&
                               mx >= acc / n_blocks + kAttnSpreadMinGain;
        const bool cut = long_batch || few_items;
        run_first = !cut ? -1 : n_blocks * (total / n_blocks);
        run_len = acc;   // all tiles, for now
        if (!cut) { counts[6] = 0; counts[7] = kAttnMinRunTiles; counts[8] = total; counts[9] = acc; }
    }
    __syncthreads();
    if (run_first < 0) return;   // short batch: every item whole, nothing more to prepare
    // tiles before each item: contiguous chunks of items per thread, scanned over the block
    const int chunk = (total + (int)blockDim.x - 1) / (int)blockDim.x;
    const int lo = min(total, (int)threadIdx.x * chunk), hi = min(total, lo + chunk);
    sum = 0;
    for (int i = lo; i < hi; ++i) sum += (items[i].kv_end + kAttnKeysPerTile - 1) / kAttnKeysPerTile;
    int incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    __syncthreads();   // warp_sum is reused
    if (lane == 31) warp_sum[wid] = incl;
    __syncthreads();
    int acc = incl - sum;
    for (int w = 0; w < wid; ++w) acc += warp_sum[w];
    for (int i = lo; i < hi; ++i) {
        items[i].split = acc;
        acc += (items[i].kv_end + kAttnKeysPerTile - 1) / kAttnKeysPerTile;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int all = run_len, first = run_first;
        const int off = first < total ? items[first].split : all;
        const int len = max((all - off + n_blocks - 1) / n_blocks, kAttnMinRunTiles);
        counts[6] = all - off;
        counts[7] = len;
        counts[8] = first;
        counts[9] = off;
        run_len = len;
        run_off = off;
    }
    __syncthreads();
    const int len = run_len, off = run_off;
    for (int i = max(lo, run_first); i < hi; ++i) {
        const int rel = items[i].split - off;
        const int n = (items[i].kv_end + kAttnKeysPerTile - 1) / kAttnKeysPerTile;
        for (int c = (rel + len - 1) / len; c * len < rel + n && c < n_blocks; ++c) cta_start[c] = i;
    }
}

// Requests that read one shared prefix cache (several adapters invoked on the same conversation: their block tables
// start with the same physical pages).  Neighbouring requests of the few-row route are put into one PREFIX GROUP when
// they have leading pages in common, so that the attention reads those pages once for all of them:
//   common(r)  = the number of leading block-table entries that requests r-1 and r have in common, counted only over
//                pages that lie wholly before both requests' first new position;
//   a group starts at an eligible request f (1 .. small_max new tokens) and is extended by f+1, f+2, ... while the
//   next request is eligible, common(next) * page_size >= kMinSharedKeys, and the stacked score rows (new tokens of
//   all members x G) still fit into 64;  a group needs at least two members;
//   its shared length is the smallest common() of its pairs, in keys, rounded down to a multiple of 64.
// Output per request: grp_first (index of the group's first request; r itself when ungrouped) and grp_shared (the
// shared keys, 0 when ungrouped).  Called by all threads of a block.
constexpr int kMinSharedKeys = 256;
__device__ __forceinline__ void metadata_prefix_groups(const int32_t *__restrict__ qsl, const int32_t *__restrict__ seq_lens,
                                                       const int32_t *__restrict__ block_tables, int max_blocks, int R,
                                                       int page_size, int G, int small_max,
                                                       int32_t *__restrict__ grp_first, int32_t *__restrict__ grp_shared) {
    // common(r) for all pairs.  First the pairs that can share at all (both on this route, same first page): most
    // pairs of unrelated requests end here.  Then a warp per pair compares the table entries below the pair's limit,
    // 128 at a time with all loads in flight, up to the first mismatch.
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        int lim = 0;
        if (r > 0) {
            const int na = qsl[r] - qsl[r - 1], nb = qsl[r + 1] - qsl[r];
            if (na > 0 && nb > 0 && na <= small_max && nb <= small_max) {
                lim = min(min((seq_lens[r - 1] - na) / page_size, (seq_lens[r] - nb) / page_size), max_blocks);
                if (lim > 0 && block_tables[(size_t)(r - 1) * max_blocks] != block_tables[(size_t)r * max_blocks]) lim = 0;
            }
        }
        grp_first[r] = max(lim, 0);    // for now: the pair's limit (0: nothing in common)
        grp_shared[r] = max(lim, 0);   // for now: the first mismatching entry found so far (none yet)
    }
    __syncthreads();
    for (int r = 1 + (int)(threadIdx.x >> 5); r < R; r += (int)(blockDim.x >> 5)) {
        const int lim = grp_first[r], lane = threadIdx.x & 31;
        if (lim <= 1) continue;
        const int32_t *ta = block_tables + (size_t)(r - 1) * max_blocks, *tb = block_tables + (size_t)r * max_blocks;
        int first = lim;   // first mismatching entry
        for (int b0 = 1; b0 < lim && first == lim; b0 += 128) {
            int mine = lim;
#pragma unroll
            for (int u = 3; u >= 0; --u) {
                const int b = b0 + 32 * u + lane;
                if (b < lim && ta[b] != tb[b]) mine = b;
            }
            first = __reduce_min_sync(0xffffffffu, mine);
        }
        if (lane == 0) grp_shared[r] = first;
    }
    __syncthreads();
    // keys in common with the left neighbour; most batches have no pair that shares enough: then nobody is grouped and
    // the serial pass below (one thread walking the requests) is not needed
    bool any = false;
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        const int keys = grp_shared[r] * page_size;
        grp_shared[r] = keys;
        any |= keys >= kMinSharedKeys;
    }
    if (!__syncthreads_or(any)) {
        for (int r = threadIdx.x; r < R; r += blockDim.x) { grp_first[r] = r; grp_shared[r] = 0; }
        __syncthreads();
        return;
    }
    if (threadIdx.x == 0) {
        int f = 0;
        while (f < R) {
            const int nf = qsl[f + 1] - qsl[f];
            int e = f + 1;
            int shared = 0;
            if (nf > 0 && nf <= small_max) {
                int rows = nf * G, mn = 0x7fffffff;
                while (e < R) {
                    const int ne = qsl[e + 1] - qsl[e];
                    const int c = grp_shared[e];
                    if (!(ne > 0 && ne <= small_max) || c < kMinSharedKeys || rows + ne * G > 64) break;
                    rows += ne * G;
                    mn = min(mn, c);
                    ++e;
                }
                if (e - f >= 2) shared = mn & ~63;
            }
            if (shared <= 0) { e = f + 1; shared = 0; }
            for (int m = f; m < e; ++m) { grp_first[m] = f; }
            // grp_shared[f + 1 .. e) still hold the pair values that the loop above read; overwrite after use
            for (int m = f; m < e; ++m) grp_shared[m] = shared;
            f = e;
        }
    }
    __syncthreads();
}

// Work list of the few-row attention kernel: requests with 1 .. small_max new tokens (at most 16 score rows (token, query
// head of the group) per KV head).  A STREAM is one block of score rows with the keys it reads: for an ungrouped
// request its rows over keys 0 .. causal limit; for a prefix group the stacked rows of all members (16 * mt, mt = 1, 2
// or 4), over the shared prefix (read once, nothing masked) followed by every member's own keys beyond it (masked so
// that only that member's rows see them).  A stream's keys are cut into ranges of at most `chunk` 64-key units, which are
// merged by whichever block finishes last.  The list holds the ranges of whole streams and shared prefixes first and
// the groups' own keys after them: those are short and fill the blocks that have no long range left.
// A group is owned by its first request: that request accounts for all of the group's items.
//
// What bounds it: latency, in front of the attention of the first layer.  Everything that is needed more than once per
// request (units, members, row tiles) is computed once in parallel; sums and offsets are block-wide scans.
__device__ __forceinline__ int units_to_ranges(int units, int chunk) { return (units + chunk - 1) / chunk; }

// Exclusive sums of v[0 .. R) and w[0 .. R) in place; returns the totals.  All threads of a block of whole warps.
__device__ __forceinline__ int2 block_scan2(int32_t *v, int32_t *w, int R) {
    __shared__ int2 warp_tot[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, n_warps = (int)blockDim.x >> 5;
    int2 carry = make_int2(0, 0);
    for (int base = 0; base < R; base += (int)blockDim.x) {
        const int r = base + (int)threadIdx.x;
        const int2 x = r < R ? make_int2(v[r], w[r]) : make_int2(0, 0);
        int2 inc = x;
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, inc.x, o), b = __shfl_up_sync(0xffffffffu, inc.y, o);
            if (lane >= o) { inc.x += a; inc.y += b; }
        }
        if (lane == 31) warp_tot[wid] = inc;
        __syncthreads();
        int2 before = carry;
        for (int i = 0; i < n_warps; ++i) {
            const int2 t = warp_tot[i];
            if (i < wid) { before.x += t.x; before.y += t.y; }
            carry.x += t.x; carry.y += t.y;
        }
        if (r < R) { v[r] = before.x + inc.x - x.x; w[r] = before.y + inc.y - x.y; }
        __syncthreads();
    }
    return carry;
}

__device__ __forceinline__ void metadata_split_items(const int32_t *__restrict__ qsl, const int32_t *__restrict__ seq_lens,
                                                     const int32_t *__restrict__ block_tables, int max_blocks, int page_size,
                                                     int R, int Hkv, int G, int n_sm, int small_max, int max_items, int max_rows,
                                                     AttnSplitWork *__restrict__ items, int32_t *__restrict__ counts,
                                                     int32_t *req_scratch /* [kSplitScratch][R] */,
                                                     int32_t *__restrict__ group_done, int32_t *__restrict__ groups_out,
                                                     int part, int n_parts, int32_t *status) {
    // (several blocks may build the list together: each repeats the cheap per-request passes and fills the items
    // part, part + n_parts, ..; block `part` 0 alone writes the counts and reports findings)
    __shared__ int chunk_units, total_items, few_ranges, max_units;
    __shared__ unsigned long long best;
    small_max = few_row_limit(qsl, R, Hkv, n_sm, small_max);
    int32_t *req_off = req_scratch, *own_off = req_scratch + 7 * R, *req_row = req_scratch + R, *grp_first = req_scratch + 2 * R, *grp_shared = req_scratch + 3 * R;
    int32_t *u_shared = req_scratch + 4 * R;   // 64-key units of the stream (of the shared prefix, for a group's owner)
    int32_t *u_own = req_scratch + 5 * R;      // a group's units beyond the shared prefix, member after member
    int32_t *shape = req_scratch + 6 * R;      // members * 8 + row tiles; 0: the request owns no items
    metadata_prefix_groups(qsl, seq_lens, block_tables, max_blocks, R, page_size, G, small_max, grp_first, grp_shared);
    if (groups_out != nullptr && part == 0)
        for (int r = threadIdx.x; r < R; r += blockDim.x) { groups_out[r] = grp_first[r]; groups_out[R + r] = grp_shared[r]; }
    if (threadIdx.x == 0) { max_units = 4; best = ~0ull; }
    __syncthreads();
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        const int n_new = qsl[r + 1] - qsl[r];
        int us = 0, uo = 0, sh = 0;
        if (n_new > 0 && n_new <= small_max && grp_first[r] == r) {
            const int shared = grp_shared[r];
            int e = r + 1;
            if (shared > 0) {
                us = shared / 64;
                uo = (seq_lens[r] - shared + 63) / 64;
                for (; e < R && grp_first[e] == r; ++e) uo += (seq_lens[e] - shared + 63) / 64;
            } else {
                us = (seq_lens[r] + 63) / 64;
            }
            const int rows = (qsl[e] - qsl[r]) * G;
            sh = (e - r) * 8 + (rows <= 16 ? 1 : (rows <= 32 ? 2 : 4));
        }
        u_shared[r] = us; u_own[r] = uo; shape[r] = sh;
        // units weighted by the row tiles (an item of mt tiles needs mt * 16 partial rows), for the sum below
        req_off[r] = (us + uo) * (sh & 7) * Hkv; req_row[r] = 0;
        if (max(us, uo) > 4) atomicMax(&max_units, max(us, uo));
    }
    __syncthreads();
    const int tot_units = block_scan2(req_off, req_row, R).x;
    if (threadIdx.x == 0) {
        // Range length: a range costs a fixed time beyond its streaming time (item claim, first table window and
        // first copies, query fetch, combining the warps, publishing the partial result, a share of the merge), and
        // the last ranges of a launch leave SMs idle for up to one range.  With t = streaming time of all units on
        // one SM (0.74 us per 64-key unit at an SM's share of the HBM bandwidth) the sum of both losses is smallest
        // near sqrt(t / c) ranges per SM, capped by the capacity of the work list; c = 12 us is what batches of 2
        // to 64 requests with 4096 to 32768 cached tokens run fastest with (3 us: 5 .. 16 % slower on the small ones).
        const float t_us = (float)tot_units * 0.74f / (float)max(n_sm, 1);
        const float per_sm = fminf(fmaxf(sqrtf(t_us / 12.f), 1.f), (float)kSplitItemsPerSm);
        const int target = (int)ceilf(per_sm * (float)max(n_sm, 1));
        chunk_units = max(4, (int)(((long long)tot_units + target - 1) / target));
        few_ranges = (tot_units > 0 && per_sm < 2.5f) ? 1 : 0;
    }
    __syncthreads();
    // With only one or two ranges per SM the rule above ignores how the ranges fall into rounds over the SMs: 192
    // equal ranges on 148 SMs take as long as 296.  Such batches (a few requests) instead take the range length that the
    // same cost model finds fastest: whole rounds of the long ranges, 12 us + length x 0.74 us each, and the groups' own
    // keys in the gaps of the last round, or after it where they do not fit.
    if (few_ranges) {
        // every thread tries one candidate length (a grid over 4 .. the longest stream)
        const int step = max((max_units - 4 + (int)blockDim.x - 1) / (int)blockDim.x, 1), cand = 4 + (int)threadIdx.x * step;
        if (cand <= max_units + step) {
            int n_long = 0, n_own = 0, own_units = 0;
#pragma unroll 4
            for (int r = 0; r < R; ++r) {
                n_long += units_to_ranges(u_shared[r], cand);
                n_own += units_to_ranges(u_own[r], cand);
                own_units += u_own[r];
            }
            n_long *= Hkv; n_own *= Hkv; own_units *= Hkv;
            const float t_long = 12.f + 0.74f * (float)cand;
            const float t_own = n_own > 0 ? 12.f + 0.74f * (float)own_units / (float)n_own : 0.f;
            const float rounds = (float)((n_long + n_sm - 1) / n_sm) * t_long;
            const float all = ((float)n_long * t_long + (float)n_own * t_own) / (float)n_sm + 0.5f * t_own;
            atomicMin(&best, ((unsigned long long)(unsigned)(fmaxf(rounds, all) * 16.f) << 32) | (unsigned)cand);
        }
        __syncthreads();
        if (threadIdx.x == 0) chunk_units = (int)(best & 0xffffffffu);
        __syncthreads();
    }
    const int chunk = chunk_units;
    for (int r = threadIdx.x; r < R; r += blockDim.x) {
        const int n = units_to_ranges(u_shared[r], chunk) * Hkv, n_own = units_to_ranges(u_own[r], chunk) * Hkv;
        req_off[r] = n; own_off[r] = n_own;
        req_row[r] = (n + n_own) * 16 * (shape[r] & 7);
        grp_first[r] = 0;   // (not needed any more: second array of the row scan)
    }
    __syncthreads();
    const int2 total = block_scan2(req_off, own_off, R);
    const int total_rows = block_scan2(req_row, grp_first, R).x;
    if (threadIdx.x == 0) {
        int n = total.x + total.y;
        if (n > max_items || total_rows > max_rows) {
            if (part == 0) report(status, ALORA_ERR_CAPACITY);
            n = 0;
        }
        total_items = n;
        if (part == 0) {
            counts[3] = n;
            counts[4] = 0;   // work counter of the few-row kernel
        }
    }
    __syncthreads();
    // one item per thread and step: owner request by binary search over the item offsets, then stream / KV head / range
    for (int i = part * (int)blockDim.x + (int)threadIdx.x; i < total_items; i += n_parts * (int)blockDim.x) {
        const bool own = i >= total.x;
        const int32_t *off = own ? own_off : req_off;
        const int idx = own ? i - total.x : i;
        int lo = 0, hi = R;   // the largest r with off[r] <= idx owns the item (requests without items share their successor's offset)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off[mid] <= idx) lo = mid; else hi = mid;
        }
        const int r = lo, n_mem = shape[r] >> 3, mt = shape[r] & 7;
        const int us = u_shared[r], uo = u_own[r];
        const int np = units_to_ranges(us, chunk), nt = units_to_ranges(uo, chunk), per_head = own ? nt : np;
        const int local = idx - off[r], kvh = local / per_head, sp = local % per_head;
        const int shared = grp_shared[r], n_tok = qsl[r + n_mem] - qsl[r];
        AttnSplitWork w;
        w.req = r; w.q_start = qsl[r]; w.q_count = n_tok; w.kv_head = kvh; w.mt = mt; w.n_splits = np + nt;
        w.split = own ? np + sp : sp;
        w.part_row0 = req_row[r] + (kvh * (np + nt) + w.split) * 16 * mt;
        if (!own) {   // (equal ranges rather than full ones and a stub)
            const int per = (us + np - 1) / np;
            const int kv_end = shared > 0 ? shared : seq_lens[r];   // last visible position + 1
            w.kv_start = sp * per * 64; w.kv_end = min(kv_end, (sp + 1) * per * 64);
            w.pos0 = shared > 0 ? shared : seq_lens[r] - n_tok;     // every row sees every key of a shared prefix
            w.pad_ = 0;
        } else {
            // a prefix group's members' own keys: stages [kv_start / 64, kv_end / 64) (not key positions: the kernel walks
            // the members to find each stage's request, key positions and rows)
            const int per = (uo + nt - 1) / nt;
            w.kv_start = sp * per * 64; w.kv_end = min(uo, (sp + 1) * per) * 64;
            w.pos0 = shared;
            w.pad_ = kSplitOwnKeys | n_mem;
        }
        if (w.split == 0) group_done[w.part_row0 / 16] = 0;
        items[i] = w;
    }
}

// FewRowMeta of a tile of at most kFewRowMax rows, thread t's applied adapter being k_mine (-1: none, or no such
// row) and `ad` that adapter: the adapters that occur, ascending, each one's padded rank and scale, and every row's slot.
// Called by all kFewRowMax threads of a block.
__device__ __forceinline__ void metadata_few_row(int k_mine, const AdapterDev &ad, int max_adapters, FewRowMeta *__restrict__ meta) {
    __shared__ uint32_t bits[32], below[32];   // adapters present, 32 to a word; how many there are in the words before
    if (threadIdx.x < 32) bits[threadIdx.x] = 0u;
    __syncthreads();
    if (k_mine >= 0 && k_mine < max_adapters && k_mine < 1024) atomicOr(&bits[k_mine >> 5], 1u << (k_mine & 31));
    else k_mine = -1;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, n = __popc(bits[lane]);
        int sum = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, sum, off);
            if (lane >= off) sum += v;
        }
        below[lane] = (uint32_t)(sum - n);
        if (lane == 31) meta->n_present = sum;
    }
    __syncthreads();
    int slot = -1;
    if (k_mine >= 0) {   // (the rows of an adapter all write the same)
        slot = (int)below[k_mine >> 5] + __popc(bits[k_mine >> 5] & ((1u << (k_mine & 31)) - 1u));
        meta->id[slot] = k_mine; meta->rpad[slot] = ad.rpad; meta->scale[slot] = ad.scale;
    }
    if ((int)threadIdx.x < kFewRowMax) meta->slot_of_row[threadIdx.x] = slot;
}

// The metadata step.  Phase bit 0: every block handles 256 tokens (request, applied adapter, slot); two blocks more
// build the projection's (row tile, adapter) pairs and (quad, adapter) entries.  Phase bit 1: the two attention
// work lists, one block each (their serial parts are O(R)).  Both phases in one launch: the last block, 1 and 2 take one
// builder each.  The attention phase alone is launched as a programmatic dependent of the projection kernel, beside
// which it runs (it reads nothing that kernel writes); its blocks wait for that kernel before they exit, so that
// whatever follows in the stream still sees the projection complete.
__global__ void __launch_bounds__(256)
metadata_kernel(const int32_t *__restrict__ positions, const int32_t *a_req, const int32_t *adapter_ids,
                const int32_t *qsl, const int32_t *seq_lens, const int32_t *__restrict__ block_tables, int max_blocks,
                int num_pages, int page_size, int max_adapters, int T, int R, int mode,
                int32_t *__restrict__ token_req, int32_t *__restrict__ row_adapter, int32_t *__restrict__ slot_map,
                int max_pairs, TilePair *__restrict__ pairs, int32_t *__restrict__ pair_off, int max_quads,
                TilePair *__restrict__ quads, int32_t *__restrict__ quad_off, int32_t *__restrict__ counts, int32_t *seg_scratch,
                int Hkv, int q_block, int max_items, AttnWork *__restrict__ items, int32_t *blk_off,
                int G, int n_sm, int small_max, int max_split_items, int max_split_rows,
                AttnSplitWork *__restrict__ split_items,
                int32_t *req_scratch, int32_t *__restrict__ group_done,
                int32_t *__restrict__ attn_cta_start, const AdapterDev *__restrict__ adapters, int n_layers, int phases,
                int32_t *__restrict__ prefix_groups, int32_t *status) {
    // The per-request inputs are read many times (binary searches, list builders): one parallel pass stages them
    // in shared memory, so that the later steps do not each pay a round trip to global memory.
    __shared__ int32_t s_req[4 * kMetaStageR + 1];
    // The first launch of a call is a dependent one too, but lets its successor start only when everything before the call
    // has completed: later kernels rely on that for what they read of the caller's before their own wait.
    if (phases & kMetaProjection) tc::grid_dep_wait();
    tc::grid_dep_launch();   // the next kernel's blocks may start their set-up; they wait for this kernel's results
    const int tok = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const int my_pos = (phases & kMetaProjection) && tok < T ? positions[tok] : 0;   // (in flight with the per-request inputs)
    if (R <= kMetaStageR) {
        int32_t *s_qsl = s_req, *s_len = s_req + R + 1, *s_ids = s_len + R, *s_areq = s_ids + R;
        for (int i = threadIdx.x; i <= R; i += blockDim.x) s_qsl[i] = qsl[i];
        for (int i = threadIdx.x; i < R; i += blockDim.x) {
            s_len[i] = seq_lens[i];
            if (adapter_ids) s_ids[i] = adapter_ids[i];
            if (a_req) s_areq[i] = a_req[i];
        }
        __syncthreads();
        qsl = s_qsl; seq_lens = s_len;
        if (adapter_ids) adapter_ids = s_ids;
        if (a_req) a_req = s_areq;
    }
    if ((phases & kMetaProjection) && tok < T)
        metadata_token(tok, my_pos, a_req, adapter_ids, qsl, seq_lens, block_tables,
                       max_blocks, num_pages, page_size, max_adapters, T, R, mode, token_req, row_adapter, slot_map, status, [](int) {});
    // The list builders are independent of one another: the last two blocks, 1 and 2 take one each (a launch of both
    // phases has at least five blocks, one of the attention phase alone two).
    const int nb = (int)gridDim.x;
    const bool proj = (phases & kMetaProjection) != 0, attn = (phases & kMetaAttention) != 0;
    const int b_pairs = proj && pairs != nullptr ? nb - 1 : -1;   // (a block without tokens of its own: the projection waits for it)
    const int b_quads = proj && quads != nullptr ? nb - 2 : -1;
    const int b_attn = !attn ? -1 : (proj ? (nb > 1 ? 1 : 0) : 0);
    const int b_split = !attn ? -1 : (proj ? (nb > 2 ? 2 : 0) : (nb > 1 ? 1 : 0));
    // the attention phase alone: block 0 builds the tensor-core kernel's list, all the others share the few-row list
    const int split_parts = (!proj && attn && nb > 1) ? nb - 1 : 1;
    const bool split_helper = !proj && attn && (int)blockIdx.x > b_split;
    if ((int)blockIdx.x != b_pairs && (int)blockIdx.x != b_quads && (int)blockIdx.x != b_attn && (int)blockIdx.x != b_split && !split_helper) {
        if (!proj) tc::grid_dep_wait();
        return;
    }
    // the per-request scratch of the list builders (their serial parts walk it) lives in shared memory when the
    // batch is small enough, else in the context's global scratch (one buffer per builder)
    __shared__ int32_t smem_scratch[kMetaSmemInts];
    if (14 * R + 5 <= kMetaSmemInts) seg_scratch = blk_off = req_scratch = smem_scratch;
    __syncthreads();
    if ((int)blockIdx.x == b_pairs) {
        metadata_pairs(a_req, adapter_ids, qsl, seq_lens, R, mode, max_adapters, T, kTileRows, max_pairs, pairs, pair_off, counts + 2,
                       seg_scratch, adapters, n_layers, status);
        __syncthreads();  // a builder that follows in this block reuses the scratch
    } else if ((int)blockIdx.x == b_quads) {
        metadata_pairs(a_req, adapter_ids, qsl, seq_lens, R, mode, max_adapters, T, kQuadRows, max_quads, quads, quad_off, nullptr,
                       seg_scratch == smem_scratch ? smem_scratch : seg_scratch + 3 * R, nullptr, 0, status);
    }
    if ((int)blockIdx.x == b_attn && items != nullptr && block_tables != nullptr) {
        metadata_attn_items(qsl, seq_lens, R, Hkv, q_block, small_max, max_items, items, counts, blk_off,
                            blk_off == smem_scratch ? smem_scratch + R + 1 : nullptr, n_sm, attn_cta_start, status);
        __syncthreads();
    }
    if (((int)blockIdx.x == b_split || split_helper) && split_items != nullptr && block_tables != nullptr)
        metadata_split_items(qsl, seq_lens, block_tables, max_blocks, page_size, R, Hkv, G, n_sm, small_max, max_split_items,
                             max_split_rows, split_items, counts, req_scratch, group_done, prefix_groups,
                             split_helper ? (int)blockIdx.x - b_split : 0, split_parts, status);
    if (!proj) tc::grid_dep_wait();
}

// The projection phase for a batch on the few-row route (at most kFewTiles tiles of kFewRowMax tokens): per-token arrays and
// the adapter facts, nothing else.  A kernel of its own because every step of a decode loop waits for it: what it costs is mostly
// the fetch of its instructions, and this one is short.  Block (tile, l) writes the tile's facts of layer l of the call (a stack call
// builds those of all layers in one launch: with a launch per layer each layer waited 10 us for it), those of layer 0 also
// the per-token arrays.  row_adapter holds the adapter of every row whose gate is open; whether it is registered on a layer
// (else: base output and a finding) goes into that layer's facts.
__global__ void __launch_bounds__(kFewRowMax)
metadata_few_row_kernel(const int32_t *__restrict__ positions, const int32_t *a_req, const int32_t *adapter_ids,
                        const int32_t *qsl, const int32_t *seq_lens, const int32_t *__restrict__ block_tables,
                        int max_blocks, int num_pages, int page_size, int max_adapters, int T, int R, int mode,
                        int32_t *__restrict__ token_req, int32_t *__restrict__ row_adapter,
                        int32_t *__restrict__ slot_map, const AdapterDev *__restrict__ adapters,
                        FewRowMeta *__restrict__ few_row_meta, int few_tiles, int32_t *status) {
    __shared__ int32_t s_req[4 * kFewRowMax + 1];
    tc::grid_dep_wait();     // (in this order: see metadata_kernel)
    tc::grid_dep_launch();
    const int tok = (int)(blockIdx.x * kFewRowMax + threadIdx.x), my_pos = tok < T ? positions[tok] : 0;   // (in flight with the per-request inputs)
    if (R <= kFewRowMax) {   // the per-request inputs are read several times (binary search): stage them
        int32_t *s_qsl = s_req, *s_len = s_req + R + 1, *s_ids = s_len + R, *s_areq = s_ids + R;
        for (int i = threadIdx.x; i <= R; i += blockDim.x) s_qsl[i] = qsl[i];
        for (int i = threadIdx.x; i < R; i += blockDim.x) {
            s_len[i] = seq_lens[i];
            if (adapter_ids) s_ids[i] = adapter_ids[i];
            if (a_req) s_areq[i] = a_req[i];
        }
        __syncthreads();
        qsl = s_qsl; seq_lens = s_len;
        if (adapter_ids) adapter_ids = s_ids;
        if (a_req) a_req = s_areq;
    }
    // (the adapter is fetched beside the block-table entry: neither waits for the other)
    const bool first = blockIdx.y == 0;
    AdapterDev ad{};
    int k = metadata_token(tok, my_pos, a_req, adapter_ids, qsl, seq_lens, first ? block_tables : nullptr,
                           max_blocks, num_pages, page_size, max_adapters, T, R, mode, first ? token_req : nullptr,
                           first ? row_adapter : nullptr, first ? slot_map : nullptr, status,
                           [&](int applied) { if (few_row_meta != nullptr && applied >= 0) ad = adapters[(size_t)blockIdx.y * max_adapters + applied]; });
    if (few_row_meta != nullptr) {
        if (k >= 0 && ad.rank == 0) { report(status, ALORA_ERR_NO_WEIGHTS); k = -1; }
        metadata_few_row(k, ad, max_adapters, few_row_meta + (size_t)blockIdx.y * few_tiles + blockIdx.x);
    }
}

int launch_metadata(alora_ctx *ctx, const BatchArgs &b, cudaStream_t s, int phases, bool timed) {
    if (b.T == 0) {
        if (phases & kMetaProjection) cudaMemsetAsync(ctx->d_counts, 0, 6 * sizeof(int32_t), s);
        return 0;
    }
    const bool saved = ctx->profiling;
    if (!timed) ctx->profiling = false;
    ProfScope prof(ctx, KK_METADATA, s);
    ctx->profiling = saved;
    const int threads = 256;
    const bool attn_only = phases == kMetaAttention;
    // (attention phase alone: one block for the tensor-core list, kSplitBuilders for the few-row list; they need the
    // shared-memory scratch, i.e. batches of at most 511 requests, else one block builds it in the global scratch)
    constexpr int kSplitBuilders = 8;
    const int grid = attn_only ? (14 * b.R + 5 <= kMetaSmemInts ? 1 + kSplitBuilders : 2) : 2 + std::max((phases & kMetaAttention) ? 3 : 1, (b.T + threads - 1) / threads);
    const AdapterDev *ads = b.layer >= 0 ? ctx->d_adapters + (size_t)b.layer * ctx->cfg.max_adapters : nullptr;
    if (phases == kMetaProjection && b.few_row) {
        FewRowMeta *few = ads != nullptr ? ctx->d_skinny_meta + (size_t)b.layer * ctx->few_tiles : nullptr;
        return launch_kernel(metadata_few_row_kernel, dim3((b.T + kFewRowMax - 1) / kFewRowMax, b.n_layers), dim3(kFewRowMax), 0, s, true,
            b.positions, b.activation_offsets, b.adapter_ids, b.query_start_loc, b.seq_lens, b.block_tables, b.max_blocks,
            b.num_pages, ctx->d.page, ctx->cfg.max_adapters, b.T, b.R, b.mode, ctx->d_token_req, ctx->d_row_adapter,
            ctx->d_slot, ads, few, ctx->few_tiles, ctx->d_status) == cudaSuccess ? 1 : -1;
    }
    const cudaError_t e = launch_kernel(metadata_kernel, dim3(grid), dim3(threads), 0, s, true,
        b.positions, b.activation_offsets, b.adapter_ids, b.query_start_loc, b.seq_lens, b.block_tables,
        b.max_blocks, b.num_pages, ctx->d.page, ctx->cfg.max_adapters, b.T, b.R, b.mode, ctx->d_token_req,
        ctx->d_row_adapter, ctx->d_slot, ctx->max_pairs, ctx->d_pairs, ctx->d_pair_off, ctx->max_quads, ctx->d_quads, ctx->d_quad_off, ctx->d_counts, ctx->d_seg_scratch,
        ctx->d.Hkv, ctx->attn_q_block, ctx->max_attn_items, ctx->d_attn_items, ctx->d_attn_off, ctx->d.G,
        ctx->sm_count, ctx->small_max_tokens, ctx->max_split_items, ctx->max_split_rows, ctx->d_split_items,
        ctx->d_req_scratch, ctx->d_group_done,
        ctx->d_attn_cta_start, ads, b.n_layers, phases, ctx->d_prefix_groups, ctx->d_status);
    return e == cudaSuccess ? 1 : -1;
}

}  // namespace alora
