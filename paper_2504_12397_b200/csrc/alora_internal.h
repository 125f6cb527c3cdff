// Internal declarations shared by the library's translation units (not part of the C ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "alora.h"

namespace alora {

constexpr int kRankPadMax = 64;  // adapters are stored padded to a multiple of 16 rows, <= 64
constexpr int kMlpChunk = 8192;   // tokens per MLP pass of the stack entry (bounds the gate/up buffer)

// Per (layer, adapter) record as the kernels see it.  A is [3][rpad_max][H] (q, k, v blocks, rows
// beyond the rank are zero), B is [N][rpad_max] (row n holds the B row of output column n, columns
// beyond the rank are zero).
struct AdapterDev {
    const void *A;
    const void *B;
    int32_t rank;   // 0 = not registered
    int32_t rpad;   // rank rounded up to 16
    float scale;
    int32_t b_odd;  // B holds an Inf or NaN: its delta may not go through a row tile's matrix product (TilePair)
};

// One adapter's part on the MLP block of one layer (gate, up and down projections share rank and scale).
struct MlpAdapterDev {
    int32_t rpad;   // rank rounded up to 16; 0 = no MLP part registered
    float scale;
    int32_t b_odd;  // a B matrix holds an Inf or NaN (as in AdapterDev)
};

struct LayerWeights {
    const void *wqkv = nullptr, *wo = nullptr, *wgate_up = nullptr, *wdown = nullptr;
    const void *norm_attn = nullptr, *norm_mlp = nullptr;
};

// The projection works on dense tiles of kTileRows rows.  A row tile meets the adapters applied to its rows (gate open)
// one after another: one TilePair per (row tile, adapter that occurs in it).  The pair's t = s A x is kept for the whole
// tile with the rows of other adapters and the rows with a closed gate set to zero, so the expand step t B^T adds
// nothing to them.  That takes a finite B (0 x Inf is a NaN in every row of the tile): where registration has met an Inf or
// NaN, the pair's matrix product is left out and the epilogue adds the delta to the adapter's own rows on the CUDA cores
// (tc::OddRow).
constexpr int kTileRows = 128;
struct TilePair {
    int32_t tile, adapter;
};
// The same for the kernel that works on four row tiles at once (gemm_duo_tcgen05.cu): one entry per (quad, adapter), `tile` the quad.
constexpr int kQuadRows = 4 * kTileRows;
// Batches of at most this many rows carry t as the sum of three bf16 values (all 24 bits of its fp32 value, for the few rows
// of a handful of requests), larger ones as one.
constexpr int kSplitTTokens = 1024;

// One unit of attention work: query tokens [q_start, q_start + q_count) of request `req` (flat
// token indices), one KV head, keys [kv_start, kv_end) of the request's sequence.
struct AttnWork {
    int32_t req;
    int32_t q_start;
    int32_t q_count;
    int32_t kv_head;
    int32_t kv_start;
    int32_t kv_end;
    int32_t split;     // 128-key tiles of all earlier items of the work list
    int32_t n_splits;
};
constexpr int kAttnKeysPerTile = 128;   // keys per K/V tile of the tensor-core attention kernel
constexpr int kAttnMinRunTiles = 8;     // shortest run of key tiles given to one block
constexpr int kAttnCutMinTiles = 128;   // items are cut into runs only when a block has at least this many tiles to do
constexpr int kAttnCutMinWaves = 3;     // ... and the items make at least this many full rounds over the blocks
constexpr int kAttnSpreadMinGain = 24; // fewer items than blocks: spread them only if the longest item is this many tiles longer than a block's run

// One unit of few-row (decode / short suffix) attention work: score rows of `q_count` tokens starting at
// flat token q_start (rows are (token, query head of the group) pairs, `mt` tiles of 16 rows), one KV
// head, keys [kv_start, kv_end) of the request.  The `n_splits` key ranges of the same rows have consecutive
// blocks of 16 * mt partial rows (range `split` the split-th one); their partial results are merged afterwards.
struct AttnSplitWork {
    int32_t req, q_start, q_count, kv_head;
    int32_t kv_start, kv_end, pos0, mt;      // pos0 = position of the first token of the block
    int32_t split, n_splits, part_row0;        // part_row0 = first row of this item in the partial-result arrays
    int32_t pad_;   // 0: every token of the block sees keys up to its own position.  kSplitOwnKeys | n_members: the item
                    // covers the OWN keys of a prefix group's members (requests req .. req + n_members - 1), i.e. their
                    // keys from position pos0 (the shared length) on, as one sequence of 64-key stages, member after
                    // member; kv_start / kv_end count those stages (x 64); a stage's keys are seen by its member's
                    // tokens only, up to each token's own position
};
constexpr int32_t kSplitOwnKeys = 0x40000000;
constexpr int kSplitScratch = 8;       // per-request integers that the builder of the few-row list needs
constexpr int kSplitItemsPerSm = 16;   // target number of (row tile, key range) pairs per SM

// Few-row projection: what it needs to know about a tile of at most kFewRowMax rows of the batch, the tile's
// adapters, written by the batch-metadata step: the adapters that occur among the rows' applied adapters
// (ascending ids), per slot the padded rank and the scale, and per row the slot of its adapter.
constexpr int kFewRowMax = 128;
constexpr int kFewTiles = 8;   // row tiles of a batch on that route
struct FewRowMeta {
    int32_t n_present;
    int32_t pad_[3];
    int32_t slot_of_row[kFewRowMax];  // -1: the row adds no delta
    int32_t id[kFewRowMax];           // adapter id of each slot
    int32_t rpad[kFewRowMax];         // its rank rounded up to 16
    float scale[kFewRowMax];
};

// Kernel families, for the optional per-kernel timing (alora_profile_*).
enum KernelKind { KK_METADATA = 0, KK_SHRINK, KK_PROJECT, KK_KV_APPEND, KK_ATTENTION, KK_ATTN_FEW_ROW, KK_LINEAR,
                  KK_GLUE, KK_COUNT };

struct ProfEvent {
    cudaEvent_t begin, end;
    int kind;
};

// All adapters' A rows [max_adapters * 192][H] in boxes of 16, 32, 48 and 64 rows: box[r / 16 - 1] fetches the rows of one q / k /
// v block of an adapter of padded rank r in one copy (a copy takes 75 ns however few rows it brings).
struct RankMaps { CUtensorMap box[4]; };

// Tensor maps of one layer that depend only on registered weights (bf16 tensor-core path).
struct TcLayerMaps {
    CUtensorMap wqkv[3];      // W_qkv [N][H], boxes of 128 / 256 / 64 rows
    CUtensorMap a_all;        // all adapters' A rows [max_adapters*192][H], box 192 rows
    RankMaps a_rank;
    CUtensorMap b_all_bn[3];  // all adapters' B rows [max_adapters*N][64], boxes of 128 / 256 / 64 rows
};

struct Dims {
    int H, Hq, Hkv, hd, G, Nq, Nkv, N, page, I, RP;  // RP = padded max rank
    float softmax_scale;
};

}  // namespace alora

namespace alora { struct BatchArgs; }

struct alora_ctx {
    alora_config cfg;
    alora::Dims d;
    size_t esize = 2;
    std::vector<alora::LayerWeights> layers;
    std::vector<alora::AdapterDev> h_adapters;  // [layer * max_adapters + id], mirrors d_adapters
    int largest_rank = 0;                        // of all registered adapters, on any layer
    alora::AdapterDev *d_adapters = nullptr;
    std::vector<void *> adapter_storage;         // context-owned A/B buffers, same indexing, 2 per entry

    // bf16 tensor-core path: per-layer adapter storage shared by all adapters of the layer
    std::vector<void *> tc_a_all, tc_b_all;          // [layer] -> [max_adapters][3*64][H], [max_adapters][N][64]
    std::vector<alora::TcLayerMaps> tc_maps;         // [layer]
    std::vector<char> layer_has_adapter;             // [layer] any adapter registered
    // adapters on the MLP block (bf16), allocated when the first one is registered on a layer: the A rows of all
    // adapters as one weight matrix per projection pair, the B rows per adapter
    std::vector<void *> mlp_a_gu, mlp_b_gu;          // [layer] -> [max_adapters][2][RP][H], [max_adapters][2 I][RP]
    std::vector<void *> mlp_a_dn, mlp_b_dn;          // [layer] -> [max_adapters][RP][I] (rows padded to 128), [max_adapters][H][RP]
    std::vector<int> mlp_n_adapters;                 // [layer] highest registered MLP adapter id + 1
    std::vector<alora::MlpAdapterDev> h_mlp_adapters;   // [layer * max_adapters + id], mirrors d_mlp_adapters
    alora::MlpAdapterDev *d_mlp_adapters = nullptr;
    void *d_mlp_t = nullptr;                         // t of the MLP adapters: [max_pairs][128][2 * RP], [max_quads][512][2 * RP], or
                                                     // (few-row route) [kFewRowMax][max_adapters * 2 * RP]
    float *d_mlp_part = nullptr;                     // K-slice partials of the shrink kernel
    size_t mlp_part_floats = 0;
    int32_t *d_mlp_done = nullptr;                   // per 64 x 64 tile of the shrink result: slices stored (zero between launches)
    int mlp_done_ints = 0;

    // per-call workspaces
    int32_t *d_token_req = nullptr, *d_row_adapter = nullptr, *d_slot = nullptr;
    alora::TilePair *d_pairs = nullptr;       // [max_pairs] (row tile, adapter) pairs of the batch, tile after tile
    int32_t *d_pair_off = nullptr;            // [row tiles + 1] first pair of each row tile
    alora::TilePair *d_quads = nullptr;       // [max_quads] (quad, adapter) entries of the batch (bf16), quad after quad
    int32_t *d_quad_off = nullptr;            // [quads + 1] first entry of each quad
    int32_t *d_quad_ready = nullptr;          // [max_quads] per entry: epilogue warps that have published t (zero between launches)
    int32_t max_quads = 0;
    int32_t *d_counts = nullptr;  // [1] attention work items, [2] (row tile, adapter) pairs,
                                  // [3] few-row attention items, [4] next unclaimed few-row item,
                                  // [6] key tiles of the attention items that are cut into runs, [7] tiles per run,
                                  // [8] attention items taken whole (the first ones), [9] key tiles of those,
                                  // [10], [11] next unclaimed projection item and blocks done, [12] few-row attention blocks done,
                                  // [13] an adapter with a non-finite B has been registered (kOddAdapters),
                                  // [15], [16] tensor-core attention items claimed (even, odd layers)
    int32_t *d_seg_scratch = nullptr;  // [14*max_requests+5] per-request values and merged row runs of the current batch
    int32_t *d_t_ready = nullptr;      // [max_pairs] per pair: epilogue warps that have published t (zero between launches)
    int32_t *d_iota = nullptr;         // 0..max_requests: query_start_loc of a decode batch
    int32_t max_pairs = 0;
    int t_slots = 0;                   // 128-row slots of d_t (bf16)
    alora::AttnWork *d_attn_items = nullptr;  // tensor-core attention work list (bf16)
    int32_t *d_attn_off = nullptr;            // [max_requests+1] block offsets per request
    int32_t max_attn_items = 0, attn_q_block = 0;
    // long batches: the tensor-core attention kernel takes some items whole and cuts the key tiles of the rest into runs
    int32_t *d_attn_cta_start = nullptr;      // [n_sm] first item of each block's run
    float *d_attn_part_o = nullptr;           // [2 * n_sm][hd][256] unnormalised outputs of the parts of cut items
    float *d_attn_part_ml = nullptr;          // [2 * n_sm][2][256] their exponent references and row sums
    // few-row attention (requests with at most small_max_tokens new tokens): split-KV work list and partials
    alora::AttnSplitWork *d_split_items = nullptr;
    int32_t *d_req_scratch = nullptr;   // [kSplitScratch][max_requests] per-request values of the few-row list's builder
    int32_t *d_prefix_groups = nullptr; // [2][max_requests] per request of the last batch: first request of its prefix
                                        // group, keys the group shares (0: ungrouped)
    float *d_part_o = nullptr, *d_part_ml = nullptr;
    int32_t *d_group_done = nullptr;    // [max_split_rows / 16] finished key ranges per (stream, KV head), at its first partial row / 16
    int32_t max_split_items = 0, max_split_rows = 0, small_max_tokens = 0;
    void *d_t = nullptr;          // rank-r intermediate: fp32 [max_tokens][3][RP]; bf16 [pair][1 or 3 summands][128][3][RP], or
                                  // [(quad, adapter) entry][1 or 3 summands][512][3][RP]
    // few-row projection (batches of <= 128 rows): K-slice partial products and partial shrink results
    float *d_skinny_part = nullptr;   // [skinny_max_items][128][256] fp32
    float *d_skinny_t = nullptr;      // [slices of the q/k/v projection][128][skinny_p_cap][192] fp32
    alora::FewRowMeta *d_skinny_meta = nullptr;   // [n_layers][few_tiles] of the current batch
    int few_tiles = 1;
    const alora::BatchArgs *pending_attn_meta = nullptr;   // run_layer: attention lists still to be built for this batch
    int skinny_max_items = 0, skinny_p_cap = 0;
    bool x_before_facts = false;   // the projection's input was complete before the batch-facts launch that precedes it
    void *d_qkv = nullptr;        // [max_tokens][N]
    void *d_act[4] = {nullptr, nullptr, nullptr, nullptr};  // stack activations
    double *d_rope_inv_freq = nullptr;   // [hd / 2] theta^(-2i/hd), only with a rotary base configured
    int32_t *d_status = nullptr;
    int32_t *h_status = nullptr;  // pinned

    bool profiling = false;
    std::vector<alora::ProfEvent> prof_events;  // event pairs recorded since profiling was enabled
    size_t prof_used = 0;
    int64_t launches = 0;
    std::string cuda_err;
    int sm_count = 148;
    int few_clusters[9] = {};   // [size] clusters of the few-row projection that fit on the device at once (0: route closed)
};

namespace alora {

// Records a CUDA failure in the context and maps it to ALORA_ERR_CUDA.
alora_status cuda_fail(alora_ctx *ctx, cudaError_t e, const char *what);

#define ALORA_CUDA(ctx, call)                                              \
    do {                                                                   \
        cudaError_t e__ = (call);                                          \
        if (e__ != cudaSuccess) return ::alora::cuda_fail(ctx, e__, #call); \
    } while (0)

// Brackets the launches of one kernel family with CUDA events while profiling is on.
// Kernel launch with the programmatic-stream-serialization attribute (`dependent`: the kernel calls
// tc::grid_dep_wait() before it touches anything its predecessor in the stream wrote or still reads).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                 bool dependent, Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

struct ProfScope {
    alora_ctx *ctx;
    cudaStream_t s;
    cudaEvent_t end = nullptr;
    ProfScope(alora_ctx *c, int kind, cudaStream_t st) : ctx(c), s(st) {
        if (!c->profiling) return;
        if (c->prof_used == c->prof_events.size()) {
            ProfEvent e{nullptr, nullptr, kind};
            if (cudaEventCreate(&e.begin) != cudaSuccess || cudaEventCreate(&e.end) != cudaSuccess) return;
            c->prof_events.push_back(e);
        }
        ProfEvent &e = c->prof_events[c->prof_used++];
        e.kind = kind;
        cudaEventRecord(e.begin, st);
        end = e.end;
    }
    ~ProfScope() { if (end) cudaEventRecord(end, s); }
};

// ---- launchers implemented in the kernel files (each returns the number of kernels launched or <0) ----
struct BatchArgs {
    const int32_t *positions, *activation_offsets, *adapter_ids, *query_start_loc, *seq_lens, *block_tables;
    int max_blocks, num_pages, T, R, mode;
    int all_small;  // host-side knowledge that no request has more than small_max_tokens new tokens (decode)
    int layer = -1; // layer whose adapter table the gate is checked against (-1: no check)
    int few_row = 0; // the projection of this batch takes the few-row route: build FewRowMeta instead of row tiles
    int n_layers = 1; // layers from `layer` on that the projection's facts are built for (a stack call: all of them at once)
    int facts_ready = 0; // bits (kMetaProjection, kMetaAttention): built by an earlier layer of the same stack call
    bool own_facts = false;    // no metadata step in front of the fp32 attention: it reads the caller's arrays itself
    bool lists_shared = false; // the attention lists built for this layer serve other layers of the call too
};

// phases: bit 0 = per-token arrays and the projection's lists, bit 1 = the attention work lists.  A launch of
// the attention lists alone is a programmatic dependent launch: it may run beside the projection kernel that
// precedes it in the stream.  `timed`: bracket it with profiling events of the metadata family.
constexpr int kMetaProjection = 1, kMetaAttention = 2;
constexpr int kOddAdapters = 13;   // index into d_counts
void few_cluster_init(alora_ctx *ctx);   // gemm_few_cluster.cu: what that route needs to know about the device
int launch_metadata(alora_ctx *ctx, const BatchArgs &b, cudaStream_t s, int phases = kMetaProjection | kMetaAttention,
                    bool timed = true);
int launch_repack_adapter(alora_ctx *ctx, int rank, const void *Aq, const void *Bq, const void *Ak,
                          const void *Bk, const void *Av, const void *Bv, void *A_dst, void *B_dst,
                          int32_t *b_odd, cudaStream_t s);
int launch_project(alora_ctx *ctx, int layer, const void *hidden, int T, int R, void *qkv, cudaStream_t s, void *kv_pool,
                   int num_pages, bool *kv_appended);
// Most (row tile, adapter) pairs that a batch of T rows and R requests can have.
inline int pair_bound(const alora_ctx *ctx, int T, int R) {
    const long long n_m = (T + kTileRows - 1) / kTileRows, na = ctx->cfg.max_adapters > 0 ? ctx->cfg.max_adapters : 1;
    long long n = n_m + R;
    if (n > T) n = T;
    if (n > n_m * na) n = n_m * na;
    return (int)n;
}
// Most (quad, adapter) entries.
inline int quad_bound(const alora_ctx *ctx, int T, int R) {
    const long long n_q = (T + kQuadRows - 1) / kQuadRows, na = ctx->cfg.max_adapters > 0 ? ctx->cfg.max_adapters : 1;
    long long n = n_q + R;
    if (n > T) n = T;
    if (n > n_q * na) n = n_q * na;
    return (int)n;
}
int launch_kv_append(alora_ctx *ctx, const void *qkv, int T, int num_pages, void *pool, cudaStream_t s);
int launch_cow_tail_pages(alora_ctx *ctx, const int32_t *qsl, const int32_t *seq_lens, int32_t *block_tables, int max_blocks,
                          int num_pages, int R, const int32_t *fresh_pages, void *pool, cudaStream_t s);
int launch_rope(alora_ctx *ctx, void *qkv, const int32_t *positions, int T, void *pool, int num_pages, cudaStream_t s);
int launch_attend(alora_ctx *ctx, const void *qkv, const BatchArgs &b, const void *pool, void *out,
                  cudaStream_t s);
// A gated low-rank delta on a dense projection (adapters on the MLP block): the A and B slabs of all adapters of the layer
// (64 padded rank columns per adapted matrix, n_blk matrices side by side in the output row), the layer's table, the
// batch's row tile of the projection's first row, the applied adapter of its rows, room for t ([max_pairs][128][64 n_blk]).
struct LinearDelta {
    const void *A, *B;
    int n_blk;
    const MlpAdapterDev *table;
    int tile0;
    const int32_t *row_adapter;
    void *t;
};
int launch_linear(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y,
                  const void *residual, cudaStream_t s, const LinearDelta *delta = nullptr);
// y = silu(x Wg^T) * (x Wu^T), W = [Wg; Wu], in one launch; 0: not for this shape (nothing launched).
int launch_glu(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y, cudaStream_t s, const LinearDelta *delta);
int launch_rmsnorm(alora_ctx *ctx, const void *x, const void *w, int T, void *y, cudaStream_t s);
int launch_swiglu(alora_ctx *ctx, const void *gate_up, int T, void *y, cudaStream_t s);

// device-side status recording: first finding wins
__device__ __forceinline__ void report(int32_t *status, int code) { atomicCAS(status, 0, code); }

}  // namespace alora
