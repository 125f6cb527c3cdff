// CUDA-core kernels: the fp32 data type's projection and attention (tiny exact-precision
// configurations), and the element-wise / copy steps shared by both data types (adapter repack,
// KV append, RMSNorm, SwiGLU).
#include "alora_internal.h"
#include "tc_common.cuh"

namespace alora {

template <typename T> __device__ __forceinline__ float ldf(const T *p);
template <> __device__ __forceinline__ float ldf<float>(const float *p) { return *p; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void stf(T *p, float v);
template <> __device__ __forceinline__ void stf<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// Adapter repack: A_dst[3][RP][H] <- (Aq, Ak, Av)[r][H] with zero rows r..RP-1;
// B_dst[N][RP] <- rows of (Bq | Bk | Bv)[.][r] with zero columns r..RP-1.  An Inf or NaN among the B values sets *b_odd (the
// adapter's record, written before this launch) and *any_odd.
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void repack_adapter_kernel(const T *Aq, const T *Ak, const T *Av, const T *Bq, const T *Bk,
                                      const T *Bv, int rank, int RP, int H, int Nq, int Nkv, T *A_dst,
                                      T *B_dst, int32_t *b_odd, int32_t *any_odd) {
    const size_t nA = (size_t)3 * RP * H, nB = (size_t)(Nq + 2 * Nkv) * RP;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nA + nB;
         i += (size_t)gridDim.x * blockDim.x) {
        if (i < nA) {
            int blk = (int)(i / ((size_t)RP * H));
            int row = (int)((i / H) % RP), h = (int)(i % H);
            const T *src = blk == 0 ? Aq : (blk == 1 ? Ak : Av);
            A_dst[i] = row < rank ? src[(size_t)row * H + h] : T(0.f);
        } else {
            size_t j = i - nA;
            int n = (int)(j / RP), c = (int)(j % RP);
            T v = T(0.f);
            if (c < rank) {
                if (n < Nq) v = Bq[(size_t)n * rank + c];
                else if (n < Nq + Nkv) v = Bk[(size_t)(n - Nq) * rank + c];
                else v = Bv[(size_t)(n - Nq - Nkv) * rank + c];
                if (!isfinite(ldf(&v))) { *b_odd = 1; *any_odd = 1; }
            }
            B_dst[j] = v;
        }
    }
}

int launch_repack_adapter(alora_ctx *ctx, int rank, const void *Aq, const void *Bq, const void *Ak,
                          const void *Bk, const void *Av, const void *Bv, void *A_dst, void *B_dst,
                          int32_t *b_odd, cudaStream_t s) {
    const Dims &d = ctx->d;
    int32_t *any_odd = ctx->d_counts + kOddAdapters;
    if (ctx->cfg.dtype == ALORA_DTYPE_FP32)
        repack_adapter_kernel<float><<<256, 256, 0, s>>>((const float *)Aq, (const float *)Ak, (const float *)Av,
                                                         (const float *)Bq, (const float *)Bk, (const float *)Bv,
                                                         rank, d.RP, d.H, d.Nq, d.Nkv, (float *)A_dst, (float *)B_dst,
                                                         b_odd, any_odd);
    else
        repack_adapter_kernel<__nv_bfloat16><<<256, 256, 0, s>>>(
            (const __nv_bfloat16 *)Aq, (const __nv_bfloat16 *)Ak, (const __nv_bfloat16 *)Av,
            (const __nv_bfloat16 *)Bq, (const __nv_bfloat16 *)Bk, (const __nv_bfloat16 *)Bv, rank, d.RP, d.H,
            d.Nq, d.Nkv, (__nv_bfloat16 *)A_dst, (__nv_bfloat16 *)B_dst, b_odd, any_odd);
    return 1;
}

// ---------------------------------------------------------------------------------------------
// CUDA-core shrink (fp32): t[row][blk][i] = scale * sum_h A[blk][i][h] x[row][h] for rows with an applied
// adapter (Eq. 5, inner product of the low-rank delta).  One block per (row, q/k/v block), one warp per output.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
shrink_simt_kernel(const float *__restrict__ x, const int32_t *__restrict__ row_adapter, const AdapterDev *__restrict__ adapters,
                   int H, int RP, float *__restrict__ t) {
    tc::grid_dep_launch();
    const int row = blockIdx.x, blk = blockIdx.y;
    const int k = row_adapter[row];
    if (k < 0) return;
    const AdapterDev ad = adapters[k];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float4 *xv = reinterpret_cast<const float4 *>(x + (size_t)row * H);
    for (int i = warp; i < RP; i += 8) {
        float acc = 0.f;
        if (i < ad.rank) {
            const float4 *av = reinterpret_cast<const float4 *>((const float *)ad.A + (size_t)(blk * RP + i) * H);
#pragma unroll 4
            for (int h = lane; h < H / 4; h += 32) {
                const float4 a = av[h], b = xv[h];
                acc += a.x * b.x; acc += a.y * b.y; acc += a.z * b.z; acc += a.w * b.w;
            }
            for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        }
        if (lane == 0) t[((size_t)row * 3 + blk) * RP + i] = acc * ad.scale;
    }
}

// ---------------------------------------------------------------------------------------------
// CUDA-core projection (fp32) y[row][n] = sum_h W[n][h] x[row][h]  (+ sum_i B[n][i] t[row][blk(n)][i] when the
// row has an applied adapter).  The sizes that run here (the exact-precision layers of the tests: 16 rows, K 256, N 512) are
// bound by latency: 32 tiles of 64 x 64 walked K through shared memory in 16 steps on 8 SMs and took 35 us.  So tiles are
// 16 x 32 and the 8 warps of a block share K (warp w takes every eighth vector of four), each straight from global
// memory, the loads of two steps in flight; their sums are added in warp order: 10 us.  The split of K does not
// depend on the row count and the base sum of a row is formed by the same instruction sequence whether or not the
// delta follows, so gated-off rows equal a base-only call bit for bit.  Optional residual: y += residual[row][n]
// (used by o_proj / down_proj); with a page pool the k and v columns also go to the rows' cache slots.
// `base_first`: x was complete before the preceding kernel of the stream began, so that the base sums do not wait for it.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
linear_simt_kernel(const float *__restrict__ x, const float *__restrict__ W, int Tn, int K, int N,
                   const int32_t *__restrict__ row_adapter, const AdapterDev *__restrict__ adapters,
                   const float *__restrict__ t, int RP, int Nq, int Nkv, const float *residual /* may alias y */, float *y,
                   float *__restrict__ pool, const int32_t *__restrict__ slot_map, int hd, int Hkv, int page_size,
                   int num_pages, int base_first, int32_t *status) {
    __shared__ float part[8][16][32 + 1];
    tc::grid_dep_launch();
    if (!base_first) tc::grid_dep_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tx = lane & 7, ty = lane >> 3;
    const int n_col = (N + 31) / 32, row0 = (int)blockIdx.x / n_col * 16, col0 = (int)blockIdx.x % n_col * 32;   // (any number of rows)
    float acc[4][4] = {};   // rows row0 + ty + 4 i, columns col0 + tx + 8 j (beyond the edge: the last one again, not stored)
    const float *xr[4], *wr[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        xr[i] = x + (size_t)min(row0 + ty + 4 * i, Tn - 1) * K;
        wr[i] = W + (size_t)min(col0 + tx + 8 * i, N - 1) * K;
    }
    auto step = [&](const float4 (&a)[4], const float4 (&b)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[i][j] += a[i].x * b[j].x; acc[i][j] += a[i].y * b[j].y;
                acc[i][j] += a[i].z * b[j].z; acc[i][j] += a[i].w * b[j].w;
            }
    };
    if (K % 4 == 0) {
#pragma unroll 2
        for (int k = warp * 4; k < K; k += 32) {
            float4 a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { a[i] = *reinterpret_cast<const float4 *>(xr[i] + k); b[i] = *reinterpret_cast<const float4 *>(wr[i] + k); }
            step(a, b);
        }
    } else {
        for (int k = warp * 4; k < K; k += 32) {
            float4 a[4], b[4];
            auto four = [&](const float *r) {
                return make_float4(r[k], k + 1 < K ? r[k + 1] : 0.f, k + 2 < K ? r[k + 2] : 0.f, k + 3 < K ? r[k + 3] : 0.f);
            };
#pragma unroll
            for (int i = 0; i < 4; ++i) { a[i] = four(xr[i]); b[i] = four(wr[i]); }
            step(a, b);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) part[warp][ty + 4 * i][tx + 8 * j] = acc[i][j];
    __syncthreads();
    if (base_first) tc::grid_dep_wait();   // t
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = row0 + (int)(threadIdx.x >> 5) + 8 * h, n = col0 + lane;
        if (row >= Tn || n >= N) continue;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += part[w][row - row0][lane];
        const int k = row_adapter ? row_adapter[row] : -1;
        const int blk = n < Nq ? 0 : (n < Nq + Nkv ? 1 : 2);
        if (k >= 0) {
            const AdapterDev ad = adapters[k];
            const float *B = (const float *)ad.B + (size_t)n * RP;
            const float *tr = t + ((size_t)row * 3 + blk) * RP;
            float dlt = 0.f;
#pragma unroll 8
            for (int r = 0; r < ad.rank; ++r) dlt += B[r] * tr[r];
            v += dlt;
        }
        if (residual) v += residual[(size_t)row * N + n];
        y[(size_t)row * N + n] = v;
        if (pool != nullptr && blk > 0) {
            const int slot = slot_map[row];
            if (slot < 0) continue;
            const int page = slot / page_size;
            if (page >= num_pages) { report(status, ALORA_ERR_PAGE_RANGE); continue; }
            const int c = n - Nq - (blk - 1) * Nkv;
            pool[((((size_t)page * 2 + blk - 1) * Hkv + c / hd) * page_size + slot % page_size) * hd + c % hd] = v;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// What a new token's row needs to know, from the caller's arrays (the same findings as the batch-metadata step; a change there or
// here is one in both): request, position, applied adapter (the gate of Eq. 5; -1: none) and cache slot (-1: rejected).
// Called by whole warps.
// ---------------------------------------------------------------------------------------------
struct RowFacts { int req, pos, adapter, slot; };
__device__ __forceinline__ RowFacts row_facts(int t, const int32_t *__restrict__ positions, const int32_t *__restrict__ a_req,
                                              const int32_t *__restrict__ adapter_ids, const int32_t *__restrict__ qsl,
                                              const int32_t *__restrict__ seq_lens, const int32_t *__restrict__ block_tables,
                                              int max_blocks, int num_pages, int page_size, int max_adapters, int R, int mode, int32_t *status) {
    const int lane = threadIdx.x & 31;
    RowFacts f;
    f.pos = positions[t];
    int r = 0;   // the last request that starts at or before t (empty requests start where their successor does): 32 places a step
    for (int n = R; n > 1;) {   // among requests r .. r + n - 1; r itself starts at or before t
        const int step = (n + 31) >> 5, at = lane * step;
        const int before = __popc(__ballot_sync(0xffffffffu, at < n && (lane == 0 || qsl[r + at] <= t))) - 1;
        r += before * step;
        n = min(step, n - before * step);
    }
    f.req = r;
    const int len = seq_lens[r], next = qsl[r + 1], first_open = a_req != nullptr && mode == ALORA_MODE_ALORA ? a_req[r] : 0;
    int k = mode != ALORA_MODE_BASE && adapter_ids != nullptr ? adapter_ids[r] : -1;
    const bool ok = f.pos == len - (next - t) && f.pos >= 0;   // positions of a request are consecutive and end at seq_len - 1
    if (!ok) report(status, ALORA_ERR_BAD_BATCH);
    if (k >= max_adapters || k < -1) { report(status, ALORA_ERR_BAD_BATCH); k = -1; }
    f.adapter = ok && f.pos >= first_open ? k : -1;
    f.slot = -1;
    if (ok) {
        const int blk = f.pos / page_size, page = blk < max_blocks ? block_tables[(size_t)r * max_blocks + blk] : -1;
        if (blk >= max_blocks) report(status, ALORA_ERR_BAD_BATCH);
        else if (page < 0 || page >= num_pages) report(status, ALORA_ERR_PAGE_RANGE);
        else f.slot = page * page_size + f.pos % page_size;
    }
    return f;
}

// ---------------------------------------------------------------------------------------------
// The first half of a small fp32 layer call in one launch: facts, shrink, projection, KV append.  Warps 0..7 form the base sums of
// a 16 x 32 tile as linear_simt_kernel does; beside them warp 8 + i finds row i's facts, its t = s A x and its delta
// for the tile's 32 columns, which lie in one of the q / k / v blocks (a column a lane).  Batch metadata, shrink and projection
// as launches of their own are chains of two to four fetches each, one after the other: 16 tokens at hidden 256 took 17 us
// until the projection was done, of 22 for the call; here the chains run side by side (call: 13 us).  t is formed again
// by every column tile, so this is for few rows and short rows of x (simt_small_layer()).  80 registers at 768 threads, one block an
// SM; 80 bytes are spilled around the batch facts.
// ---------------------------------------------------------------------------------------------
constexpr int kSmallVecs = 8;   // 16-byte vectors of x a lane holds: hidden <= 1024
__global__ void __launch_bounds__(768)
project_small_simt_kernel(const float *__restrict__ x, const float *__restrict__ W, int Tn, int K, int N, int Nq, int Nkv, int RP,
                          const AdapterDev *__restrict__ adapters, const int32_t *__restrict__ positions,
                          const int32_t *__restrict__ a_req, const int32_t *__restrict__ adapter_ids, const int32_t *__restrict__ qsl,
                          const int32_t *__restrict__ seq_lens, const int32_t *__restrict__ block_tables, int max_blocks, int num_pages,
                          int page_size, int max_adapters, int R, int mode, int hd, int Hkv, float *__restrict__ pool,
                          int32_t *__restrict__ token_req, int32_t *__restrict__ row_adapter, int32_t *__restrict__ slot_map,
                          float *__restrict__ y, int32_t *status) {
    __shared__ float part[8][16][32 + 1], delta_s[16][32 + 1];
    __shared__ int adapter_s[16], slot_s[16];
    tc::grid_dep_wait();     // (in this order: the attention kernel relies on it for what it reads before its own wait)
    tc::grid_dep_launch();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_col = (N + 31) / 32, row0 = (int)blockIdx.x / n_col * 16, col0 = (int)blockIdx.x % n_col * 32;
    if (warp < 8) {
        const int tx = lane & 7, ty = lane >> 3;
        float acc[4][4] = {};   // rows row0 + ty + 4 i, columns col0 + tx + 8 j (beyond the edge: the last one again, not stored)
        const float *xr[4], *wr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            xr[i] = x + (size_t)min(row0 + ty + 4 * i, Tn - 1) * K;
            wr[i] = W + (size_t)min(col0 + tx + 8 * i, N - 1) * K;
        }
#pragma unroll 2
        for (int k = warp * 4; k < K; k += 32) {
            float4 a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { a[i] = *reinterpret_cast<const float4 *>(xr[i] + k); b[i] = *reinterpret_cast<const float4 *>(wr[i] + k); }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] += a[i].x * b[j].x; acc[i][j] += a[i].y * b[j].y;
                    acc[i][j] += a[i].z * b[j].z; acc[i][j] += a[i].w * b[j].w;
                }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) part[warp][ty + 4 * i][tx + 8 * j] = acc[i][j];
    } else if (const int row = row0 + warp - 8; row < Tn) {
        const int i_row = warp - 8, blk = col0 < Nq ? 0 : (col0 < Nq + Nkv ? 1 : 2);
        float4 xv[kSmallVecs];
#pragma unroll
        for (int v = 0; v < kSmallVecs; ++v)
            xv[v] = (lane + 32 * v) * 4 < K ? reinterpret_cast<const float4 *>(x + (size_t)row * K)[lane + 32 * v] : make_float4(0.f, 0.f, 0.f, 0.f);
        const RowFacts f = row_facts(row, positions, a_req, adapter_ids, qsl, seq_lens, block_tables, max_blocks, num_pages, page_size,
                                     max_adapters, R, mode, status);
        float dlt = 0.f;
        if (f.adapter >= 0) {
            const AdapterDev ad = adapters[f.adapter];
            if (ad.rank == 0) report(status, ALORA_ERR_NO_WEIGHTS);
            const float *A = (const float *)ad.A + (size_t)blk * RP * K, *B = (const float *)ad.B + (size_t)min(col0 + lane, N - 1) * RP;
            for (int i0 = 0; i0 < ad.rank; i0 += 8) {   // (rows and columns of the padding are zero; RP is a multiple of 16)
                float t[8];
                float4 b[2];
                b[0] = *reinterpret_cast<const float4 *>(B + i0); b[1] = *reinterpret_cast<const float4 *>(B + i0 + 4);
#pragma unroll
                for (int i = 0; i < 8; ++i) t[i] = 0.f;
#pragma unroll
                for (int v = 0; v < kSmallVecs; ++v) {
                    if (v * 128 >= K) break;
                    const bool in = (lane + 32 * v) * 4 < K;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 a = in ? reinterpret_cast<const float4 *>(A + (size_t)(i0 + i) * K)[lane + 32 * v] : make_float4(0.f, 0.f, 0.f, 0.f);
                        t[i] += a.x * xv[v].x; t[i] += a.y * xv[v].y; t[i] += a.z * xv[v].z; t[i] += a.w * xv[v].w;
                    }
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    for (int off = 16; off; off >>= 1) t[i] += __shfl_xor_sync(0xffffffffu, t[i], off);
                    t[i] *= ad.scale;
                }
                const float bb[8] = {b[0].x, b[0].y, b[0].z, b[0].w, b[1].x, b[1].y, b[1].z, b[1].w};
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i0 + i < ad.rank) dlt += bb[i] * t[i];
            }
        }
        delta_s[i_row][lane] = dlt;
        if (lane == 0) {
            adapter_s[i_row] = f.adapter; slot_s[i_row] = f.slot;
            if (col0 == 0) { token_req[row] = f.req; row_adapter[row] = f.adapter; slot_map[row] = f.slot; }
        }
    }
    __syncthreads();
    const int row = row0 + warp, n = col0 + lane;
    if (warp >= 16 || row >= Tn || n >= N) return;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += part[w][warp][lane];
    if (adapter_s[warp] >= 0) v += delta_s[warp][lane];
    y[(size_t)row * N + n] = v;
    const int slot = slot_s[warp];
    if (pool == nullptr || n < Nq || slot < 0) return;
    const int plane = n < Nq + Nkv ? 0 : 1, c = n - Nq - plane * Nkv;
    pool[((((size_t)(slot / page_size) * 2 + plane) * Hkv + c / hd) * page_size + slot % page_size) * hd + c % hd] = v;
}

// ---------------------------------------------------------------------------------------------
// KV append (both data types): one 16-byte vector per thread.  Row t's k part
// qkv[t][Nq .. Nq+Nkv) goes to pool[page][0][head][row][:], its v part to plane 1.  Tokens whose
// slot is -1 (rejected by the metadata step) are skipped.
// ---------------------------------------------------------------------------------------------
__global__ void kv_append_kernel(const uint4 *__restrict__ qkv, const int32_t *__restrict__ slot_map,
                                 int T, int N_vec, int Nq_vec, int Nkv_vec, int hd_vec, int Hkv,
                                 int page_size, int num_pages, uint4 *__restrict__ pool, int32_t *status) {
    const size_t total = (size_t)T * 2 * Nkv_vec;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int t = (int)(i / (2 * Nkv_vec));
        const int c = (int)(i % (2 * Nkv_vec));   // vector column inside [k | v]
        const int plane = c / Nkv_vec, cc = c % Nkv_vec;
        const int head = cc / hd_vec, dv = cc % hd_vec;
        const int slot = slot_map[t];
        if (slot < 0) continue;
        const int page = slot / page_size, row = slot % page_size;
        if (page >= num_pages) { report(status, ALORA_ERR_PAGE_RANGE); continue; }
        const size_t dst = ((((size_t)page * 2 + plane) * Hkv + head) * page_size + row) * hd_vec + dv;
        pool[dst] = qkv[(size_t)t * N_vec + Nq_vec + c];
    }
}

int launch_kv_append(alora_ctx *ctx, const void *qkv, int T, int num_pages, void *pool, cudaStream_t s) {
    if (T == 0) return 0;
    const Dims &d = ctx->d;
    ProfScope prof(ctx, KK_KV_APPEND, s);
    const int vec = 16 / (int)ctx->esize;  // elements per 16-byte vector
    const size_t total = (size_t)T * 2 * (d.Nkv / vec);
    int blocks = (int)((total + 255) / 256);
    if (blocks > ctx->sm_count * 16) blocks = ctx->sm_count * 16;
    kv_append_kernel<<<blocks, 256, 0, s>>>((const uint4 *)qkv, ctx->d_slot, T, d.N / vec, d.Nq / vec,
                                            d.Nkv / vec, d.hd / vec, d.Hkv, d.page, num_pages, (uint4 *)pool,
                                            ctx->d_status);
    return 1;
}

// ---------------------------------------------------------------------------------------------
// Optional rotary position embedding fused with the KV append (both data types).  The paper's equations carry no
// positional rotation; with a base theta configured, the new query and key rows are rotated by their positions
// ("rotate-half": column i of a head pairs with column i + hd/2, angle p * theta^(-2i/hd)) after the projection and
// before the keys are cached, so the cache holds post-rotation keys.  One thread per (token, head, 16-byte vector
// of pair indices): it rotates the pairs in place in the fused q/k/v row and, for key heads, also writes the rotated
// vectors to the token's cache slot; a second index range copies the value rows to the cache.  The angle is formed
// and reduced to [-pi, pi] in double precision (positions reach tens of thousands of radians), the sine and
// cosine of the remainder in single.  Without a pool only the in-place rotation happens.
// ---------------------------------------------------------------------------------------------
template <typename T> struct Vec16;
template <> struct Vec16<float> { static constexpr int kElems = 4; };
template <> struct Vec16<__nv_bfloat16> { static constexpr int kElems = 8; };

__device__ __forceinline__ void unpack16(const uint4 &u, float (&f)[4]) {
    f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y); f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
}
__device__ __forceinline__ void unpack16(const uint4 &u, float (&f)[8]) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 b2 = *reinterpret_cast<const __nv_bfloat162 *>(&w[e]);
        f[2 * e] = __low2float(b2); f[2 * e + 1] = __high2float(b2);
    }
}
__device__ __forceinline__ uint4 pack16(const float (&f)[4]) {
    return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
}
__device__ __forceinline__ uint4 pack16(const float (&f)[8]) {
    uint4 u;
    __nv_bfloat162 v;
    v = __floats2bfloat162_rn(f[0], f[1]); u.x = *reinterpret_cast<uint32_t *>(&v);
    v = __floats2bfloat162_rn(f[2], f[3]); u.y = *reinterpret_cast<uint32_t *>(&v);
    v = __floats2bfloat162_rn(f[4], f[5]); u.z = *reinterpret_cast<uint32_t *>(&v);
    v = __floats2bfloat162_rn(f[6], f[7]); u.w = *reinterpret_cast<uint32_t *>(&v);
    return u;
}

template <typename T>
__global__ void rope_append_kernel(uint4 *__restrict__ qkv, const int32_t *__restrict__ positions,
                                   const int32_t *__restrict__ slot_map, const double *__restrict__ inv_freq, int Tn,
                                   int N_vec, int n_rot_heads, int n_q_heads, int hd_vec, int Hkv, int page_size,
                                   int num_pages, uint4 *__restrict__ pool, int32_t *status) {
    constexpr int kE = Vec16<T>::kElems;
    const int half_vec = hd_vec / 2;                       // vectors per half head
    const int rot_units = n_rot_heads * half_vec;          // per token: (head, vector of pair indices)
    const int copy_units = pool != nullptr ? Hkv * hd_vec : 0;   // per token: vectors of the value row
    const int per_tok = rot_units + copy_units;
    const size_t total = (size_t)Tn * per_tok;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
        const int t = (int)(idx / per_tok), u = (int)(idx % per_tok);
        int page = -1, prow = 0;
        if (pool != nullptr) {
            const int slot = slot_map[t];
            if (slot >= 0) {
                page = slot / page_size; prow = slot % page_size;
                if (page >= num_pages) { report(status, ALORA_ERR_PAGE_RANGE); page = -1; }
            }
        }
        uint4 *row = qkv + (size_t)t * N_vec;
        if (u < rot_units) {
            const int h = u / half_vec, iv = u % half_vec;   // heads 0 .. n_q_heads-1 are queries, the rest keys
            uint4 *lo_p = row + (size_t)h * hd_vec + iv, *hi_p = lo_p + half_vec;
            float lo[kE], hi[kE];
            unpack16(*lo_p, lo); unpack16(*hi_p, hi);
            const double p = (double)positions[t];
#pragma unroll
            for (int e = 0; e < kE; ++e) {
                const double a = p * inv_freq[iv * kE + e];
                const float r = (float)(a - 6.283185307179586476925 * rint(a * 0.15915494309189533577));
                float sn, cs;
                sincosf(r, &sn, &cs);
                const float x0 = lo[e], x1 = hi[e];
                lo[e] = x0 * cs - x1 * sn;
                hi[e] = x1 * cs + x0 * sn;
            }
            const uint4 lo_u = pack16(lo), hi_u = pack16(hi);
            *lo_p = lo_u; *hi_p = hi_u;
            if (h >= n_q_heads && page >= 0) {   // a key head: the rotated vectors also go to the cache slot
                const int kh = h - n_q_heads;
                uint4 *dst = pool + ((((size_t)page * 2 + 0) * Hkv + kh) * page_size + prow) * hd_vec + iv;
                dst[0] = lo_u; dst[half_vec] = hi_u;
            }
        } else if (page >= 0) {
            const int c = u - rot_units, kh = c / hd_vec, dv = c % hd_vec;
            pool[((((size_t)page * 2 + 1) * Hkv + kh) * page_size + prow) * hd_vec + dv] =
                row[(size_t)(n_rot_heads + kh) * hd_vec + dv];
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Copy-on-write of a shared partial tail page.  Requests that reuse one base-model cache point at the same physical
// pages; when the reused length is not a multiple of the page size, the page that holds the last cached positions
// would also receive the request's first new rows.  Before the layer call, every such request gets a page of its
// own: rows 0 .. (first new position % page_size) - 1 of the shared page are copied to the fresh page (both planes,
// all KV heads) and the request's block-table entry is redirected.  One block per request.
// ---------------------------------------------------------------------------------------------
__global__ void cow_tail_pages_kernel(const int32_t *__restrict__ qsl, const int32_t *__restrict__ seq_lens,
                                      int32_t *__restrict__ block_tables, int max_blocks, int num_pages, int page_size,
                                      int Hkv, int hd_vec, const int32_t *__restrict__ fresh_pages,
                                      uint4 *__restrict__ pool, int32_t *status) {
    const int r = blockIdx.x;
    const int fresh = fresh_pages[r];
    if (fresh < 0) return;
    const int n_new = qsl[r + 1] - qsl[r];
    const int p_first = seq_lens[r] - n_new;
    const int blk = p_first / page_size, rows = p_first % page_size;
    if (n_new <= 0 || p_first < 0 || blk >= max_blocks) { if (threadIdx.x == 0) report(status, ALORA_ERR_BAD_BATCH); return; }
    const int old = block_tables[(size_t)r * max_blocks + blk];
    if (fresh >= num_pages || old < 0 || old >= num_pages) { if (threadIdx.x == 0) report(status, ALORA_ERR_PAGE_RANGE); return; }
    const int per_head = rows * hd_vec, total = 2 * Hkv * per_head;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int ph = i / per_head, v = i % per_head;    // (plane, head), vector inside the head's first `rows` rows
        const size_t off = (size_t)ph * page_size * hd_vec + v;
        pool[(size_t)fresh * 2 * Hkv * page_size * hd_vec + off] = pool[(size_t)old * 2 * Hkv * page_size * hd_vec + off];
    }
    __syncthreads();
    if (threadIdx.x == 0) block_tables[(size_t)r * max_blocks + blk] = fresh;
}

int launch_cow_tail_pages(alora_ctx *ctx, const int32_t *qsl, const int32_t *seq_lens, int32_t *block_tables, int max_blocks,
                          int num_pages, int R, const int32_t *fresh_pages, void *pool, cudaStream_t s) {
    if (R == 0) return 0;
    const Dims &d = ctx->d;
    const int vec = 16 / (int)ctx->esize;
    cow_tail_pages_kernel<<<R, 256, 0, s>>>(qsl, seq_lens, block_tables, max_blocks, num_pages, d.page, d.Hkv, d.hd / vec,
                                            fresh_pages, (uint4 *)pool, ctx->d_status);
    return 1;
}

// Rotates the query and key parts of qkv[T][N] in place; with a pool also appends the (rotated) keys and the values.
int launch_rope(alora_ctx *ctx, void *qkv, const int32_t *positions, int T, void *pool, int num_pages, cudaStream_t s) {
    if (T == 0) return 0;
    const Dims &d = ctx->d;
    if (ctx->d_rope_inv_freq == nullptr) return -1;
    const int vec = 16 / (int)ctx->esize;
    if (d.hd % (2 * vec) != 0) return -1;
    ProfScope prof(ctx, KK_KV_APPEND, s);
    const int hd_vec = d.hd / vec;
    const size_t per_tok = (size_t)(d.Hq + d.Hkv) * (hd_vec / 2) + (pool ? (size_t)d.Hkv * hd_vec : 0);
    const size_t total = (size_t)T * per_tok;
    int blocks = (int)std::min<size_t>((total + 255) / 256, (size_t)ctx->sm_count * 16);
    if (ctx->cfg.dtype == ALORA_DTYPE_FP32)
        rope_append_kernel<float><<<blocks, 256, 0, s>>>((uint4 *)qkv, positions, ctx->d_slot, ctx->d_rope_inv_freq, T,
                                                         d.N / vec, d.Hq + d.Hkv, d.Hq, hd_vec, d.Hkv, d.page, num_pages,
                                                         (uint4 *)pool, ctx->d_status);
    else
        rope_append_kernel<__nv_bfloat16><<<blocks, 256, 0, s>>>((uint4 *)qkv, positions, ctx->d_slot,
                                                                 ctx->d_rope_inv_freq, T, d.N / vec, d.Hq + d.Hkv, d.Hq,
                                                                 hd_vec, d.Hkv, d.page, num_pages, (uint4 *)pool,
                                                                 ctx->d_status);
    return 1;
}

// ---------------------------------------------------------------------------------------------
// CUDA-core attention (fp32; Eq. 1 / Eq. 3): a block per (token, KV head, HC of the query heads that share it).  Bound by the
// latency of a key's loads and sums at the lengths that run here: its 32 groups of 8 lanes are streams of their own, stream g
// taking keys g, g + 32, ... with its own running maximum and sum (online softmax), a lane an eighth of the head
// dimension, the keys and values of U of the stream's keys in flight; the streams are put together at the end.  (A warp per
// head that scored a key per lane, element by element, and went over the values one key after the other took 24 us for 16
// tokens on 64 cached ones, 27 with its launch: 4 us.)
// ---------------------------------------------------------------------------------------------
// kOwnFacts: the kernel finds its token's request and slot itself, beside the small layer's projection kernel in front of it; else they
// come from the metadata step.  (Where every block of every fp32 call looked for its request, 4096 one-token requests of 4 heads
// took 180 us instead of 90, 64 requests of 64 tokens 116 instead of 98.)
template <int HD, int HC, bool kOwnFacts>
__global__ void __launch_bounds__(256)
attn_simt_kernel(const float *__restrict__ qkv, const int32_t *__restrict__ token_req, const int32_t *__restrict__ slot_map,
                 const int32_t *__restrict__ positions, const int32_t *__restrict__ qsl,
                 const int32_t *__restrict__ seq_lens, const int32_t *__restrict__ block_tables, int max_blocks, int num_pages,
                 int page_size, int N, int Nq, int Hkv, int G, int R, float scale, const float *pool,
                 float *__restrict__ out, int32_t *status) {
    constexpr int V = HD / 32, U = HD == 128 ? 2 : 4;   // 16-byte vectors of a lane; keys of a stream in flight
    __shared__ float o_s[8][HC][HD], m_s[8][HC], l_s[8][HC];
    tc::grid_dep_launch();
    const int t = blockIdx.x, kvh = blockIdx.y, h0 = (int)blockIdx.z * HC, nh = min(HC, G - h0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, stream = warp * 4 + (lane >> 3), d0 = (lane & 7) * 4;
    // kOwnFacts: the caller's arrays were complete before the preceding kernel of the call let this one start: they are read beside it.  Rows
    // of the page pool are read after it, those before this request's new tokens too: another request of the call may have appended them.
    RowFacts f;
    if constexpr (kOwnFacts) {
        f = row_facts(t, positions, nullptr, nullptr, qsl, seq_lens, block_tables, max_blocks, num_pages, page_size, 0, R,
                      ALORA_MODE_BASE, status);
    } else {
        tc::grid_dep_wait();
        f.req = token_req[t]; f.pos = positions[t]; f.slot = slot_map[t];
    }
    const int r = f.req, p = f.pos;
    float *orow = out + (size_t)t * Nq + (size_t)(kvh * G + h0) * HD;
    if (f.slot < 0) {  // a token that the metadata step rejects: defined output, no cache access
        if (kOwnFacts) tc::grid_dep_wait();
        for (int d = threadIdx.x; d < nh * HD; d += 256) orow[d] = 0.f;
        return;
    }
    float4 q[HC][V], acc[HC][V];
    float m[HC], l[HC];
    const size_t plane = (size_t)Hkv * page_size * HD;
    const int32_t *table = block_tables + (size_t)r * max_blocks;
    int page[U];   // of the stream's next keys
    auto fetch_pages = [&](int j0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = j0 + 32 * u;
            page[u] = j <= p ? table[j / page_size] : -1;
            if (j <= p && (page[u] < 0 || page[u] >= num_pages)) report(status, ALORA_ERR_PAGE_RANGE);
        }
    };
    auto key_row = [&](int u, int j) { return pool + ((size_t)page[u] * 2 * Hkv + kvh) * page_size * HD + (size_t)(j % page_size) * HD; };
    fetch_pages(stream);
    if (kOwnFacts) {
#pragma unroll
        for (int u = 0; u < U; ++u)   // the first keys and values on their way to L2 (a lane a line of 32 elements)
            if (page[u] >= 0 && page[u] < num_pages && (lane & 7) < 2 * V)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(key_row(u, stream + 32 * u) + ((lane & 7) < V ? (lane & 7) * 32 : plane + ((lane & 7) - V) * 32)));
        tc::grid_dep_wait();
    }
#pragma unroll
    for (int c = 0; c < HC; ++c) {
        m[c] = -INFINITY; l[c] = 0.f;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const float4 a = *reinterpret_cast<const float4 *>(qkv + (size_t)t * N + (size_t)(kvh * G + min(h0 + c, G - 1)) * HD + d0 + 32 * v);
            q[c][v] = make_float4(a.x * scale, a.y * scale, a.z * scale, a.w * scale);
            acc[c][v] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    for (int j0 = stream; j0 - stream <= p; j0 += 32 * U) {
        float4 kv[U][V], vv[U][V];
        bool on[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            on[u] = page[u] >= 0 && page[u] < num_pages;
            const float *kr = on[u] ? key_row(u, j0 + 32 * u) + d0 : pool;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                kv[u][v] = on[u] ? *reinterpret_cast<const float4 *>(kr + 32 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
                vv[u][v] = on[u] ? *reinterpret_cast<const float4 *>(kr + plane + 32 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        fetch_pages(j0 + 32 * U);
#pragma unroll
        for (int c = 0; c < HC; ++c) {
            float s[U], mx = m[c];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float dot = 0.f;
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    dot += q[c][v].x * kv[u][v].x; dot += q[c][v].y * kv[u][v].y;
                    dot += q[c][v].z * kv[u][v].z; dot += q[c][v].w * kv[u][v].w;
                }
                for (int off = 1; off < 8; off <<= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
                s[u] = on[u] ? dot : -INFINITY;
                mx = fmaxf(mx, s[u]);
            }
            if (mx != -INFINITY) {   // (else nothing visible yet to this stream; its 8 lanes agree)
                const float corr = m[c] == -INFINITY ? 0.f : __expf(m[c] - mx);
                m[c] = mx; l[c] *= corr;
#pragma unroll
                for (int v = 0; v < V; ++v) { acc[c][v].x *= corr; acc[c][v].y *= corr; acc[c][v].z *= corr; acc[c][v].w *= corr; }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float w = on[u] ? __expf(s[u] - mx) : 0.f;
                    l[c] += w;
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        acc[c][v].x += w * vv[u][v].x; acc[c][v].y += w * vv[u][v].y;
                        acc[c][v].z += w * vv[u][v].z; acc[c][v].w += w * vv[u][v].w;
                    }
                }
            }
        }
    }
    __syncwarp();
    // the four streams of a warp, then the eight warps
#pragma unroll
    for (int c = 0; c < HC; ++c) {
        for (int off = 8; off < 32; off <<= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, m[c], off), l2 = __shfl_xor_sync(0xffffffffu, l[c], off);
            const float mx = fmaxf(m[c], m2);
            const float w1 = m[c] == -INFINITY ? 0.f : __expf(m[c] - mx), w2 = m2 == -INFINITY ? 0.f : __expf(m2 - mx);
            m[c] = mx; l[c] = l[c] * w1 + l2 * w2;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                acc[c][v].x = acc[c][v].x * w1 + __shfl_xor_sync(0xffffffffu, acc[c][v].x, off) * w2;
                acc[c][v].y = acc[c][v].y * w1 + __shfl_xor_sync(0xffffffffu, acc[c][v].y, off) * w2;
                acc[c][v].z = acc[c][v].z * w1 + __shfl_xor_sync(0xffffffffu, acc[c][v].z, off) * w2;
                acc[c][v].w = acc[c][v].w * w1 + __shfl_xor_sync(0xffffffffu, acc[c][v].w, off) * w2;
            }
        }
        if (lane < 8) {
#pragma unroll
            for (int v = 0; v < V; ++v) *reinterpret_cast<float4 *>(&o_s[warp][c][d0 + 32 * v]) = acc[c][v];
            if (lane == 0) { m_s[warp][c] = m[c]; l_s[warp][c] = l[c]; }
        }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nh * HD; d += 256) {
        const int c = d / HD;
        float mx = -INFINITY, lsum = 0.f, o = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) mx = fmaxf(mx, m_s[w][c]);
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const float e = m_s[w][c] == -INFINITY ? 0.f : __expf(m_s[w][c] - mx);
            lsum += l_s[w][c] * e; o += o_s[w][c][d % HD] * e;
        }
        orow[d] = lsum > 0.f ? o / lsum : 0.f;
    }
}

// ---------------------------------------------------------------------------------------------
// RMSNorm and SwiGLU (decoder-stack glue; both data types, fp32 arithmetic).
// ---------------------------------------------------------------------------------------------
template <typename T>
__global__ void rmsnorm_kernel(const T *__restrict__ x, const T *__restrict__ w, int H, float eps,
                               T *__restrict__ y) {
    const size_t row = blockIdx.x;
    __shared__ float red[32];
    float ss = 0.f;
    for (int h = threadIdx.x; h < H; h += blockDim.x) { float v = ldf(x + row * H + h); ss += v * v; }
    for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x < 32) {
        float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
        for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (threadIdx.x == 0) red[0] = rsqrtf(v / (float)H + eps);
    }
    __syncthreads();
    const float inv = red[0];
    for (int h = threadIdx.x; h < H; h += blockDim.x)
        stf(y + row * H + h, ldf(x + row * H + h) * inv * ldf(w + h));
}

template <typename T>
__global__ void swiglu_kernel(const T *__restrict__ gate_up, int I, size_t total, T *__restrict__ y) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const size_t row = i / I, c = i % I;
        const float g = ldf(gate_up + row * 2 * I + c), u = ldf(gate_up + row * 2 * I + I + c);
        stf(y + i, tc::silu_mul(g, u));
    }
}

// bf16 rows of up to 8192 elements (H a multiple of 8): the row is read once, 16 bytes per load and all of a thread's
// loads in flight together, kept in registers across the reduction, and written with 16-byte stores.  (The generic
// kernel above reads the row twice with one dependent 2-byte load per loop trip: 17 us for 8 rows of 4096, most of it
// memory latency.)  Launched as a programmatic dependent: the next kernel's prologue may start under this one.
constexpr int kNormVecs = 4;
__global__ void __launch_bounds__(256) rmsnorm_bf16_kernel(const __nv_bfloat16 *__restrict__ x,
                                                           const __nv_bfloat16 *__restrict__ w, int H, float eps,
                                                           __nv_bfloat16 *__restrict__ y) {
    tc::grid_dep_launch();
    tc::grid_dep_wait();
    const size_t row = blockIdx.x;
    const int nvec = H >> 3;
    __shared__ float red[32];
    uint4 v[kNormVecs];
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < kNormVecs; ++i) {
        const int idx = (int)threadIdx.x + i * 256;
        v[i] = idx < nvec ? *reinterpret_cast<const uint4 *>(x + row * H + (size_t)idx * 8) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < kNormVecs; ++i) {
        const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(&v[i]);
#pragma unroll
        for (int e = 0; e < 4; ++e) { const float2 f = __bfloat1622float2(p[e]); ss = fmaf(f.x, f.x, fmaf(f.y, f.y, ss)); }
    }
    for (int off = 16; off; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = threadIdx.x < 8 ? red[threadIdx.x] : 0.f;
        for (int off = 4; off; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (threadIdx.x == 0) red[0] = rsqrtf(t / (float)H + eps);
    }
    __syncthreads();
    const float inv = red[0];
#pragma unroll
    for (int i = 0; i < kNormVecs; ++i) {
        const int idx = (int)threadIdx.x + i * 256;
        if (idx >= nvec) continue;
        const uint4 wv = *reinterpret_cast<const uint4 *>(w + (size_t)idx * 8);
        const __nv_bfloat162 *px = reinterpret_cast<const __nv_bfloat162 *>(&v[i]);
        const __nv_bfloat162 *pw = reinterpret_cast<const __nv_bfloat162 *>(&wv);
        uint4 o;
        __nv_bfloat162 *po = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 a = __bfloat1622float2(px[e]), g = __bfloat1622float2(pw[e]);
            po[e] = __floats2bfloat162_rn(a.x * inv * g.x, a.y * inv * g.y);
        }
        *reinterpret_cast<uint4 *>(y + row * H + (size_t)idx * 8) = o;
    }
}

// SwiGLU on bf16 rows, eight columns per thread (I a multiple of 8): 16-byte loads of gate and up, 16-byte store.
__global__ void __launch_bounds__(256) swiglu_bf16_kernel(const __nv_bfloat16 *__restrict__ gate_up, int I, size_t total_vecs,
                                                          __nv_bfloat16 *__restrict__ y) {
    tc::grid_dep_launch();
    tc::grid_dep_wait();
    const int vecs_per_row = I >> 3;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total_vecs; i += (size_t)gridDim.x * blockDim.x) {
        const size_t row = i / vecs_per_row, c = (i - row * vecs_per_row) * 8;
        const uint4 gv = *reinterpret_cast<const uint4 *>(gate_up + row * 2 * I + c);
        const uint4 uv = *reinterpret_cast<const uint4 *>(gate_up + row * 2 * I + I + c);
        const __nv_bfloat162 *pg = reinterpret_cast<const __nv_bfloat162 *>(&gv);
        const __nv_bfloat162 *pu = reinterpret_cast<const __nv_bfloat162 *>(&uv);
        uint4 o;
        __nv_bfloat162 *po = reinterpret_cast<__nv_bfloat162 *>(&o);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 g = __bfloat1622float2(pg[e]), u = __bfloat1622float2(pu[e]);
            po[e] = __floats2bfloat162_rn(tc::silu_mul(g.x, u.x), tc::silu_mul(g.y, u.y));
        }
        *reinterpret_cast<uint4 *>(y + row * I + c) = o;
    }
}

int launch_rmsnorm(alora_ctx *ctx, const void *x, const void *w, int T, void *y, cudaStream_t s) {
    if (T == 0) return 0;
    ProfScope prof(ctx, KK_GLUE, s);
    const int H = ctx->d.H;
    const bool al16 = (((uintptr_t)x | (uintptr_t)w | (uintptr_t)y) & 15) == 0;
    if (ctx->cfg.dtype == ALORA_DTYPE_BF16 && H % 8 == 0 && H <= 8 * 256 * kNormVecs && al16)
        return launch_kernel(rmsnorm_bf16_kernel, dim3(T), dim3(256), 0, s, true, (const __nv_bfloat16 *)x,
                             (const __nv_bfloat16 *)w, H, ctx->cfg.rms_eps, (__nv_bfloat16 *)y) == cudaSuccess ? 1 : -1;
    if (ctx->cfg.dtype == ALORA_DTYPE_FP32)
        rmsnorm_kernel<float><<<T, 256, 0, s>>>((const float *)x, (const float *)w, ctx->d.H, ctx->cfg.rms_eps, (float *)y);
    else
        rmsnorm_kernel<__nv_bfloat16><<<T, 256, 0, s>>>((const __nv_bfloat16 *)x, (const __nv_bfloat16 *)w, ctx->d.H,
                                                        ctx->cfg.rms_eps, (__nv_bfloat16 *)y);
    return 1;
}

int launch_swiglu(alora_ctx *ctx, const void *gate_up, int T, void *y, cudaStream_t s) {
    if (T == 0) return 0;
    ProfScope prof(ctx, KK_GLUE, s);
    const size_t total = (size_t)T * ctx->d.I;
    int blocks = (int)((total + 255) / 256);
    if (blocks > ctx->sm_count * 16) blocks = ctx->sm_count * 16;
    if (ctx->cfg.dtype == ALORA_DTYPE_BF16 && ctx->d.I % 8 == 0 && (((uintptr_t)gate_up | (uintptr_t)y) & 15) == 0) {
        const size_t vecs = total / 8;
        const int vblocks = (int)std::min<size_t>((vecs + 255) / 256, (size_t)ctx->sm_count * 16);
        return launch_kernel(swiglu_bf16_kernel, dim3(vblocks), dim3(256), 0, s, true, (const __nv_bfloat16 *)gate_up,
                             ctx->d.I, vecs, (__nv_bfloat16 *)y) == cudaSuccess ? 1 : -1;
    }
    if (ctx->cfg.dtype == ALORA_DTYPE_FP32)
        swiglu_kernel<float><<<blocks, 256, 0, s>>>((const float *)gate_up, ctx->d.I, total, (float *)y);
    else
        swiglu_kernel<__nv_bfloat16><<<blocks, 256, 0, s>>>((const __nv_bfloat16 *)gate_up, ctx->d.I, total,
                                                           (__nv_bfloat16 *)y);
    return 1;
}

// ---- launchers of the fp32 projection / attention ------------------------------------------------------------------
int launch_project_simt(alora_ctx *ctx, int layer, const void *hidden, int T, void *qkv, cudaStream_t s, void *kv_pool,
                        int num_pages) {
    if (T == 0) return 0;
    const Dims &d = ctx->d;
    const AdapterDev *ads = ctx->d_adapters + (size_t)layer * ctx->cfg.max_adapters;
    {   // (an ordinary launch: x is complete before it begins, and so before the projection's base sums)
        ProfScope prof(ctx, KK_SHRINK, s);
        shrink_simt_kernel<<<dim3(T, 3), 256, 0, s>>>((const float *)hidden, ctx->d_row_adapter, ads, d.H, d.RP, (float *)ctx->d_t);
    }
    ProfScope prof(ctx, KK_PROJECT, s);
    const cudaError_t e = launch_kernel(linear_simt_kernel, dim3((d.N + 31) / 32 * ((T + 15) / 16)), dim3(256), 0, s, true,
        (const float *)hidden, (const float *)ctx->layers[layer].wqkv, T, d.H, d.N, (const int32_t *)ctx->d_row_adapter, ads,
        (const float *)ctx->d_t, d.RP, d.Nq, d.Nkv, (const float *)nullptr, (float *)qkv, (float *)kv_pool, (const int32_t *)ctx->d_slot,
        d.hd, d.Hkv, d.page, num_pages, 1, ctx->d_status);
    return e == cudaSuccess ? 2 : -1;
}

// Whether a layer call takes project_small_simt_kernel: x rows that a warp holds in registers, and few enough blocks (one is resident on
// an SM, so up to two rounds).  Every column tile forms t of its rows again, one warp a row, which for few rows and a large
// hidden x rank costs more than metadata, shrink and projection as launches of their own.  Those in turn take twice as long where the
// shrink's blocks and the tiles, which start beside them, are more than there are SMs.  Calls on 64 cached tokens, N 768, here / there, us:
//   hidden x rank      1 token   4          16         32         40
//   512 x 32           23 / 25   23 / 25    28 / 33    28 / 33    29 / 66
//   768 x 32           30 / 29   31 / 31    35 / 37    36 / 39    37 / 80
//   512 x 64           34 / 25   34 / 28    41 / 41    42 / 43    42 / 86
//   1024 x 64          58 / 35   59 / 37    67 / 51    68 / 53    69 / 115
// Both routes form the same base sums, so the rows without an adapter keep their bits whichever one a mode takes.
bool simt_small_layer(const alora_ctx *ctx, const BatchArgs &b) {
    const Dims &d = ctx->d;
    if (ctx->cfg.dtype != ALORA_DTYPE_FP32 || b.T <= 0 || d.H % 4 != 0 || d.H > 128 * kSmallVecs) return false;
    const long long tiles = (long long)((d.N + 31) / 32) * ((b.T + 15) / 16), work = (long long)d.H * ctx->largest_rank;
    const bool may_adapt = b.mode != ALORA_MODE_BASE && b.adapter_ids != nullptr;
    if (may_adapt && work > (b.T <= 4 ? 18432 : 30720) && 3 * b.T + tiles <= ctx->sm_count) return false;
    return tiles <= 2ll * ctx->sm_count;
}
int launch_project_small_simt(alora_ctx *ctx, int layer, const void *hidden, const BatchArgs &b, void *qkv, void *kv_pool, cudaStream_t s) {
    const Dims &d = ctx->d;
    ProfScope prof(ctx, KK_PROJECT, s);
    return launch_kernel(project_small_simt_kernel, dim3((d.N + 31) / 32 * ((b.T + 15) / 16)), dim3(768), 0, s, true,
        (const float *)hidden, (const float *)ctx->layers[layer].wqkv, b.T, d.H, d.N, d.Nq, d.Nkv, d.RP,
        ctx->d_adapters + (size_t)layer * ctx->cfg.max_adapters, b.positions, b.activation_offsets, b.adapter_ids, b.query_start_loc,
        b.seq_lens, b.block_tables, b.max_blocks, b.num_pages, d.page, ctx->cfg.max_adapters, b.R, b.mode, d.hd, d.Hkv, (float *)kv_pool,
        ctx->d_token_req, ctx->d_row_adapter, ctx->d_slot, (float *)qkv, ctx->d_status) == cudaSuccess ? 1 : -1;
}

int launch_linear_simt(alora_ctx *ctx, const void *x, const void *W, int T, int K, int N, void *y,
                       const void *residual, cudaStream_t s) {
    if (T == 0) return 0;
    ProfScope prof(ctx, KK_LINEAR, s);
    const cudaError_t e = launch_kernel(linear_simt_kernel, dim3((N + 31) / 32 * ((T + 15) / 16)), dim3(256), 0, s, true, (const float *)x,
        (const float *)W, T, K, N, (const int32_t *)nullptr, (const AdapterDev *)nullptr, (const float *)nullptr, 0, 0, 0,
        (const float *)residual, (float *)y, (float *)nullptr, (const int32_t *)nullptr, 0, 0, 0, 0, 0, ctx->d_status);
    return e == cudaSuccess ? 1 : -1;
}

int launch_attend_simt(alora_ctx *ctx, const void *qkv, const BatchArgs &b, const void *pool, void *out,
                       cudaStream_t s) {
    if (b.T == 0) return 0;
    const Dims &d = ctx->d;
    ProfScope prof(ctx, KK_ATTENTION, s);
    auto go = [&](auto kernel, int hc) {
        return launch_kernel(kernel, dim3(b.T, d.Hkv, (d.G + hc - 1) / hc), dim3(256), 0, s, true, (const float *)qkv,
                             (const int32_t *)ctx->d_token_req, (const int32_t *)ctx->d_slot, b.positions, b.query_start_loc, b.seq_lens, b.block_tables, b.max_blocks, b.num_pages,
                             d.page, d.N, d.Nq, d.Hkv, d.G, b.R, d.softmax_scale, (const float *)pool, (float *)out, ctx->d_status);
    };
    auto go_hd = [&](auto own) {
        constexpr bool kOwn = decltype(own)::value;
        const bool two = d.G > 1;
        return d.hd == 32 ? (two ? go(attn_simt_kernel<32, 2, kOwn>, 2) : go(attn_simt_kernel<32, 1, kOwn>, 1))
               : d.hd == 64 ? (two ? go(attn_simt_kernel<64, 2, kOwn>, 2) : go(attn_simt_kernel<64, 1, kOwn>, 1))
                            : (two ? go(attn_simt_kernel<128, 2, kOwn>, 2) : go(attn_simt_kernel<128, 1, kOwn>, 1));
    };
    return (b.own_facts ? go_hd(std::true_type{}) : go_hd(std::false_type{})) == cudaSuccess ? 1 : -1;
}

}  // namespace alora
