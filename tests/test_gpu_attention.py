"""GPU parity of the attention step alone (alora_kv_append + alora_attend) against the CPU oracle, on
seeded random caches: short suffixes and decode rows (the few-row split-KV kernel), long suffixes (the
tensor-core kernel), both mixed in one batch, head dims / group sizes / page sizes the kernels are
built for, and a cache whose unused slots hold NaN (nothing outside a row's causal range may leak)."""
import numpy as np
import pytest

from paper_2504_12397_b200 import binding as ab
from paper_2504_12397_b200 import workloads as wl

import helpers as hp

pytestmark = pytest.mark.gpu


def _attend_case(oracle, shape, P, S, seed, nan_canaries=True, scale_q=1.0):
    """Random cache + random new q/k/v rows -> append + attend on the GPU, oracle on the same values."""
    import torch
    rng = np.random.default_rng(seed)
    b = wl.make_batch(shape, P, S, [-1] * len(P), rng, shuffle_pages=True, with_hidden=False)
    T, R = b.T, b.R
    pool_np = wl.random_kv_pool(shape, b.num_pages, rng)
    qkv_np = wl.bf16_round(rng.standard_normal((T, shape.N), dtype=np.float32))
    qkv_np[:, :shape.Nq] *= scale_q
    qkv_np = wl.bf16_round(qkv_np)
    if nan_canaries:
        # every slot that holds no cached position (tails of last pages, spare pages) is NaN
        keep = np.zeros((b.num_pages, shape.page_size), bool)
        for r in range(R):
            for p in range(int(b.prefix_lens[r])):
                keep[b.block_tables[r, p // shape.page_size], p % shape.page_size] = True
        mask = ~keep[:, None, None, :, None]
        pool_np = np.where(np.broadcast_to(mask, pool_np.shape), np.float32(np.nan), pool_np)
    g = hp.GpuLayers(shape, [dict(wqkv=np.zeros((shape.N, shape.hidden), np.float32))], [[]], max(T, 1), max(R, 1))
    try:
        pool = hp.to_dev(pool_np, "bf16")
        qkv = hp.to_dev(qkv_np, "bf16")
        d = hp.DevBatch(b, "bf16")
        out = torch.full((T, shape.Nq), float("nan"), dtype=torch.bfloat16, device="cuda")
        ab.alora_kv_append(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, d.bt, d.max_blocks, b.num_pages, T, R, pool)
        ab.alora_attend(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, pool, d.bt, d.max_blocks, b.num_pages, T, R, out)
        assert g.status() == 0
        got = hp.to_host(out)
    finally:
        g.close()
    # oracle: contiguous K/V per request = cached prefix (from the pool) ++ the new rows
    Ks, Vs, kvl = [], [], [0]
    clean = np.nan_to_num(pool_np, nan=0.0)
    for r in range(R):
        Pr = int(b.prefix_lens[r])
        K0, V0 = oracle.paged_gather(clean, b.block_tables[r], Pr, shape.n_kv_heads, shape.page_size, shape.head_dim)
        rows = slice(b.query_start_loc[r], b.query_start_loc[r + 1])
        Ks.append(np.concatenate([K0, qkv_np[rows, shape.Nq:shape.Nq + shape.Nkv]]))
        Vs.append(np.concatenate([V0, qkv_np[rows, shape.Nq + shape.Nkv:]]))
        kvl.append(kvl[-1] + len(Ks[-1]))
    want, _ = oracle.attention(qkv_np[:, :shape.Nq], np.concatenate(Ks), np.concatenate(Vs), kvl, b.positions,
                               b.query_start_loc, shape.n_q_heads, shape.n_kv_heads, shape.head_dim)
    assert np.isfinite(got).all(), "a value from outside a row's causal range reached an output"
    return hp.rel_err(got, want), got, want


SHAPE_G4 = wl.LayerShape(hidden=256, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16")


def test_decode_rows_split_kv(oracle64):
    """One new token per request, contexts from 1 key to several key ranges (split-KV and its merge)."""
    P = [0, 1, 15, 16, 63, 64, 65, 255, 256, 257, 1000, 2049, 3333]
    err, _, _ = _attend_case(oracle64, SHAPE_G4, P, [1] * len(P), seed=101)
    assert err <= 2e-2


@pytest.mark.parametrize("S", [2, 3, 4, 5, 8, 13, 16])
def test_short_suffixes_split_kv(oracle64, S):
    """Suffixes of 2..16 tokens (16, 32 or 64 score rows per KV head) with range boundaries that fall
    between the positions of the block's tokens."""
    P = [0, 7, 250, 255, 256, 1021, 2500]
    err, _, _ = _attend_case(oracle64, SHAPE_G4, P, [S] * len(P), seed=200 + S)
    assert err <= 2e-2


def test_mixed_short_and_long_requests(oracle64):
    """Short requests (few-row kernel) and long ones (tensor-core kernel) in one call, ragged."""
    P = [300, 0, 1500, 64, 900, 10, 0]
    S = [1, 16, 17, 200, 4, 129, 1]
    err, got, want = _attend_case(oracle64, SHAPE_G4, P, S, seed=301)
    assert err <= 2e-2


def test_large_scores_do_not_overflow(oracle64):
    """Queries scaled up so that scores reach a few hundred: the running-maximum subtraction must hold."""
    err, _, _ = _attend_case(oracle64, SHAPE_G4, [700, 100, 2100], [1, 16, 3], seed=401, scale_q=24.0)
    assert err <= 2e-2


@pytest.mark.parametrize("hq,hkv,hd,page", [(4, 4, 128, 16), (4, 2, 64, 16), (16, 2, 128, 16), (8, 1, 64, 32),
                                            (4, 1, 128, 8), (8, 2, 128, 64), (8, 2, 128, 128)])
def test_shapes_group_sizes_and_page_sizes(oracle64, hq, hkv, hd, page):
    shape = wl.LayerShape(hidden=256, n_q_heads=hq, n_kv_heads=hkv, head_dim=hd, page_size=page, dtype="bf16")
    P = [0, 130, 777, 31, 1300]
    S = [1, 5, 16, 150, 2]
    err, _, _ = _attend_case(oracle64, shape, P, S, seed=500 + hq + hd + page)
    assert err <= 2e-2


def _attend_values(shape, b, pool_np, qkv_np):
    """Append + attend on the GPU with the given cache and q/k/v rows; the output rows."""
    import torch
    g = hp.GpuLayers(shape, [dict(wqkv=np.zeros((shape.N, shape.hidden), np.float32))], [[]], b.T, b.R)
    try:
        pool, qkv, d = hp.to_dev(pool_np, "bf16"), hp.to_dev(qkv_np, "bf16"), hp.DevBatch(b, "bf16")
        out = torch.full((b.T, shape.Nq), float("nan"), dtype=torch.bfloat16, device="cuda")
        ab.alora_kv_append(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, d.bt, d.max_blocks, b.num_pages, b.T, b.R, pool)
        ab.alora_attend(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, pool, d.bt, d.max_blocks, b.num_pages, b.T, b.R, out)
        assert g.status() == 0
        return hp.to_host(out)
    finally:
        g.close()


def _oracle_values(oracle, shape, b, pool_np, qkv_np):
    Ks, Vs, kvl = [], [], [0]
    for r in range(b.R):
        K0, V0 = oracle.paged_gather(pool_np, b.block_tables[r], int(b.prefix_lens[r]), shape.n_kv_heads, shape.page_size,
                                     shape.head_dim)
        rows = slice(b.query_start_loc[r], b.query_start_loc[r + 1])
        Ks.append(np.concatenate([K0, qkv_np[rows, shape.Nq:shape.Nq + shape.Nkv]]))
        Vs.append(np.concatenate([V0, qkv_np[rows, shape.Nq + shape.Nkv:]]))
        kvl.append(kvl[-1] + len(Ks[-1]))
    return oracle.attention(qkv_np[:, :shape.Nq], np.concatenate(Ks), np.concatenate(Vs), kvl, b.positions, b.query_start_loc,
                            shape.n_q_heads, shape.n_kv_heads, shape.head_dim)[0]


def _write_keys(shape, b, pool_np, r, first, keys):
    """Puts `keys` [n, head_dim] (for every KV head) into request r's cached positions first, first + 1, ..."""
    for i, k in enumerate(keys):
        pool_np[b.block_tables[r, (first + i) // shape.page_size], 0, :, (first + i) % shape.page_size] = k


@pytest.mark.parametrize("page", [8, 16, 64])
@pytest.mark.parametrize("S", [20, 40])
@pytest.mark.parametrize("nats", [60, 100, 200])
def test_one_late_key_far_above_the_reference(oracle64, page, S, nats):
    """A key in the middle of the context whose score lies `nats` above all others, at each of 32 neighbouring positions in
    turn (one request each): the softmax works on a running reference, and whatever unit takes this key's exponential, the
    row has to become that key's value."""
    shape = wl.LayerShape(hidden=256, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=page, dtype="bf16")
    rng = np.random.default_rng(700 + page + S + nats)
    R = 32
    b = wl.make_batch(shape, [1000] * R, [S] * R, [-1] * R, rng, shuffle_pages=True, with_hidden=False)
    pool = wl.random_kv_pool(shape, b.num_pages, rng)
    qkv = wl.bf16_round(rng.standard_normal((b.T, shape.N), dtype=np.float32))
    u = rng.choice([-1.0, 1.0], shape.head_dim).astype(np.float32)
    qkv[:, :shape.Nq] = np.tile(u, shape.n_q_heads)
    for r in range(R):
        _write_keys(shape, b, pool, r, 640 + r, wl.bf16_round(u * np.float32(nats / shape.head_dim ** 0.5))[None])
    got, want = _attend_values(shape, b, pool, qkv), _oracle_values(oracle64, shape, b, pool, qkv)
    hp.assert_close(got, want, 2e-2, f"a key {nats} nats above the others", block=shape.head_dim)


@pytest.mark.parametrize("S", [24, 48])
def test_a_row_does_not_depend_on_the_rows_beside_it(S):
    """Every third token of a request gets queries whose scores jump by tens of nats from tile to tile, so that its rows
    take their maximum again and again; the other tokens (which share their warps) keep the bits that they have without
    that, as rows before an activation offset have to."""
    shape = wl.LayerShape(hidden=256, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16")
    rng = np.random.default_rng(800 + S)
    R = 8
    b = wl.make_batch(shape, [1500 + 61 * r for r in range(R)], [S] * R, [-1] * R, rng, shuffle_pages=True, with_hidden=False)
    pool = wl.random_kv_pool(shape, b.num_pages, rng)
    qkv = wl.bf16_round(rng.standard_normal((b.T, shape.N), dtype=np.float32))
    jumpy = qkv.copy()
    loud = np.arange(b.T) % 3 == 1
    jumpy[loud, :shape.Nq] = wl.bf16_round(jumpy[loud, :shape.Nq] * 30)
    calm_rows, jumpy_rows = _attend_values(shape, b, pool, qkv), _attend_values(shape, b, pool, jumpy)
    assert np.array_equal(calm_rows[~loud].view(np.uint32), jumpy_rows[~loud].view(np.uint32))
    assert hp.rel_err(jumpy_rows[loud], calm_rows[loud]) > 0.1


@pytest.mark.parametrize("S", [20, 40])
@pytest.mark.parametrize("dead", [64, 128, 300])
def test_leading_keys_with_scores_of_minus_infinity(oracle64, S, dead):
    """The first keys of a context give every query a score of -inf, the others scores far below zero: the row has no
    reference when it meets the first finite score, and takes that score's maximum however low it is."""
    shape = wl.LayerShape(hidden=256, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16")
    rng = np.random.default_rng(900 + S + dead)
    P = [1000, 77 + dead, 2000]
    b = wl.make_batch(shape, P, [S] * 3, [-1] * 3, rng, shuffle_pages=True, with_hidden=False)
    pool = wl.random_kv_pool(shape, b.num_pages, rng)
    qkv = wl.bf16_round(rng.standard_normal((b.T, shape.N), dtype=np.float32))
    qkv[:, :shape.Nq] = np.abs(qkv[:, :shape.Nq]) + 0.5
    qkv[:, :shape.Nq] = wl.bf16_round(qkv[:, :shape.Nq])
    new_k = slice(shape.Nq, shape.Nq + shape.Nkv)
    qkv[:, new_k] -= 13   # scores of about -13 * sum(q) / sqrt(128): -190
    qkv[:, new_k] = wl.bf16_round(qkv[:, new_k])
    pool[:, 0] = wl.bf16_round(pool[:, 0] - 13)
    for r in range(3):
        keys = wl.bf16_round(rng.standard_normal((dead, shape.head_dim), dtype=np.float32))
        keys[:, 5] = -np.inf
        _write_keys(shape, b, pool, r, 0, keys)
    got = _attend_values(shape, b, pool, qkv)
    want = _oracle_values(oracle64, shape, b, np.where(np.isinf(pool), np.float32(-1e30), pool), qkv)
    hp.assert_close(got, want, 2e-2, "keys of -inf in front", block=shape.head_dim)


@pytest.mark.parametrize("S", [[33], [32, 64, 65, 31], [127, 128, 129], [33, 64] * 19, [40, 33] * 45])
def test_blocks_of_half_size_and_claimed_items(oracle64, S):
    """Few items: blocks of 32 tokens instead of 64, at the edges of both; 38 requests in blocks of 64, nearly one a block; 90 requests
    with more items than blocks, which the blocks claim."""
    P = [(i * 613) % 1500 for i in range(len(S))]
    err, _, _ = _attend_case(oracle64, SHAPE_G4, P, S, seed=700 + len(S))
    assert err <= 2e-2


@pytest.mark.parametrize("more", [0, 1])
def test_blocks_of_half_size_up_to_one_an_sm(oracle64, more):
    """The largest list of half-size blocks (two a request, two KV heads: one item an SM), and the first batch that keeps whole ones."""
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count // 4 + more
    P = [(i * 613) % 1500 for i in range(n)]
    err, _, _ = _attend_case(oracle64, SHAPE_G4, P, [33 + (i * 7) % 32 for i in range(n)], seed=800 + more)
    assert err <= 2e-2
