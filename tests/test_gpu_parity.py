"""GPU parity: every step of the hot path through the C ABI against the CPU oracle, element by
element, on seeded inputs that span several tiles and ragged tails.  Integer outputs and gated-off
rows must match exactly; floating-point outputs within the tolerance of tests/helpers.tol."""
import numpy as np
import pytest

from paper_2504_12397_b200 import binding as ab
from paper_2504_12397_b200 import workloads as wl

import helpers as hp

pytestmark = pytest.mark.gpu

# reduced 8B-like bf16 shape: same head_dim / group size as the 8B layer, smaller widths
MID = wl.LayerShape(hidden=1024, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16",
                    intermediate=1536)


def _mid_workload(seed=11, a_req_shift=True):
    """Ragged multi-adapter batch: 6 requests over adapters of ranks 8/16/32/64 and the base model,
    prefixes 0..700, suffixes 1..300, some activation offsets inside the new chunk, shuffled pages."""
    rng = np.random.default_rng(seed)
    w = wl.make_wqkv(MID, rng)
    ads = [wl.make_adapter(MID, r, rng, scale=s) for r, s in ((8, 1.0), (16, 2.0), (32, 1.0), (64, 0.5))]
    for a in ads:  # lift the delta well above bf16 rounding noise so a wrong or missing delta is visible
        for n in ("Bq", "Bk", "Bv"):
            setattr(a, n, wl.bf16_round(getattr(a, n) * 8))
    P = [0, 37, 700, 129, 256, 300]
    S = [150, 300, 1, 131, 128, 17]
    ids = [2, 0, 3, -1, 1, 2]
    a_req = [0, 37 + 130, 700, 0, 256 + 5, 300]
    b = wl.make_batch(MID, P, S, ids, rng, activation_offsets=a_req if a_req_shift else None,
                      shuffle_pages=True, with_prefix_hidden=True)
    return w, ads, b


def _run_base_prefill(g: hp.GpuLayers, shape, b, pool, layer=0):
    pb = hp.prefix_only_batch(shape, b)
    if pb.T == 0:
        return
    d = hp.DevBatch(pb, shape.dtype)
    out = g.empty(pb.T, shape.Nq)
    ab.alora_full_lora_prefill_layer(g.ctx, layer, d.hidden, d.positions, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                                     d.max_blocks, b.num_pages, d.T, d.R, out)


def _gather_pool(orc, shape, pool_np, b):
    return [orc.paged_gather(pool_np, b.block_tables[r], int(b.seq_lens[r]), shape.n_kv_heads, shape.page_size,
                             shape.head_dim) for r in range(b.R)]


@pytest.mark.parametrize("mode", [ab.MODE_ALORA, ab.MODE_FULL_LORA, ab.MODE_BASE])
def test_batch_metadata_is_exact(oracle64, mode):
    w, ads, b = _mid_workload()
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], b.T, b.R)
    try:
        import torch
        d = hp.DevBatch(b, MID.dtype)
        tok = torch.full((b.T,), -9, dtype=torch.int32, device="cuda")
        row = torch.full((b.T,), -9, dtype=torch.int32, device="cuda")
        slot = torch.full((b.T,), -9, dtype=torch.int32, device="cuda")
        ab.alora_batch_metadata(g.ctx, mode, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, d.bt, d.max_blocks,
                                b.num_pages, d.T, d.R, tok, row, slot)
        assert g.status() == 0
        want_slot = oracle64.slot_mapping(b.positions, b.query_start_loc, b.block_tables, MID.page_size)
        np.testing.assert_array_equal(slot.cpu().numpy().astype(np.int64), want_slot)
        # the oracle's gate, read off a projection with throw-away 4-wide weights
        from oracle import Adapter
        z14, z11 = np.zeros((1, 4)), np.zeros((1, 1))
        _, gate = oracle64.project_qkv(np.zeros((b.T, 4)), np.zeros((3, 4), np.float32), 1, 1, b.positions,
                                       b.query_start_loc, b.activation_offsets, b.adapter_ids,
                                       [Adapter(1, 1.0, z14, z11, z14, z11, z14, z11) for _ in ads],
                                       force_all=(mode == ab.MODE_FULL_LORA))
        req = np.repeat(np.arange(b.R), np.diff(b.query_start_loc))
        np.testing.assert_array_equal(tok.cpu().numpy(), req)
        want_row = np.where(gate.astype(bool), b.adapter_ids[req], -1)
        if mode == ab.MODE_BASE:
            want_row[:] = -1
        np.testing.assert_array_equal(row.cpu().numpy(), want_row)
    finally:
        g.close()


def test_config1_tiny_fp32_layer(oracle64):
    """Config 1 end to end: base prefill builds the cache, the aLoRA suffix prefill reuses it."""
    w = wl.config1()
    shape, b = w.shape, w.batch
    g = hp.GpuLayers(shape, [dict(wqkv=w.wqkv)], [w.adapters], 128, 4)
    try:
        pool = g.new_pool(b.num_pages)
        _run_base_prefill(g, shape, b, pool)
        d = hp.DevBatch(b, shape.dtype)
        out = g.empty(b.T, shape.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        qkv = g.empty(b.T, shape.N)
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens,
                             d.T, d.R, qkv)
        assert g.status() == 0
        Ks, Vs = hp.oracle_base_prefix(oracle64, shape, w.wqkv, b)
        want = hp.oracle_block(oracle64, shape, w.wqkv, w.adapters, b, Ks, Vs)
        assert want["gate"].all()
        hp.assert_close(hp.to_host(qkv), want["qkv"], 1e-5, "")
        hp.assert_close(hp.to_host(out), want["out"], 1e-5, "")
        got = _gather_pool(oracle64, shape, hp.to_host(pool), b)
        for r in range(b.R):
            hp.assert_close(got[r][0], want["K"][r], 1e-5, "")
            hp.assert_close(got[r][1], want["V"][r], 1e-5, "")
        # the delta matters in this configuration: the base model's answer is outside the tolerance
        b0 = wl.Batch(**{**b.__dict__, "adapter_ids": np.array([-1], np.int32)})
        base = hp.oracle_block(oracle64, shape, w.wqkv, w.adapters, b0, Ks, Vs)
        assert hp.rel_err(base["qkv"], want["qkv"]) > 1e-3
    finally:
        g.close()


@pytest.mark.parametrize("hidden,heads,kv_heads,hd,new", [(36, 3, 1, 32, (1, 16)), (100, 4, 4, 128, (33, 5)), (64, 5, 1, 64, (17, 130))])
def test_fp32_layer_tile_and_head_edges(oracle64, hidden, heads, kv_heads, hd, new):
    """Rows, widths and K that do not fill the fp32 tiles, one and several query heads per KV head (an odd number too), every
    head dimension, gates opening inside a request, keys from none but the token's own to more than a block's streams."""
    shape = wl.LayerShape(hidden=hidden, n_q_heads=heads, n_kv_heads=kv_heads, head_dim=hd, page_size=16, dtype="fp32", intermediate=64)
    rng = np.random.default_rng(hidden)
    w = wl.make_wqkv(shape, rng)
    ads = [wl.make_adapter(shape, 3, rng), wl.make_adapter(shape, 8, rng, scale=2.0)]
    b = wl.make_batch(shape, [0, 70], list(new), [1, 0], rng, activation_offsets=[0, 73], shuffle_pages=True, with_prefix_hidden=True)
    g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], 256, 4)
    try:
        pool = g.new_pool(b.num_pages)
        _run_base_prefill(g, shape, b, pool)
        d = hp.DevBatch(b, shape.dtype)
        out = g.empty(b.T, shape.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        assert g.status() == 0
        Ks, Vs = hp.oracle_base_prefix(oracle64, shape, w, b)
        want = hp.oracle_block(oracle64, shape, w, ads, b, Ks, Vs)
        hp.assert_close(hp.to_host(out), want["out"], 1e-5, "")   # the bound of the other fp32 layer test
        got = _gather_pool(oracle64, shape, hp.to_host(pool), b)
        for r in range(b.R):
            hp.assert_close(got[r][0], want["K"][r], 1e-5, "")
            hp.assert_close(got[r][1], want["V"][r], 1e-5, "")
    finally:
        g.close()


@pytest.mark.parametrize("hidden,n_req", [(64, 32), (64, 33), (64, 70), (64, 1030), (1028, 33), (1028, 70)])
def test_fp32_layer_of_many_requests(oracle64, hidden, n_req):
    """More requests than a warp has lanes, and than it has lanes squared, with empty ones in between and at the end: each token's
    request is found by the small layer's own kernels (hidden 64) and by the metadata step (1028)."""
    shape = wl.LayerShape(hidden=hidden, n_q_heads=2, n_kv_heads=1, head_dim=32, page_size=16, dtype="fp32")
    rng = np.random.default_rng(n_req)
    w = wl.make_wqkv(shape, rng)
    ads = [wl.make_adapter(shape, 3, rng), wl.make_adapter(shape, 8, rng, scale=2.0)]
    P = [(i * 7) % 40 for i in range(n_req)]
    S = [(1, 0, 2, 1, 0)[i % 5] for i in range(n_req)]
    S[0], S[-1] = 0, (0 if n_req % 2 else 1)
    b = wl.make_batch(shape, P, S, [(i % 3) - 1 for i in range(n_req)], rng, activation_offsets=[p + (i % 4 == 1) for i, p in enumerate(P)],
                      shuffle_pages=True)
    fill = wl.random_kv_pool(shape, b.num_pages, rng)
    g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], b.T, b.R)
    try:
        d = hp.DevBatch(b, shape.dtype)
        pool, out = g.new_pool(b.num_pages, fill), g.empty(b.T, shape.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt, d.max_blocks,
                               b.num_pages, d.T, d.R, out)
        assert g.status() == 0
        kv = [oracle64.paged_gather(fill, b.block_tables[r], P[r], shape.n_kv_heads, shape.page_size, shape.head_dim) if P[r] else (None, None)
              for r in range(n_req)]
        want = hp.oracle_block(oracle64, shape, w, ads, b, [k for k, _ in kv], [v for _, v in kv])
        hp.assert_close(hp.to_host(out), want["out"], 1e-5, "")   # the bound of the other fp32 layer tests
        slots = oracle64.slot_mapping(b.positions, b.query_start_loc, b.block_tables, shape.page_size)
        got, old = hp.to_host(pool).swapaxes(1, 3).reshape(-1, shape.n_kv_heads, 2, shape.head_dim), fill.swapaxes(1, 3).reshape(-1, shape.n_kv_heads, 2, shape.head_dim)
        hp.assert_close(got[slots][:, 0, 0], want["qkv"][:, shape.Nq:shape.Nq + shape.Nkv], 1e-5, "")
        rest = np.setdiff1d(np.arange(len(got)), slots)
        assert np.array_equal(got[rest], old[rest])
    finally:
        g.close()


def test_fp32_attention_of_many_requests_costs_what_few_cost():
    """4096 one-token requests against 512 of eight tokens, the same number of rows and fewer keys: the attention does not look for
    its request among all of them in every block (1.6 times as long where it did, 1.0 now)."""
    import torch
    shape = wl.LayerShape(hidden=64, n_q_heads=4, n_kv_heads=2, head_dim=64, page_size=16, dtype="fp32")
    rng = np.random.default_rng(3)
    T, times = 4096, []
    g = hp.GpuLayers(shape, [dict(wqkv=wl.make_wqkv(shape, rng))], [[]], T, T)
    try:
        for n_req in (512, 4096):
            b = wl.make_batch(shape, [0] * n_req, [T // n_req] * n_req, [-1] * n_req, rng, with_hidden=False)
            d = hp.DevBatch(b, shape.dtype)
            pool, qkv, out = g.new_pool(b.num_pages), torch.randn(T, shape.N, device="cuda"), g.empty(T, shape.Nq)
            best = float("inf")
            for i in range(8):
                ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                ev[0].record()
                for _ in range(20):
                    ab.alora_attend(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, pool, d.bt, d.max_blocks, b.num_pages, T, n_req, out)
                ev[1].record()
                torch.cuda.synchronize()
                best = min(best, ev[0].elapsed_time(ev[1])) if i >= 2 else best
            times.append(best)
        assert g.status() == 0
    finally:
        g.close()
    assert times[1] < 1.3 * times[0], times


@pytest.mark.parametrize("hidden,rank,S,launches", [(512, 36, (2, 2), 2), (512, 37, (2, 2), 4), (512, 60, (3, 2), 2), (512, 61, (3, 2), 4),
                                                    (1024, 64, (20, 13), 4), (1024, 64, (20, 14), 2)])
def test_fp32_small_layer_at_its_limits(oracle64, hidden, rank, S, launches):
    """Few rows and a large hidden x rank (of the largest registered adapter) take metadata, shrink and projection as launches of their
    own, as long as their blocks fit on the SMs (148) side by side; else a small fp32 layer is two launches.  Calls without adapters take
    those anyway; rows whose gate is closed have the same bits on either route."""
    shape = wl.LayerShape(hidden=hidden, n_q_heads=4, n_kv_heads=2, head_dim=64, page_size=16, dtype="fp32")
    rng = np.random.default_rng(rank)
    w = wl.make_wqkv(shape, rng)
    ads = [wl.make_adapter(shape, 8, rng), wl.make_adapter(shape, rank, rng)]
    b = wl.make_batch(shape, [5, 9], list(S), [0, 1], rng, activation_offsets=[5 + S[0] // 2, 9 + 1], with_prefix_hidden=True)
    g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], 64, 4)
    try:
        d = hp.DevBatch(b, shape.dtype)
        pools = [g.new_pool(b.num_pages) for _ in range(2)]
        for pool in pools:
            _run_base_prefill(g, shape, b, pool)
        outs = [g.empty(b.T, shape.Nq) for _ in range(2)]
        n = [ab.alora_launch_count(g.ctx)]
        for ids, pool, out in ((d.ids, pools[0], outs[0]), (None, pools[1], outs[1])):
            ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, ids, d.qsl, d.seq_lens, pool, d.bt, d.max_blocks,
                                   b.num_pages, d.T, d.R, out)
            n.append(ab.alora_launch_count(g.ctx))
        assert g.status() == 0
        assert (n[1] - n[0], n[2] - n[1]) == (launches, 2)
        Ks, Vs = hp.oracle_base_prefix(oracle64, shape, w, b)
        want = hp.oracle_block(oracle64, shape, w, ads, b, Ks, Vs)
        hp.assert_close(hp.to_host(outs[0]), want["out"], 1e-5, "")
        off = want["gate"] == 0
        assert 0 < off.sum() < b.T
        assert np.array_equal(hp.to_host(outs[0])[off].view(np.uint32), hp.to_host(outs[1])[off].view(np.uint32))
        slots = oracle64.slot_mapping(b.positions, b.query_start_loc, b.block_tables, shape.page_size)[off]
        kept = [hp.to_host(p).swapaxes(1, 3).reshape(-1, 2 * shape.Nkv)[slots] for p in pools]
        assert np.array_equal(kept[0].view(np.uint32), kept[1].view(np.uint32))
    finally:
        g.close()


def test_ragged_multi_adapter_layer_bf16(oracle64):
    """Projection, append and attention on a ragged multi-adapter batch with mid-chunk activation."""
    w, ads, b = _mid_workload()
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], 2048, 8)
    try:
        pool = g.new_pool(b.num_pages)
        _run_base_prefill(g, MID, b, pool)
        pool_before = hp.to_host(pool).copy()
        d = hp.DevBatch(b, MID.dtype)
        out = g.empty(b.T, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        qkv = g.empty(b.T, MID.N)
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens,
                             d.T, d.R, qkv)
        base = g.empty(b.T, MID.N)
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_BASE, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens,
                             d.T, d.R, base)
        assert g.status() == 0
        Ks, Vs = hp.oracle_base_prefix(oracle64, MID, w, b)
        want = hp.oracle_block(oracle64, MID, w, ads, b, Ks, Vs)
        qkv_h, base_h, out_h = hp.to_host(qkv), hp.to_host(base), hp.to_host(out)
        hp.assert_close(qkv_h, want["qkv"], 2e-2, "")
        hp.assert_close(out_h, want["out"], 2e-2, "")
        # rows whose gate is closed: bit-identical to the GPU base-only projection (Prop. 1)
        off = want["gate"] == 0
        assert off.sum() > 100 and (~off).sum() > 100
        assert np.array_equal(qkv_h[off].view(np.uint32), base_h[off].view(np.uint32))
        # rows whose gate is open really carry the delta
        assert hp.rel_err(base_h[~off], want["qkv"][~off]) > 5e-2
        # KV append: new rows equal the projection's k/v parts bit for bit, every other byte untouched
        pool_after = hp.to_host(pool)
        slots = oracle64.slot_mapping(b.positions, b.query_start_loc, b.block_tables, MID.page_size)
        expect = pool_before.copy()
        oracle64.paged_append(expect, qkv_h[:, MID.Nq:MID.Nq + MID.Nkv], qkv_h[:, MID.Nq + MID.Nkv:], slots,
                              MID.n_kv_heads, MID.page_size, MID.head_dim)
        assert np.array_equal(pool_after.view(np.uint32), expect.view(np.uint32))
        # prefix rows in the cache are the base model's (made by the base prefill) within tolerance
        got = _gather_pool(oracle64, MID, pool_after, b)
        for r in range(b.R):
            hp.assert_close(got[r][0], want["K"][r], 2e-2, "")
            hp.assert_close(got[r][1], want["V"][r], 2e-2, "")
    finally:
        g.close()


def test_sub_steps_compose_to_the_layer_call(oracle64):
    """alora_project_qkv + alora_kv_append + alora_attend == alora_prefill_layer, bit for bit."""
    w, ads, b = _mid_workload(seed=12)
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], 2048, 8)
    try:
        rng = np.random.default_rng(0)
        fill = wl.random_kv_pool(MID, b.num_pages, rng)
        d = hp.DevBatch(b, MID.dtype)
        pool1, pool2 = g.new_pool(b.num_pages, fill), g.new_pool(b.num_pages, fill)
        out1, out2 = g.empty(b.T, MID.Nq), g.empty(b.T, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool1, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out1)
        qkv = g.empty(b.T, MID.N)
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens,
                             d.T, d.R, qkv)
        ab.alora_kv_append(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, d.bt, d.max_blocks, b.num_pages, d.T, d.R, pool2)
        ab.alora_attend(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, pool2, d.bt, d.max_blocks, b.num_pages, d.T, d.R, out2)
        assert g.status() == 0
        assert np.array_equal(hp.to_host(pool1).view(np.uint32), hp.to_host(pool2).view(np.uint32))
        assert np.array_equal(hp.to_host(out1).view(np.uint32), hp.to_host(out2).view(np.uint32))
        # attention alone against the oracle on a random (non-projected) cache
        pool_h, qkv_h = hp.to_host(pool2), hp.to_host(qkv)
        kv = _gather_pool(oracle64, MID, pool_h, b)
        kvl = np.concatenate([[0], np.cumsum(b.seq_lens)])
        want, _ = oracle64.attention(qkv_h[:, :MID.Nq], np.concatenate([k for k, _ in kv]),
                                     np.concatenate([v for _, v in kv]), kvl, b.positions, b.query_start_loc,
                                     MID.n_q_heads, MID.n_kv_heads, MID.head_dim)
        hp.assert_close(hp.to_host(out2), want, 2e-2, "")
    finally:
        g.close()


def _boosted_adapters(shape, rng, spec):
    ads = [wl.make_adapter(shape, r, rng, scale=s) for r, s in spec]
    for a in ads:  # lift the delta well above bf16 rounding noise so a wrong or missing delta is visible
        for n in ("Bq", "Bk", "Bv"):
            setattr(a, n, wl.bf16_round(getattr(a, n) * 8))
    return ads


def _check_projection(oracle64, shape, w, ads, b, n_off_expected=None, on_pairs=None):
    """on_pairs: whether the kernel on pairs of SMs has to serve the batch (None: not looked at)."""
    g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], b.T, b.R)
    try:
        if on_pairs is not None:
            assert (ab.alora_selftest_pair_tile(g.ctx, 0, 0, b.T, b.R) > 0) == on_pairs
        d = hp.DevBatch(b, shape.dtype)
        qkv, base, again = g.empty(b.T, shape.N), g.empty(b.T, shape.N), g.empty(b.T, shape.N)
        for mode, dst in ((ab.MODE_ALORA, qkv), (ab.MODE_BASE, base), (ab.MODE_ALORA, again)):
            ab.alora_project_qkv(g.ctx, 0, mode, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, d.T, d.R, dst)
        assert g.status() == 0
        want, gate = oracle64.project_qkv(b.hidden, w, shape.Nq, shape.Nkv, b.positions, b.query_start_loc,
                                          b.activation_offsets, b.adapter_ids, hp.oracle_adapters(ads))
        qkv_h, base_h = hp.to_host(qkv), hp.to_host(base)
        hp.assert_close(qkv_h, want, 2e-2, "")
        off = gate == 0
        if n_off_expected is not None:
            assert off.sum() == n_off_expected
        assert off.sum() > 0 and (~off).sum() > 0
        # rows whose gate is closed: bit-identical to the GPU base-only projection (Prop. 1)
        assert np.array_equal(qkv_h[off].view(np.uint32), base_h[off].view(np.uint32))
        # rows whose gate is open really carry the delta
        assert hp.rel_err(base_h[~off], want[~off]) > 5e-2
        # run-to-run determinism
        assert np.array_equal(hp.to_host(again).view(np.uint32), qkv_h.view(np.uint32))
    finally:
        g.close()


def test_projection_row_tile_route_with_fused_shrink(oracle64):
    """Long requests at 256-wide column tiles: row tiles segmented by (adapter, gate), the rank-r shrink
    running as leading work items of the projection kernel."""
    rng = np.random.default_rng(43)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, ((8, 1.0), (64, 0.5), (32, 2.0)))
    b = wl.make_batch(MID, [0, 300, 20, 5], [500, 390, 130, 260], [1, 0, -1, 2], rng, activation_offsets=[130, 300, 0, 200])
    _check_projection(oracle64, MID, w, ads, b, n_off_expected=130 + 130 + 195)


def test_projection_of_many_rows_on_single_sms(oracle64):
    """Many rows on tiles of 128 x 256, one a block, where those take fewer rounds than the tiles of pairs of SMs, with the shrink as leading
    work items: 36 row tiles in two rounds, one request on the base model, gates that open in the middle of requests."""
    rng = np.random.default_rng(45)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, ((8, 1.0), (64, 0.5), (32, 2.0)))
    b = wl.make_batch(MID, [0, 300, 20, 5, 0], [1500, 1390, 530, 760, 428], [1, 0, -1, 2, 0], rng,
                      activation_offsets=[130, 300, 0, 200, 77])
    _check_projection(oracle64, MID, w, ads, b, n_off_expected=130 + 530 + 195 + 77, on_pairs=False)


def test_projection_row_wise_route_many_short_requests(oracle64):
    """Many requests of 1..9 new tokens over different adapters and the base model, some gated off: every row tile
    holds rows of all four adapters, a few each."""
    rng = np.random.default_rng(44)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, ((8, 1.0), (64, 0.5), (32, 2.0), (16, 1.0)))
    R = 40
    S = [1 + (i * 7) % 9 for i in range(R)]
    P = [(i * 37) % 200 for i in range(R)]
    ids = [(i % 5) - 1 for i in range(R)]
    a_req = [P[i] + (3 if i % 4 == 0 else 0) for i in range(R)]   # every fourth request opens its gate 3 tokens late
    b = wl.make_batch(MID, P, S, ids, rng, activation_offsets=a_req)
    _check_projection(oracle64, MID, w, ads, b)


@pytest.mark.parametrize("n_req,each", [(129, 1), (140, 1), (33, 5), (257, 4)])
def test_projection_row_tiles_with_many_adapters(oracle64, n_req, each):
    """More requests and more adapters in a row tile than a warp has lanes, a last tile of one row, requests across the
    tile boundary, with t in three summands (up to 1024 rows) and in one (257 x 4 rows)."""
    rng = np.random.default_rng(49)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, tuple((8, 0.5 + 0.1 * (i % 7)) for i in range(36)))
    P = [(i * 37) % 200 for i in range(n_req)]
    ids = [(i * 5) % 37 - 1 for i in range(n_req)]
    b = wl.make_batch(MID, P, [each] * n_req, ids, rng, activation_offsets=[p + (i % 6 == 0) for i, p in enumerate(P)])
    _check_projection(oracle64, MID, w, ads, b)


@pytest.mark.parametrize("T", [1, 24, 33, 64, 65, 128])
def test_projection_few_row_route_mixed_adapters(oracle64, T):
    """Batches of at most 128 rows (decode steps): the weight-streaming route, K split over the SMs, the shrink of
    every present adapter riding along, slice partials added in fixed order.  One token per request, requests mixing
    the base model and four adapters of different ranks in no particular order, every third adapter request with
    its gate still closed.  Checked: oracle, closed-gate rows bit-identical to the base-only call, determinism."""
    rng = np.random.default_rng(100 + T)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, ((8, 1.0), (64, 0.5), (32, 2.0), (16, 1.0)))
    R = T
    ids = [int(x) for x in rng.integers(-1, 4, R)]
    if R >= 24:
        ids[:5] = [3, -1, 0, 2, 1]
    else:
        ids[0] = 2
    P = [int(x) for x in rng.integers(0, 300, R)]
    a_req = [P[i] + (1 if (ids[i] >= 0 and i % 3 == 1) else 0) for i in range(R)]   # gate closed on this step
    if R == 1:
        b2 = wl.make_batch(MID, P + [7], [1, 1], ids + [1], rng, activation_offsets=a_req + [8])   # one open, one closed row
        return _check_projection(oracle64, MID, w, ads, b2)
    b = wl.make_batch(MID, P, [1] * R, ids, rng, activation_offsets=a_req)
    _check_projection(oracle64, MID, w, ads, b)


@pytest.mark.parametrize("T,n_ad,rank", [(16, 1, 64), (17, 2, 24), (32, 16, 16), (127, 3, 40), (40, 17, 16), (129, 3, 40), (385, 2, 64)])
def test_projection_few_row_route_row_boxes_and_adapter_limits(oracle64, T, n_ad, rank):
    """Row counts at the edges of the 16 / 32 / 64 / 128-row boxes, ranks that padding rounds up, the most rank columns that
    the one-launch kernel takes (16 adapters of rank 16) and one adapter more (the two-kernel route); several row tiles, the
    last of one row."""
    rng = np.random.default_rng(300 + T)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, tuple((max(1, rank - i % 5), 0.5 + 0.25 * (i % 3)) for i in range(n_ad)))
    P = [int(x) for x in rng.integers(0, 300, T)]
    ids = [(i * 7) % (n_ad + 1) - 1 for i in range(T)]
    b = wl.make_batch(MID, P, [1] * T, ids, rng, activation_offsets=[p + (i % 6 == 1) for i, p in enumerate(P)])
    _check_projection(oracle64, MID, w, ads, b)


@pytest.mark.parametrize("T,n_ad,rank", [(1, 1, 64), (33, 3, 24), (128, 16, 16), (300, 0, 8)])
def test_few_row_layer_call_equals_its_sub_steps(T, n_ad, rank):
    """In a layer call W x starts before the batch's adapter facts are there and A x takes a second pass over x; the
    projection alone does both in one pass.  The new K / V rows and the attention rows have to be the same bits."""
    rng = np.random.default_rng(400 + T)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, tuple((rank, 1.0) for _ in range(n_ad)))
    P = [int(x) for x in rng.integers(0, 300, T)]
    ids = [(i * 7) % (n_ad + 1) - 1 if T > 1 else 0 for i in range(T)]
    b = wl.make_batch(MID, P, [1] * T, ids, rng, activation_offsets=[p + (i % 6 == 1) for i, p in enumerate(P)])
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], 512, 512)
    try:
        fill = wl.random_kv_pool(MID, b.num_pages, rng)
        d = hp.DevBatch(b, MID.dtype)
        pool1, pool2 = g.new_pool(b.num_pages, fill), g.new_pool(b.num_pages, fill)
        out1, out2, qkv = g.empty(b.T, MID.Nq), g.empty(b.T, MID.Nq), g.empty(b.T, MID.N)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool1, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out1)
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens,
                             d.T, d.R, qkv)
        ab.alora_kv_append(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, d.bt, d.max_blocks, b.num_pages, d.T, d.R, pool2)
        ab.alora_attend(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, pool2, d.bt, d.max_blocks, b.num_pages, d.T, d.R, out2)
        assert g.status() == 0
        assert np.array_equal(hp.to_host(pool1).view(np.uint32), hp.to_host(pool2).view(np.uint32))
        assert np.array_equal(hp.to_host(out1).view(np.uint32), hp.to_host(out2).view(np.uint32))
    finally:
        g.close()


def test_projection_few_row_route_short_suffixes_one_adapter(oracle64):
    """8 requests x 16 new tokens (128 rows), one adapter, gates opening inside the chunk."""
    rng = np.random.default_rng(49)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, ((32, 1.0),))
    P = [100 + 13 * i for i in range(8)]
    a_req = [P[i] + (5 if i % 2 else 0) for i in range(8)]
    b = wl.make_batch(MID, P, [16] * 8, [0] * 8, rng, activation_offsets=a_req)
    _check_projection(oracle64, MID, w, ads, b, n_off_expected=20)


def test_decode_sized_stack_takes_the_few_row_projections(oracle64):
    """Two decoder layers on a batch of 40 rows (requests of 1 .. 6 new tokens on cached prefixes made by a base
    prefill through the same stack): q/k/v, o_proj, gate/up and down all run on the few-row route, two of the
    last three with the residual added."""
    shape = wl.LayerShape(hidden=512, n_q_heads=4, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16",
                          intermediate=1024)
    rng = np.random.default_rng(33)
    layers = [wl.make_stack_weights(shape, rng) for _ in range(2)]
    ads = [[wl.make_adapter(shape, 16, rng), wl.make_adapter(shape, 8, rng)] for _ in range(2)]
    for per in ads:
        for a in per:
            for n in ("Bq", "Bk", "Bv"):
                setattr(a, n, wl.bf16_round(getattr(a, n) * 8))
    S = [1, 6, 2, 5, 3, 4, 1, 6, 2, 5, 3, 2]
    assert sum(S) == 40
    ids = [0, 1, -1, 0, 1, -1, 1, 0, -1, 1, 0, 1]
    b = wl.make_batch(shape, [0] * len(S), S, ids, rng, activation_offsets=[2 if i % 4 == 1 else 0 for i in range(len(S))],
                      shuffle_pages=True)
    g = hp.GpuLayers(shape, layers, ads, 128, 16)
    try:
        d = hp.DevBatch(b, shape.dtype)
        pools = [g.new_pool(b.num_pages) for _ in range(2)]
        hout = g.empty(b.T, shape.hidden)
        ab.alora_forward_stack(g.ctx, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pools,
                               d.bt, d.max_blocks, b.num_pages, d.T, d.R, hout)
        assert g.status() == 0
        x = b.hidden.astype(np.float64)
        for l in range(2):
            x, blk = oracle64.decoder_layer(x, layers[l], shape.Nq, shape.Nkv, shape.n_q_heads, shape.n_kv_heads,
                                            shape.head_dim, 1e-5, b.positions, b.query_start_loc,
                                            b.activation_offsets, b.adapter_ids, hp.oracle_adapters(ads[l]),
                                            [None] * b.R, [None] * b.R)
            got = _gather_pool(oracle64, shape, hp.to_host(pools[l]), b)
            for r in range(b.R):
                hp.assert_close(got[r][0], blk["K"][r], 2e-2, f"layer {l} K rows of request {r}")
        hp.assert_close(hp.to_host(hout), x, 2e-2, "stack output")
    finally:
        g.close()


def test_projection_with_128_wide_kv_blocks(oracle64):
    """One KV head of 128 columns: the q/k/v block boundaries force 128-wide column tiles, and the rank-r
    shrink then runs as the separate cluster split-K kernel."""
    shape = wl.LayerShape(hidden=1536, n_q_heads=4, n_kv_heads=1, head_dim=128, page_size=16, dtype="bf16")
    rng = np.random.default_rng(41)
    w = wl.make_wqkv(shape, rng)
    ads = _boosted_adapters(shape, rng, ((64, 1.0), (8, 2.0)))
    b = wl.make_batch(shape, [0, 50, 10], [600, 440, 277], [0, 1, 0], rng, activation_offsets=[100, 50, 0])
    _check_projection(oracle64, shape, w, ads, b, n_off_expected=100)


def test_short_suffixes_on_an_empty_or_tiny_cache(oracle64):
    """Requests with 5 .. 40 new tokens and 0 .. 70 cached ones: attention work items of one or two key tiles whose
    rows all fall into one query group of the tensor-core kernel (both groups then share the item, one 64-key half
    of the tile each), including items where one half holds no visible key at all, and the NaN-proofing of V rows
    beyond the causal limit (the pool starts as all-ones bit patterns)."""
    import torch
    rng = np.random.default_rng(47)
    w = wl.make_wqkv(MID, rng)
    ads = _boosted_adapters(MID, rng, ((8, 1.0), (32, 1.0)))
    P = [0, 0, 3, 0, 70, 0, 12]
    S = [5, 9, 20, 40, 6, 32, 33]
    ids = [0, 1, -1, 0, 1, 0, 1]
    b = wl.make_batch(MID, P, S, ids, rng, shuffle_pages=True, with_prefix_hidden=True)
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], 256, 8)
    try:
        pool = g.new_pool(b.num_pages)
        pool.view(torch.int16).fill_(-1)   # bf16 NaN everywhere a kernel does not write
        _run_base_prefill(g, MID, b, pool)
        d = hp.DevBatch(b, MID.dtype)
        out = g.empty(b.T, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        assert g.status() == 0
        Ks, Vs = hp.oracle_base_prefix(oracle64, MID, w, b)
        want = hp.oracle_block(oracle64, MID, w, ads, b, Ks, Vs)
        out_h = hp.to_host(out)
        assert np.isfinite(out_h).all()
        for r in range(b.R):
            q0, q1 = int(b.query_start_loc[r]), int(b.query_start_loc[r + 1])
            hp.assert_close(out_h[q0:q1], want["out"][q0:q1], 2e-2, f"request {r}")
    finally:
        g.close()


def test_full_lora_recompute_matches_eq4(oracle64):
    w, ads, b = _mid_workload(seed=13)
    fb = hp.full_sequence_batch(MID, b)
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], fb.T, fb.R)
    try:
        d = hp.DevBatch(fb, MID.dtype)
        pool = g.new_pool(b.num_pages)
        out = g.empty(fb.T, MID.Nq)
        ab.alora_full_lora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                                         d.max_blocks, b.num_pages, d.T, d.R, out)
        assert g.status() == 0
        want = hp.oracle_block(oracle64, MID, w, ads, fb, [None] * fb.R, [None] * fb.R, force_all=True)
        hp.assert_close(hp.to_host(out), want["out"], 2e-2, "")
        got = _gather_pool(oracle64, MID, hp.to_host(pool), fb)
        for r in range(fb.R):
            hp.assert_close(got[r][0], want["K"][r], 2e-2, "")
            hp.assert_close(got[r][1], want["V"][r], 2e-2, "")
    finally:
        g.close()


def test_cache_reuse_identity_on_gpu(oracle64):
    """Prop. 1 on the GPU: masked aLoRA prefill of the whole sequence from scratch leaves the same
    cache as base prefill of the prefix + aLoRA suffix prefill, and the same suffix outputs."""
    w, ads, b = _mid_workload(seed=14, a_req_shift=False)
    fb = hp.full_sequence_batch(MID, b)
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], fb.T, fb.R)
    try:
        pool_a = g.new_pool(b.num_pages)
        _run_base_prefill(g, MID, b, pool_a)
        d = hp.DevBatch(b, MID.dtype)
        out_a = g.empty(b.T, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool_a, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out_a)
        df = hp.DevBatch(fb, MID.dtype)
        pool_b = g.new_pool(b.num_pages)
        out_b = g.empty(fb.T, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, df.hidden, df.positions, df.a_req, df.ids, df.qsl, df.seq_lens, pool_b,
                               df.bt, df.max_blocks, b.num_pages, df.T, df.R, out_b)
        assert g.status() == 0
        pa, pb = hp.to_host(pool_a), hp.to_host(pool_b)
        ka = _gather_pool(oracle64, MID, pa, b); kb = _gather_pool(oracle64, MID, pb, b)
        oa, ob = hp.to_host(out_a), hp.to_host(out_b)
        for r in range(b.R):
            P = int(b.prefix_lens[r])
            # prefix rows: exact (both are base-only arithmetic on the same inputs)
            assert np.array_equal(ka[r][0][:P].view(np.uint32), kb[r][0][:P].view(np.uint32))
            assert np.array_equal(ka[r][1][:P].view(np.uint32), kb[r][1][:P].view(np.uint32))
            hp.assert_close(ka[r][0], kb[r][0], 2e-2, "K")
            hp.assert_close(ka[r][1], kb[r][1], 2e-2, "V")
            lo, hi = b.query_start_loc[r], b.query_start_loc[r + 1]
            tail = slice(fb.query_start_loc[r] + P, fb.query_start_loc[r + 1])
            hp.assert_close(ob[tail], oa[lo:hi], 2e-2, "")
    finally:
        g.close()


def test_decode_steps_match_prefill_rows(oracle64):
    """Prop. 1, second sentence: decoding the suffix token by token reproduces the prefill."""
    rng = np.random.default_rng(21)
    w = wl.make_wqkv(MID, rng)
    ads = [wl.make_adapter(MID, 32, rng), wl.make_adapter(MID, 16, rng)]
    for a in ads:
        for n in ("Bq", "Bk", "Bv"):
            setattr(a, n, wl.bf16_round(getattr(a, n) * 8))
    P, S = [40, 333, 17, 64, 100], [6, 6, 6, 6, 6]
    ids = [0, -1, 1, 0, 1]
    a_req = [42, 0, 17, 0, 103]
    b = wl.make_batch(MID, P, S, ids, rng, activation_offsets=a_req, shuffle_pages=True, with_prefix_hidden=True)
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], 1024, 8)
    try:
        import torch
        pool = g.new_pool(b.num_pages)
        _run_base_prefill(g, MID, b, pool)
        pool_dec = pool.clone()
        d = hp.DevBatch(b, MID.dtype)
        out = g.empty(b.T, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        out_h = hp.to_host(out)
        dec = np.zeros_like(out_h)
        for i in range(6):
            rows = b.query_start_loc[:-1] + i
            hid = d.hidden[torch.from_numpy(rows).cuda().long()].contiguous()
            pos = hp.idev(b.positions[rows]); sl = hp.idev(b.positions[rows] + 1)
            o = g.empty(b.R, MID.Nq)
            ab.alora_decode_step(g.ctx, 0, hid, pos, d.a_req, d.ids, sl, pool_dec, d.bt, d.max_blocks, b.num_pages,
                                 b.R, o)
            dec[rows] = hp.to_host(o)
        assert g.status() == 0
        Ks, Vs = hp.oracle_base_prefix(oracle64, MID, w, b)
        want = hp.oracle_block(oracle64, MID, w, ads, b, Ks, Vs)
        hp.assert_close(out_h, want["out"], 2e-2, "")
        hp.assert_close(dec, want["out"], 2e-2, "")
        hp.assert_close(hp.to_host(pool_dec), hp.to_host(pool), 2e-2, "")
    finally:
        g.close()


def test_two_layer_stack(oracle64):
    """Reduced decoder stack end to end (RMSNorm, attention block, o_proj, SwiGLU MLP, residuals)."""
    shape = wl.LayerShape(hidden=512, n_q_heads=4, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16",
                          intermediate=1024)
    rng = np.random.default_rng(31)
    layers = [wl.make_stack_weights(shape, rng) for _ in range(2)]
    ads = [[wl.make_adapter(shape, 16, rng)] for _ in range(2)]
    for per in ads:
        for a in per:
            for n in ("Bq", "Bk", "Bv"):
                setattr(a, n, wl.bf16_round(getattr(a, n) * 8))
    b = wl.make_batch(shape, [0, 0], [200, 77], [0, -1], rng, activation_offsets=[150, 0], shuffle_pages=True)
    g = hp.GpuLayers(shape, layers, ads, 512, 4)
    try:
        d = hp.DevBatch(b, shape.dtype)
        pools = [g.new_pool(b.num_pages) for _ in range(2)]
        hout = g.empty(b.T, shape.hidden)
        ab.alora_forward_stack(g.ctx, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pools,
                               d.bt, d.max_blocks, b.num_pages, d.T, d.R, hout)
        assert g.status() == 0
        x = b.hidden.astype(np.float64)
        for l in range(2):
            x, blk = oracle64.decoder_layer(x, layers[l], shape.Nq, shape.Nkv, shape.n_q_heads, shape.n_kv_heads,
                                            shape.head_dim, 1e-5, b.positions, b.query_start_loc,
                                            b.activation_offsets, b.adapter_ids, hp.oracle_adapters(ads[l]),
                                            [None] * b.R, [None] * b.R)
            got = _gather_pool(oracle64, shape, hp.to_host(pools[l]), b)
            for r in range(b.R):
                hp.assert_close(got[r][0], blk["K"][r], 2e-2, "")
        hp.assert_close(hp.to_host(hout), x, 2e-2, "")
    finally:
        g.close()


def test_stack_layer_with_many_rows_and_a_short_k(oracle64):
    """One decoder layer on 2048 tokens with a wide MLP and a hidden size of 256: gate / up (2048 x 9472 outputs = 592 tiles of 128 x 256) on
    the 128-row kernel with SwiGLU in a kernel of its own, as are o_proj and q/k/v; down (K 4736, two column tiles) on pairs of SMs."""
    shape = wl.LayerShape(hidden=256, n_q_heads=4, n_kv_heads=2, head_dim=64, page_size=16, dtype="bf16",
                          intermediate=4736)
    rng = np.random.default_rng(41)
    layers = [wl.make_stack_weights(shape, rng)]
    ads = [[wl.make_adapter(shape, 8, rng)]]
    b = wl.make_batch(shape, [0] * 8, [256] * 8, [0, -1] * 4, rng, activation_offsets=[100] * 8, shuffle_pages=True)
    g = hp.GpuLayers(shape, layers, ads, 2048, 8)
    try:
        assert [ab.alora_selftest_pair_tile(g.ctx, 0, m, b.T, b.R) > 0 for m in range(4)] == [False, False, False, True]
        d = hp.DevBatch(b, shape.dtype)
        pools = [g.new_pool(b.num_pages)]
        hout = g.empty(b.T, shape.hidden)
        ab.alora_forward_stack(g.ctx, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pools,
                               d.bt, d.max_blocks, b.num_pages, d.T, d.R, hout)
        assert g.status() == 0
        x, _ = oracle64.decoder_layer(b.hidden.astype(np.float64), layers[0], shape.Nq, shape.Nkv, shape.n_q_heads,
                                      shape.n_kv_heads, shape.head_dim, 1e-5, b.positions, b.query_start_loc,
                                      b.activation_offsets, b.adapter_ids, hp.oracle_adapters(ads[0]),
                                      [None] * b.R, [None] * b.R)
        hp.assert_close(hp.to_host(hout), x, 2e-2, "")
    finally:
        g.close()


def test_stack_layer_at_the_8b_shape_with_1024_rows(oracle64):
    """One decoder layer at the 8B layer shape on 4 x 256 new tokens: q/k/v with its adapter, o_proj, gate / up (28672 columns, SwiGLU in
    the epilogue) and down (K = 14336) on pairs of SMs, the 16-byte norm kernel at its real row length.  Every row against the
    oracle (about 0.23 TFLOP of oracle work)."""
    shape = wl.SHAPE_8B
    rng = np.random.default_rng(48)
    layers = [wl.make_stack_weights(shape, rng)]
    ads = [[wl.make_adapter(shape, 32, rng)]]
    for n in ("Bq", "Bk", "Bv"):
        setattr(ads[0][0], n, wl.bf16_round(getattr(ads[0][0], n) * 8))
    b = wl.make_batch(shape, [0] * 4, [256] * 4, [0, -1, 0, 0], rng, activation_offsets=[100, 0, 0, 255],
                      shuffle_pages=True)
    g = hp.GpuLayers(shape, layers, ads, 1024, 4)
    try:
        assert all(ab.alora_selftest_pair_tile(g.ctx, 0, m, b.T, b.R) for m in range(4))
        d = hp.DevBatch(b, shape.dtype)
        pools = [g.new_pool(b.num_pages)]
        hout = g.empty(b.T, shape.hidden)
        ab.alora_forward_stack(g.ctx, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pools,
                               d.bt, d.max_blocks, b.num_pages, d.T, d.R, hout)
        assert g.status() == 0
        x, _ = oracle64.decoder_layer(b.hidden.astype(np.float64), layers[0], shape.Nq, shape.Nkv, shape.n_q_heads,
                                      shape.n_kv_heads, shape.head_dim, 1e-5, b.positions, b.query_start_loc,
                                      b.activation_offsets, b.adapter_ids, hp.oracle_adapters(ads[0]),
                                      [None] * b.R, [None] * b.R)
        hp.assert_close(hp.to_host(hout), x, 2e-2, "8B-shape layer, 1024 rows", block=shape.head_dim)
    finally:
        g.close()


@pytest.mark.parametrize("T", [200, 600, 2048])
def test_profile_counts_only_groups_that_launched(T):
    """One layer with adapters on the MLP block, whose rows take the row tiles or the pairs of SMs: a launcher that passes a batch on
    to the next one leaves no empty group behind."""
    shape = wl.LayerShape(hidden=1024, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16", intermediate=2048)
    rng = np.random.default_rng(3)
    b = wl.make_batch(shape, [0, 0], [T - 70, 70], [0, -1], rng)
    g = hp.GpuLayers(shape, [wl.make_stack_weights(shape, rng)], [[wl.make_adapter(shape, 8, rng)]], T, 2,
                     mlp_adapters_per_layer=[[wl.make_mlp_adapter(shape, 8, rng)]])
    try:
        d = hp.DevBatch(b, shape.dtype)
        pool, hout = g.new_pool(b.num_pages), g.empty(T, shape.hidden)
        ab.alora_profile_enable(g.ctx, True)
        n = ab.alora_launch_count(g.ctx)
        ab.alora_forward_stack(g.ctx, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, [pool], d.bt, d.max_blocks,
                               b.num_pages, T, 2, hout)
        n = ab.alora_launch_count(g.ctx) - n
        groups = {k: v[1] for k, v in ab.alora_profile_read(g.ctx).items()}
        assert g.status() == 0
    finally:
        g.close()
    assert groups["project_qkv"] == 1 and groups["linear"] == 3, groups   # o_proj, gate / up, down
    assert sum(groups.values()) <= n, (groups, n)


def test_empty_and_degenerate_batches():
    w, ads, b = _mid_workload()
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], 256, 8)
    try:
        import torch
        # T = 0: nothing launched that touches memory, status stays clean
        z = torch.zeros(1, dtype=torch.int32, device="cuda")
        pool = g.new_pool(4)
        out = g.empty(1, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, out, z, z, z, z, z, pool, z, 1, 4, 0, 0, out)
        assert g.status() == 0
        # a request with zero new tokens between two non-empty ones
        rng = np.random.default_rng(5)
        b2 = wl.make_batch(MID, [5, 9, 0], [3, 0, 2], [0, 1, -1], rng, shuffle_pages=True)
        d = hp.DevBatch(b2, MID.dtype)
        fill = wl.random_kv_pool(MID, b2.num_pages, rng)
        pool = g.new_pool(b2.num_pages, fill)
        out = g.empty(b2.T, MID.Nq)
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b2.num_pages, d.T, d.R, out)
        assert g.status() == 0
        assert np.isfinite(hp.to_host(out)).all()
        # host-side rejections: nothing is launched
        n0 = ab.alora_launch_count(g.ctx)
        for bad in (dict(T=10 ** 6), dict(layer=3), dict(hidden=None)):
            args = dict(layer=0, hidden=d.hidden, T=d.T)
            args.update(bad)
            with pytest.raises(ab.AloraError):
                ab.alora_prefill_layer(g.ctx, args["layer"], args["hidden"], d.positions, d.a_req, d.ids, d.qsl,
                                       d.seq_lens, pool, d.bt, d.max_blocks, b2.num_pages, args["T"], d.R, out)
        assert ab.alora_launch_count(g.ctx) == n0
    finally:
        g.close()


def test_device_side_findings_are_reported_not_trapped():
    """A block-table entry outside the pool and inconsistent positions are recorded in the status
    word; the offending rows are skipped and the context stays usable."""
    w, ads, b = _mid_workload()
    g = hp.GpuLayers(MID, [dict(wqkv=w)], [ads], 2048, 8)
    try:
        rng = np.random.default_rng(6)
        fill = wl.random_kv_pool(MID, b.num_pages, rng)
        d = hp.DevBatch(b, MID.dtype)
        pool = g.new_pool(b.num_pages, fill)
        out = g.empty(b.T, MID.Nq)
        bt = b.block_tables.copy()
        last_blk = (int(b.seq_lens[0]) - 1) // MID.page_size
        bt[0, last_blk] = b.num_pages + 5
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, hp.idev(bt),
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        assert g.status() == 7
        pos = b.positions.copy(); pos[3] += 2
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, hp.idev(pos), d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        assert g.status() == 6
        ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt,
                               d.max_blocks, b.num_pages, d.T, d.R, out)
        assert g.status() == 0
    finally:
        g.close()


def test_decode_steps_through_the_stack_match_the_prefill_rows(oracle64):
    """Two decoder layers: a prefill of all but the last three tokens of every request, then three decode steps
    through alora_decode_stack; the rows the steps produce equal the rows of the oracle's stack over the whole
    sequences (Prop. 1, second sentence), for requests on two adapters and on the base model, with gates that open
    before, inside and after the prefilled part."""
    shape = wl.LayerShape(hidden=512, n_q_heads=4, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16",
                          intermediate=1024)
    rng = np.random.default_rng(37)
    layers = [wl.make_stack_weights(shape, rng) for _ in range(2)]
    ads = [[wl.make_adapter(shape, 16, rng), wl.make_adapter(shape, 8, rng)] for _ in range(2)]
    for per in ads:
        for a in per:
            for n in ("Bq", "Bk", "Bv"):
                setattr(a, n, wl.bf16_round(getattr(a, n) * 8))
    L = [40, 23, 64, 9, 31]
    ids = [0, 1, -1, 0, 1]
    a_req = [10, 22, 0, 0, 100]
    n_dec = 3
    full = wl.make_batch(shape, [0] * len(L), L, ids, rng, activation_offsets=a_req, shuffle_pages=True)
    R = full.R
    g = hp.GpuLayers(shape, layers, ads, 256, 8)
    try:
        pools = [g.new_pool(full.num_pages) for _ in range(2)]
        # prefill part: tokens 0 .. L-4 of every request
        keep = np.concatenate([np.arange(full.query_start_loc[r], full.query_start_loc[r + 1] - n_dec) for r in range(R)])
        pre = wl.Batch(positions=full.positions[keep],
                       query_start_loc=np.concatenate([[0], np.cumsum(np.array(L) - n_dec)]).astype(np.int32),
                       seq_lens=(np.array(L) - n_dec).astype(np.int32), prefix_lens=np.zeros(R, np.int32),
                       activation_offsets=full.activation_offsets, adapter_ids=full.adapter_ids,
                       block_tables=full.block_tables, num_pages=full.num_pages, hidden=full.hidden[keep])
        d = hp.DevBatch(pre, shape.dtype)
        hout = g.empty(pre.T, shape.hidden)
        ab.alora_forward_stack(g.ctx, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pools,
                               d.bt, d.max_blocks, full.num_pages, d.T, d.R, hout)
        got = np.zeros((R, n_dec, shape.hidden), np.float32)
        for i in range(n_dec):
            rows = full.query_start_loc[1:] - n_dec + i
            pos = full.positions[rows]
            hid = hp.to_dev(full.hidden[rows], "bf16")
            o = g.empty(R, shape.hidden)
            ab.alora_decode_stack(g.ctx, hid, hp.idev(pos), d.a_req, d.ids, hp.idev(pos + 1), pools, d.bt, d.max_blocks,
                                  full.num_pages, R, o)
            got[:, i] = hp.to_host(o)
        assert g.status() == 0
        x = full.hidden.astype(np.float64)
        for l in range(2):
            x, _ = oracle64.decoder_layer(x, layers[l], shape.Nq, shape.Nkv, shape.n_q_heads, shape.n_kv_heads,
                                          shape.head_dim, 1e-5, full.positions, full.query_start_loc,
                                          full.activation_offsets, full.adapter_ids, hp.oracle_adapters(ads[l]),
                                          [None] * R, [None] * R)
        for i in range(n_dec):
            rows = full.query_start_loc[1:] - n_dec + i
            hp.assert_close(got[:, i], x[rows], 2e-2, f"decode step {i} through the stack")
        hp.assert_close(hp.to_host(hout), x[keep], 2e-2, "prefilled rows")
    finally:
        g.close()


def test_stack_layers_on_different_projection_routes_share_the_attention_list(oracle64):
    """Three decoder layers of which only the first has adapters, more of them than the few-row projection takes (5 x 64 rank
    columns): its q/k/v go through the row tiles, those of the other layers through the few-row kernel, while the attention
    list of the 200 decode rows (800 streams, more than there are blocks, the long ones cut into key ranges) is built once.
    Every layer has to see all of it."""
    shape = wl.LayerShape(hidden=512, n_q_heads=8, n_kv_heads=4, head_dim=64, page_size=16, dtype="bf16", intermediate=512)
    rng = np.random.default_rng(61)
    n, R = 3, 200
    layers = [wl.make_stack_weights(shape, rng) for _ in range(n)]
    ads = [_boosted_adapters(shape, rng, [(64, 1.0)] * 5), [], []]
    P = [int(p) for p in rng.integers(1, 300, R)]
    P[7], P[150] = 2900, 2111
    b = wl.make_batch(shape, P, [1] * R, [-1] * R, rng, shuffle_pages=True)   # (the route is chosen by what is registered)
    pools_np = [wl.random_kv_pool(shape, b.num_pages, rng) for _ in range(n)]
    g = hp.GpuLayers(shape, layers, ads, R, R)
    try:
        d = hp.DevBatch(b, shape.dtype)
        hout = g.empty(R, shape.hidden)
        for _ in range(2):   # (a second call finds what the first one left)
            pools = [g.new_pool(b.num_pages, fill=p) for p in pools_np]
            ab.alora_decode_stack(g.ctx, d.hidden, d.positions, d.a_req, d.ids, d.seq_lens, pools, d.bt, d.max_blocks,
                                  b.num_pages, R, hout)
            assert g.status() == 0
            x = b.hidden.astype(np.float64)
            for l in range(n):
                kv = [oracle64.paged_gather(pools_np[l], b.block_tables[r], P[r], shape.n_kv_heads, shape.page_size,
                                            shape.head_dim) for r in range(R)]
                x, _ = oracle64.decoder_layer(x, layers[l], shape.Nq, shape.Nkv, shape.n_q_heads, shape.n_kv_heads,
                                              shape.head_dim, 1e-5, b.positions, b.query_start_loc, b.activation_offsets,
                                              b.adapter_ids, [], [k for k, _ in kv], [v for _, v in kv])
            hp.assert_close(hp.to_host(hout), x, 2e-2, "decode step through layers on different routes", block=shape.head_dim)
    finally:
        g.close()


def test_stack_layers_hand_the_claim_counter_of_the_attention_on(oracle64):
    """Four layers on a batch with more attention items (180) than blocks, which the blocks claim from a counter: layers 0 and 2 use one
    counter, 1 and 3 the other, each cleared by the layer in between.  A second call begins with what the first one left."""
    shape = wl.LayerShape(hidden=256, n_q_heads=4, n_kv_heads=2, head_dim=64, page_size=16, dtype="bf16", intermediate=256)
    rng = np.random.default_rng(67)
    n, R = 4, 90
    layers = [wl.make_stack_weights(shape, rng) for _ in range(n)]
    P = [int(p) for p in rng.integers(0, 400, R)]
    b = wl.make_batch(shape, P, [int(s) for s in rng.integers(33, 65, R)], [-1] * R, rng, shuffle_pages=True)
    pools_np = [wl.random_kv_pool(shape, b.num_pages, rng) for _ in range(n)]
    g = hp.GpuLayers(shape, layers, [[]] * n, b.T, R)
    try:
        d = hp.DevBatch(b, shape.dtype)
        outs = []
        for _ in range(2):
            pools, hout = [g.new_pool(b.num_pages, fill=p) for p in pools_np], g.empty(b.T, shape.hidden)
            ab.alora_forward_stack(g.ctx, ab.MODE_BASE, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pools, d.bt, d.max_blocks,
                                   b.num_pages, d.T, d.R, hout)
            assert g.status() == 0
            outs.append(hp.to_host(hout))
        assert np.array_equal(outs[0].view(np.uint32), outs[1].view(np.uint32))
        x = b.hidden.astype(np.float64)
        for l in range(n):
            kv = [oracle64.paged_gather(pools_np[l], b.block_tables[r], P[r], shape.n_kv_heads, shape.page_size, shape.head_dim) if P[r]
                  else (None, None) for r in range(R)]
            x, _ = oracle64.decoder_layer(x, layers[l], shape.Nq, shape.Nkv, shape.n_q_heads, shape.n_kv_heads, shape.head_dim, 1e-5,
                                          b.positions, b.query_start_loc, b.activation_offsets, b.adapter_ids, [],
                                          [k for k, _ in kv], [v for _, v in kv])
        hp.assert_close(outs[0], x, 2e-2, "four layers, items claimed", block=shape.head_dim)
    finally:
        g.close()


@pytest.mark.parametrize("n_req,each,kv_heads,slots", [(9, 12, 2, 3), (9, 12, 2, 5), (20, 30, 2, 3), (20, 30, 2, 5), (47, 17, 2, 5),
                                                       (30, 45, 2, 3), (11, 50, 1, 5)])
def test_non_finite_adapter_values_stay_in_the_rows_that_use_them(oracle64, n_req, each, kv_heads, slots):
    """One of three adapters has Inf, -Inf and NaN among its B values.  On every projection route (few rows in one launch or,
    with five adapter slots, in two; one row tile per block, two, 128-wide column tiles) the rows of the other adapters and of the base model, which share its row tiles, keep
    the bits they have beside a finite adapter; its own rows are non-finite in those columns and right in all others."""
    shape = wl.LayerShape(hidden=512, n_q_heads=4, n_kv_heads=kv_heads, head_dim=128, page_size=16, dtype="bf16")
    rng = np.random.default_rng(71 + n_req)
    w = wl.make_wqkv(shape, rng)
    ads = _boosted_adapters(shape, rng, [(16, 1.0), (24, 0.5), (64, 1.0)])
    ids = [(r % 4) - 1 for r in range(n_req)]
    b = wl.make_batch(shape, [40] * n_req, [each] * n_req, ids, rng, activation_offsets=[40 + (3 if r % 3 == 0 else 0) for r in range(n_req)])
    want, gate = oracle64.project_qkv(b.hidden, w, shape.Nq, shape.Nkv, b.positions, b.query_start_loc, b.activation_offsets,
                                      b.adapter_ids, hp.oracle_adapters(ads))
    odd_cols = [(0, 5, np.inf), (0, 300, -np.inf), (1, 17, np.nan), (2, 100, np.inf), (2, 101, np.nan)]   # block, row of B, value

    def project():
        g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], b.T, b.R, n_adapters=slots)
        try:
            d = hp.DevBatch(b, shape.dtype)
            out = g.empty(b.T, shape.N)
            ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, d.T, d.R, out)
            assert g.status() == 0
            return hp.to_host(out)
        finally:
            g.close()

    finite = project()
    for blk, row, v in odd_cols:
        m = getattr(ads[1], ("Bq", "Bk", "Bv")[blk])
        m[row, 3] = v
    odd = project()
    own = (np.repeat(np.array(ids), each) == 1) & (gate != 0)
    cols = [(0, shape.Nq, shape.Nq + shape.Nkv)[blk] + row for blk, row, _ in odd_cols]
    assert own.any() and (~own).any()
    assert np.array_equal(odd[~own].view(np.uint32), finite[~own].view(np.uint32))
    assert not np.isfinite(odd[own][:, cols]).any()
    others = np.setdiff1d(np.arange(shape.N), cols)
    hp.assert_close(odd[own][:, others], want[own][:, others], 2e-2, "the adapter's own rows")


def test_fp32_projection_of_more_rows_than_one_grid_dimension_holds_tiles(oracle64):
    """The fp32 projection takes 16 rows a tile; 65536 tiles and one row more, a sample of rows against the oracle."""
    import torch
    shape = wl.LayerShape(hidden=32, n_q_heads=1, n_kv_heads=1, head_dim=32, page_size=16, dtype="fp32")
    rng = np.random.default_rng(81)
    T = 16 * 65536 + 1
    w = wl.make_wqkv(shape, rng)
    g = hp.GpuLayers(shape, [dict(wqkv=w)], [[]], T, 1)
    try:
        gen = torch.Generator(device="cuda"); gen.manual_seed(81)
        x = torch.randn(T, shape.hidden, device="cuda", generator=gen)
        out = torch.full((T, shape.N), float("nan"), device="cuda")
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_BASE, x, torch.arange(T, dtype=torch.int32, device="cuda"), None, None,
                             hp.idev([0, T]), hp.idev([T]), T, 1, out)
        assert g.status() == 0
        rows = np.unique(np.concatenate([rng.integers(0, T, 200), [0, T - 17, T - 2, T - 1]]))
        idx = torch.from_numpy(rows).cuda()
        want = oracle64.linear(hp.to_host(x[idx]).astype(np.float64), w)
        hp.assert_close(hp.to_host(out[idx]), want, hp.tol(shape), "rows of a million-row fp32 projection")
        assert bool(torch.isfinite(out).all())
    finally:
        g.close()


@pytest.mark.parametrize("n_req,each,heads,kv_heads,slots", [(9, 12, 4, 2, 3), (9, 12, 4, 2, 5), (100, 1, 16, 4, 200), (20, 30, 4, 2, 3),
                                                             (20, 30, 4, 2, 5), (47, 17, 4, 2, 5), (11, 50, 4, 1, 5)])
def test_projection_of_at_most_1024_rows_loses_nothing_of_t(n_req, each, heads, kv_heads, slots):
    """Whole numbers for which every product and sum is exact in 32 bits, t = A x taking up to 22 of them; the adapters
    subtract one, two and three times rows of the base product.  On every route of few rows (one launch, two, row tiles of
    64, 256 and 128 columns) the result is the exact one, rounded once: t as one or two bf16 values is off by whole numbers
    where the difference is zero."""
    shape = wl.LayerShape(hidden=512, n_q_heads=heads, n_kv_heads=kv_heads, head_dim=128, page_size=16, dtype="bf16")
    rng = np.random.default_rng(91 + n_req)
    whole = lambda *d: rng.integers(-255, 256, d).astype(np.float32)  # noqa: E731
    w = whole(shape.N, shape.hidden)
    starts = (0, shape.Nq, shape.Nq + shape.Nkv)
    ads = []
    for times in (1, 2, 3):
        a = wl.make_adapter(shape, 64, rng)
        for name, s in zip("qkv", starts):
            b_m = np.zeros_like(getattr(a, "B" + name))
            b_m[:64] = -times * np.eye(64, dtype=np.float32)
            setattr(a, "B" + name, b_m)
            setattr(a, "A" + name, w[s:s + 64].copy())
        ads.append(a)
    ids = [(r % 4) - 1 for r in range(n_req)]
    b = wl.make_batch(shape, [40] * n_req, [each] * n_req, ids, rng)
    b.hidden[:] = whole(b.T, shape.hidden)
    y = b.hidden.astype(np.int64) @ w.astype(np.int64).T
    assert np.abs(y).max() * 4 < 2 ** 24
    for s in starts:
        y[:, s:s + 64] *= (1 - (np.repeat(np.array(ids), each) + 1))[:, None]
    g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], b.T, b.R, n_adapters=slots)
    try:
        d = hp.DevBatch(b, shape.dtype)
        out = g.empty(b.T, shape.N)
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, d.T, d.R, out)
        assert g.status() == 0
        got = hp.to_host(out)
    finally:
        g.close()
    assert np.array_equal(got, wl.bf16_round(y.astype(np.float32)))


@pytest.mark.parametrize("S", [[1500, 900, 600, 201], [900, 1200, 700, 600], [700, 1313, 880, 692, 1]])
def test_projection_on_pairs_of_sms(oracle64, S):
    """Batches that the kernel on pairs of SMs serves, four row tiles an item: two, three and one row tiles in the last quad, a
    last tile of one row; column tiles that straddle the q | k | v boundaries, gates that open inside requests.  The cache rows
    of a layer call are those of its sub-steps, and a non-finite B reaches only the rows that use it."""
    shape = wl.LayerShape(hidden=1024, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16")
    rng = np.random.default_rng(101)
    w = wl.make_wqkv(shape, rng)
    ads = _boosted_adapters(shape, rng, ((8, 1.0), (64, 0.5), (32, 2.0)))
    R = len(S)
    ids = ([1, 0, -1, 2, 1])[:R]
    b = wl.make_batch(shape, [20] * R, S, ids, rng, activation_offsets=[150, 20, 20, 220, 20][:R])
    assert (b.T + 127) // 128 in (26, 27, 29)
    _check_projection(oracle64, shape, w, ads, b, on_pairs=True)

    def run():
        g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], b.T, b.R)
        try:
            d = hp.DevBatch(b, shape.dtype)
            fill = np.zeros((b.num_pages, 2, shape.n_kv_heads, shape.page_size, shape.head_dim), np.float32)
            pool, pool2, out, qkv = g.new_pool(b.num_pages, fill), g.new_pool(b.num_pages, fill), g.empty(b.T, shape.Nq), g.empty(b.T, shape.N)
            ab.alora_prefill_layer(g.ctx, 0, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, pool, d.bt, d.max_blocks,
                                   b.num_pages, d.T, d.R, out)
            ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, d.T, d.R, qkv)
            ab.alora_kv_append(g.ctx, qkv, d.positions, d.qsl, d.seq_lens, d.bt, d.max_blocks, b.num_pages, d.T, d.R, pool2)
            assert g.status() == 0
            return hp.to_host(pool), hp.to_host(pool2), hp.to_host(qkv)
        finally:
            g.close()

    pool, pool2, finite = run()
    assert np.array_equal(pool.view(np.uint32), pool2.view(np.uint32))
    ads[0].Bq[7, 3] = np.inf
    ads[0].Bk[100, 2] = np.nan
    pool, pool2, odd = run()
    assert np.array_equal(pool.view(np.uint32), pool2.view(np.uint32))
    own = np.repeat(np.array(ids), S) == 0
    assert np.array_equal(odd[~own].view(np.uint32), finite[~own].view(np.uint32))
    assert not np.isfinite(odd[own][:, [7, shape.Nq + 100]]).any()
    others = np.setdiff1d(np.arange(shape.N), [7, shape.Nq + 100])
    hp.assert_close(odd[own][:, others], finite[own][:, others], 2e-2, "the adapter's own rows")


@pytest.mark.parametrize("n_req,each", [(1, 777), (8, 112), (5, 204)])
def test_projection_of_600_to_1024_rows_on_pairs_of_sms_loses_nothing_of_t(n_req, each):
    """The whole numbers of the test above at the 8B widths, where batches of these sizes with one or two adapters go to the
    pairs of SMs: t takes up to 21 bits, three summands hold it, two would not."""
    shape = wl.SHAPE_8B
    rng = np.random.default_rng(111 + n_req)
    whole = lambda n, *d: rng.integers(-n, n + 1, d).astype(np.float32)  # noqa: E731
    w = whole(63, shape.N, shape.hidden)
    starts = (0, shape.Nq, shape.Nq + shape.Nkv)
    ads = []
    for times in (1, 2)[:1 if n_req == 1 else 2]:
        a = wl.make_adapter(shape, 32, rng)
        for name, s in zip("qkv", starts):
            b_m = np.zeros_like(getattr(a, "B" + name))
            b_m[:32] = -times * np.eye(32, dtype=np.float32)
            setattr(a, "B" + name, b_m)
            setattr(a, "A" + name, w[s:s + 32].copy())
        ads.append(a)
    ids = [r % len(ads) if n_req == 1 else (r % 3) - 1 for r in range(n_req)]
    b = wl.make_batch(shape, [40] * n_req, [each] * n_req, ids, rng)
    b.hidden[:] = whole(255, b.T, shape.hidden)
    y = b.hidden.astype(np.float64) @ w.astype(np.float64).T
    assert 2 ** 18 < np.abs(y[:, :32]).max() and np.abs(y).max() * 4 < 2 ** 24
    for s in starts:
        y[:, s:s + 32] *= (1 - (np.repeat(np.array(ids), each) + 1))[:, None]
    g = hp.GpuLayers(shape, [dict(wqkv=w)], [ads], b.T, b.R)
    try:
        assert ab.alora_selftest_pair_tile(g.ctx, 0, 0, b.T, b.R) > 0
        d = hp.DevBatch(b, shape.dtype)
        out = g.empty(b.T, shape.N)
        ab.alora_project_qkv(g.ctx, 0, ab.MODE_ALORA, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, d.T, d.R, out)
        assert g.status() == 0
        got = hp.to_host(out)
    finally:
        g.close()
    assert np.array_equal(got, wl.bf16_round(y.astype(np.float32)))


@pytest.mark.parametrize("T,inter", [(1, 1096), (17, 2048), (40, 1096), (128, 4744), (200, 2048)])
def test_few_rows_through_gate_and_up_with_swiglu_in_the_epilogue(oracle64, T, inter):
    """One layer of a few rows: gate / up in one launch with SwiGLU, at the row boxes' edges, with a last column tile that is cut
    off (1096, 4744: half tiles of 64 .. 128 columns) and over two row tiles."""
    shape = wl.LayerShape(hidden=1024, n_q_heads=8, n_kv_heads=2, head_dim=128, page_size=16, dtype="bf16", intermediate=inter)
    rng = np.random.default_rng(120 + T)
    layers = [wl.make_stack_weights(shape, rng)]
    b = wl.make_batch(shape, [0], [T], [-1], rng, shuffle_pages=True)
    g = hp.GpuLayers(shape, layers, [[]], T, 1)
    try:
        d = hp.DevBatch(b, shape.dtype)
        hout = g.empty(T, shape.hidden)
        ab.alora_forward_stack(g.ctx, ab.MODE_BASE, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, [g.new_pool(b.num_pages)],
                               d.bt, d.max_blocks, b.num_pages, d.T, d.R, hout)
        assert g.status() == 0
        x, _ = oracle64.decoder_layer(b.hidden.astype(np.float64), layers[0], shape.Nq, shape.Nkv, shape.n_q_heads, shape.n_kv_heads,
                                      shape.head_dim, 1e-5, b.positions, b.query_start_loc, b.activation_offsets, b.adapter_ids, [],
                                      [None], [None])
        hp.assert_close(hp.to_host(hout), x, 2e-2, "a layer of few rows", block=shape.head_dim)
    finally:
        g.close()


@pytest.mark.parametrize("dtype,T,inter", [("bf16", 8, 2048), ("bf16", 200, 2048), ("bf16", 300, 1024), ("bf16", 2048, 2048), ("fp32", 8, 64)])
def test_swiglu_of_large_negative_gates(dtype, T, inter):
    """A gate of -88 with an up value of 2^120: silu(-88) = -5.3e-37 is a normal number, the product -0.71.  On every route of the
    gate / up projection (few rows, pairs of SMs, SwiGLU in a kernel of its own, fp32), with rows of ones that only column 0 of the
    weights reads; the down projection hands every second column of the MLP on."""
    import torch
    H = 1024
    shape = wl.LayerShape(hidden=H, n_q_heads=4, n_kv_heads=2, head_dim=64, page_size=16, dtype=dtype, intermediate=inter)
    lw = dict(wqkv=np.zeros((shape.N, H), np.float32), wo=np.zeros((H, shape.Nq), np.float32), wgate_up=np.zeros((2 * inter, H), np.float32),
              wdown=np.zeros((H, inter), np.float32), norm_attn=np.ones(H, np.float32), norm_mlp=np.ones(H, np.float32))
    lw["wgate_up"][:inter, 0] = -88.0
    lw["wgate_up"][inter:, 0] = 2.0 ** 120
    n = min(H, inter) // 2
    lw["wdown"][2 * np.arange(n), 2 * np.arange(n)] = 1.0
    b = wl.make_batch(shape, [0], [T], [-1], np.random.default_rng(7))
    b.hidden[:] = 1.0
    g = hp.GpuLayers(shape, [lw], [[]], T, 1)
    try:
        d = hp.DevBatch(b, dtype)
        hout = g.empty(T, H)
        ab.alora_forward_stack(g.ctx, ab.MODE_BASE, d.hidden, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens, [g.new_pool(b.num_pages)],
                               d.bt, d.max_blocks, b.num_pages, T, 1, hout)
        assert g.status() == 0
        got = hp.to_host(hout)
    finally:
        g.close()
    want = np.ones((T, H))
    gate, up = -88.0 / np.sqrt(1 + 1e-5), 2.0 ** 120 / np.sqrt(1 + 1e-5)   # (of the norm; bf16 rows read 1)
    if dtype == "bf16":
        gate, up = -88.0, 2.0 ** 120
    want[:, 2 * np.arange(n)] += gate / (1 + np.exp(-gate)) * up
    # bf16: one rounding of the product (2^-9 x 0.71) and one of the sum; fp32: exp of an argument rounded to 2^-18
    assert np.abs(got - want).max() < (4e-3 if dtype == "bf16" else 1e-4)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_stack_input_and_output_buffers(dtype):
    """The stack call reads its input where it is: the same result in a buffer of its own, in place, from rows that are not 16-byte
    aligned (copied first), and from rows that overlap the output in part, on either side (copied through the workspace); the
    input stays as it was unless the output covers it."""
    import torch
    shape = wl.LayerShape(hidden=256, n_q_heads=4, n_kv_heads=2, head_dim=64, page_size=16, dtype=dtype, intermediate=512)
    rng = np.random.default_rng(131)
    layers = [wl.make_stack_weights(shape, rng) for _ in range(2)]
    b = wl.make_batch(shape, [0, 0], [30, 21], [-1, -1], rng)
    g = hp.GpuLayers(shape, layers, [[], []], b.T, b.R)
    try:
        d = hp.DevBatch(b, dtype)
        x, n = d.hidden.clone(), b.T * shape.hidden

        def run(src, dst):
            ab.alora_forward_stack(g.ctx, ab.MODE_BASE, src, d.positions, d.a_req, d.ids, d.qsl, d.seq_lens,
                                   [g.new_pool(b.num_pages) for _ in range(2)], d.bt, d.max_blocks, b.num_pages, d.T, d.R, dst)
            assert g.status() == 0
            return dst.clone()

        want = run(x, g.empty(b.T, shape.hidden))
        assert torch.equal(x, d.hidden) and not torch.equal(want, x)
        y = x.clone()
        assert torch.equal(run(y, y), want)
        buf = torch.empty(n + 8192, dtype=x.dtype, device="cuda")
        src, dst = buf[1:1 + n].view(b.T, -1), torch.empty_like(x)
        src.copy_(x)
        assert torch.equal(run(src, dst), want) and torch.equal(src, x)
        for at_src, at_dst in ((0, 8), (8, 0), (1, 8), (9, 0), (0, 4096), (4096, 0)):   # elements into the buffer
            src, dst = buf[at_src:at_src + n].view(b.T, -1), buf[at_dst:at_dst + n].view(b.T, -1)
            src.copy_(x)
            assert torch.equal(run(src, dst), want), (at_src, at_dst)
        # an output that is not aligned: fp32 rows are stored element by element, bf16 rows are refused before any launch
        src, dst = x.clone(), buf[1:1 + n].view(b.T, -1)
        if dtype == "fp32":
            assert torch.equal(run(src, dst), want)
        else:
            launches = ab.alora_launch_count(g.ctx)
            with pytest.raises(ab.AloraError) as e:
                run(src, dst)
            assert e.value.status == 1 and ab.alora_launch_count(g.ctx) == launches
    finally:
        g.close()
