"""The calls that users of this library make, as timing cases: one activated-LoRA layer or a few decoder layers, through the
public entry points of the binding.

A case is a dict of plain values:
  call         prefill_layer | decode_step | full_prefill_layer | forward_stack | decode_stack
  shape        a key of SHAPES; `page` overrides its page size
  requests     requests in the batch; `prefix` cached positions and `new` new tokens each, "lo..hi" = uniform over that range
  lengths      seed of the lengths and of the adapter of every request (sizes belong to the case, values to prepare()'s seed)
  ranks        ranks of the registered adapters, comma separated; "" = base model only
  base_share   share of the requests that run on the base model alone
  into_chunk   tokens of the new chunk that lie before the activation offset
  sharers      neighbouring requests whose block tables begin with the same cached pages (N adapters on one conversation)
  layers, mlp_adapters, rope   stack depth, adapters on gate / up / down as well, rotary option
"""
import random

import torch

from paper_2504_12397_b200 import binding as ab
from paper_2504_12397_b200.workloads import SHAPE_8B, TINY, LayerShape

# the 8B layer shape of the benchmark, the tiny exact-precision layer, and a narrower layer with head dim 64
SHAPES = {"8b": SHAPE_8B, "tiny": TINY,
          "narrow": LayerShape(hidden=2048, n_q_heads=32, n_kv_heads=8, head_dim=64, dtype="bf16", intermediate=8192)}
ROPE_THETA = 10000.0


def _case(name, call, requests, prefix, new, shape="8b", page=16, lengths=1, ranks="32", base_share=0.0, into_chunk=0,
          sharers=1, layers=1, mlp_adapters=False, rope=False):
    c = dict(call=call, shape=shape, page=page, requests=requests, prefix=prefix, new=new, lengths=lengths, ranks=ranks,
             base_share=base_share, into_chunk=into_chunk, sharers=sharers, layers=layers, mlp_adapters=mlp_adapters, rope=rope)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: the tiny fp32 layer on which numerics are pinned; latency only
        _case("tiny_fp32_suffix", "prefill_layer", 1, "64..64", "16..16", shape="tiny", ranks="8"),
        # an intrinsic invoked on a few conversations: a short invocation sequence each
        _case("invoke_8x16", "prefill_layer", 8, "4096..4096", "16..16"),
        # an invocation of every waiting request: a handful of tokens each, odd lengths, mixed with base requests
        _case("invoke_48_ragged", "prefill_layer", 48, "700..9000", "3..29", ranks="8,16,32,64", base_share=0.1, lengths=12),
        # the benchmark's layer call: suffix prefill on a reused base cache
        _case("suffix_8x256", "prefill_layer", 8, "4096..4096", "256..256"),
        # a serving batch of requests of all sizes over four adapters, pages scattered over the pool
        _case("suffix_ragged_32", "prefill_layer", 32, "512..16384", "16..512", ranks="8,16,32,64", lengths=3),
        # an uncached tail of the context and the invocation in one chunk, rotary positions, one long conversation
        _case("tail_then_invoke_rope", "prefill_layer", 1, "20011..20011", "777..777", into_chunk=650, rope=True),
        # the narrower layer with head dim 64 and larger pages, medium batch
        _case("narrow_16", "prefill_layer", 16, "256..3000", "5..150", shape="narrow", page=32, ranks="16,32", lengths=7),
        # generation after activation: 64 requests of very different lengths, base model and four adapters
        _case("decode_64", "decode_step", 64, "1023..32767", "1..1", ranks="32,32,32,32", base_share=0.2, lengths=5),
        # filling the base cache that everything else reuses
        _case("base_prefill_8x4096", "full_prefill_layer", 8, "0..0", "4096..4096", ranks=""),
        # long documents through whole layers: 32K cached, 1K new
        _case("stack_4x1024_on_32k", "forward_stack", 4, "32768..32768", "1024..1024", layers=2),
        # the 8K-prefix comparison with adapters on the MLP block too
        _case("stack_mlp_8x256_on_8k", "forward_stack", 8, "8192..8192", "256..256", layers=2, mlp_adapters=True),
        # five evaluators each on eight conversations, one decode step through whole layers
        _case("evaluators_decode_40", "decode_stack", 40, "4352..4368", "1..1", ranks="32,32,32,32,32", sharers=5, layers=4,
              lengths=9),
    ]


def _log(rng, lo, hi):
    """A whole number of [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    kind = rng.choice(("prefill", "prefill", "prefill", "few", "decode", "decode", "base", "stack", "decode_stack", "tiny"))
    seed = rng.randrange(1, 1 << 20)
    ranks = ",".join(str(rng.choice((8, 16, 32, 64))) for _ in range(rng.randint(1, 4)))
    base = rng.choice((0.0, 0.0, 0.25))
    shape, page = rng.choice((("8b", 16), ("8b", 16), ("8b", 32), ("narrow", 16), ("narrow", 64)))

    def span(lo, hi):   # a ragged batch: lengths between a part of the largest and the largest
        top = _log(rng, lo, hi)
        return "%d..%d" % (max(lo, rng.choice((top, top // 2, top // 8))), top)

    if kind == "tiny":
        return _case(None, "prefill_layer", rng.randint(1, 4), span(16, 200), span(2, 40), shape="tiny", ranks="8", lengths=seed,
                     base_share=base)
    if kind == "base":
        return _case(None, "full_prefill_layer", _log(rng, 1, 8), "0..0", span(100, 4096), shape=shape, page=page, lengths=seed,
                     ranks=rng.choice(("", "16,32")))
    if kind == "decode":
        return _case(None, "decode_step", _log(rng, 1, 96), span(100, 20000), "1..1", shape=shape, page=page, ranks=ranks,
                     base_share=base, lengths=seed, rope=rng.random() < 0.25)
    if kind == "decode_stack":
        sharers = rng.choice((1, 2, 5))
        return _case(None, "decode_stack", sharers * _log(rng, 1, 8), span(500, 8000), "1..1", page=page, ranks=ranks,
                     base_share=base, sharers=sharers, layers=2, lengths=seed)
    if kind == "stack":
        return _case(None, "forward_stack", _log(rng, 1, 8), span(500, 16384), span(16, 512), page=page, ranks=ranks,
                     base_share=base, layers=2, lengths=seed, mlp_adapters=rng.random() < 0.3)
    if kind == "few":
        return _case(None, "prefill_layer", _log(rng, 1, 64), span(500, 16384), span(2, 32), shape=shape, page=page, ranks=ranks,
                     base_share=base, lengths=seed, rope=rng.random() < 0.25)
    new_hi = _log(rng, 33, 1024)
    return _case(None, "prefill_layer", _log(rng, 1, 32), span(500, 16384), "%d..%d" % (new_hi // 3, new_hi), shape=shape, page=page,
                 ranks=ranks, base_share=base, lengths=seed, into_chunk=rng.choice((0, 0, new_hi // 4)), rope=rng.random() < 0.25)


class _Sizes:
    """What a case says about its batch: the layer shape, the adapters, and per request lengths and adapter."""

    def __init__(self, c):
        s = SHAPES[c["shape"]]
        self.shape = LayerShape(s.hidden, s.n_q_heads, s.n_kv_heads, s.head_dim, c["page"], s.dtype, s.intermediate)
        self.ranks = [int(r) for r in c["ranks"].split(",") if r]
        rng = random.Random(c["lengths"])
        R, per = c["requests"], c["sharers"]
        among = lambda text: rng.randint(*(int(x) for x in text.split("..")))  # noqa: E731
        common = [among(c["prefix"]) for _ in range(-(-R // per))]              # one length per conversation
        self.prefix = [common[r // per] for r in range(R)]
        self.new = [among(c["new"]) for _ in range(R)]
        self.ids = [-1 if not self.ranks or rng.random() < c["base_share"] else
                    (r % per if per > 1 else rng.randrange(1 << 20)) % len(self.ranks) for r in range(R)]
        self.T = sum(self.new)
        # cached positions that the batch reads: those of a conversation once, however many requests share them
        self.cached = sum(common)


def work(case):
    z = _Sizes(case)
    s, L = z.shape, case["layers"]
    e = 4 if s.dtype == "fp32" else 2
    stack = case["call"].endswith("stack")
    used = [z.ranks[i] for i in sorted({i for i in z.ids if i >= 0})]
    on = case["call"] != "full_prefill_layer" and case["into_chunk"]
    lora_rows = [(n - min(n, on or 0), z.ranks[i]) for n, i in zip(z.new, z.ids) if i >= 0]
    elems = s.N * s.hidden + sum(r * (3 * s.hidden + s.N) for r in used) + 2 * s.Nkv * (z.cached + z.T)
    flops = 2.0 * z.T * s.hidden * s.N + sum(2.0 * n * r * (3 * s.hidden + s.N) for n, r in lora_rows)
    flops += 4.0 * s.Nq * sum(n * p + n * (n + 1) / 2 for n, p in zip(z.new, z.prefix))
    if stack:
        H, F = s.hidden, s.intermediate
        elems += H * s.Nq + 3 * H * F + 2 * H
        flops += 2.0 * z.T * (H * s.Nq + 3 * H * F)
        if case["mlp_adapters"]:
            elems += sum(3 * r * (H + F) for r in used)
            flops += sum(6.0 * n * r * (H + F) for n, r in lora_rows)
    ends = 2 * z.T * s.hidden if stack else z.T * (s.hidden + s.Nq)
    return {"bytes": e * (L * elems + ends), "flops": L * flops}


def tolerance(case):
    # Against the same path restated in float64: fp32 layers rel 3e-7, max 2e-6; bf16 layers rel 0.003 .. 0.005, max
    # 0.02 .. 0.14 (rows of few visible keys); 2 .. 4 whole layers rel 0.007 .. 0.010, max 0.03 .. 0.05.
    if SHAPES[case["shape"]].dtype == "fp32":
        return {"rel": 2e-6, "max": 1e-5}
    if case["call"].endswith("stack"):
        return {"rel": 0.028, "max": 0.2}
    return {"rel": 0.016, "max": 0.4}


class _State:
    """A context with its weights and adapters, a page pool per layer, and one batch, all on the device."""

    def __init__(self, case, seed):
        z = _Sizes(case)
        s, L, R = z.shape, case["layers"], case["requests"]
        dt = torch.float32 if s.dtype == "fp32" else torch.bfloat16
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        stack = case["call"].endswith("stack")
        H, F = s.hidden, s.intermediate
        self.ctx = None
        self.case, self.T, self.R = case, z.T, R

        def normal(*dims, std=0.02, mean=0.0):
            return torch.empty(dims, device="cuda", dtype=dt).normal_(mean, std, generator=g)

        self.ctx = ab.alora_create(ab.make_config(
            hidden=H, n_q_heads=s.n_q_heads, n_kv_heads=s.n_kv_heads, head_dim=s.head_dim, page_size=s.page_size, n_layers=L,
            intermediate=F if stack else 0, max_adapters=max(1, len(z.ranks)), max_rank=max(z.ranks + [8]),
            dtype=ab.DTYPE_FP32 if s.dtype == "fp32" else ab.DTYPE_BF16, max_tokens=z.T, max_requests=R,
            rope_theta=ROPE_THETA if case["rope"] else 0.0))
        self.weights = []
        for layer in range(L):
            w = [normal(s.N, H)]
            if stack:
                w += [normal(H, s.Nq), normal(2 * F, H), normal(H, F), normal(H, mean=1.0, std=0.1), normal(H, mean=1.0, std=0.1)]
            self.weights.append(w)
            ab.alora_set_layer_weights(self.ctx, layer, *w)
            for i, r in enumerate(z.ranks):   # copied by the library
                ab.alora_register_adapter(self.ctx, i, layer, r, 1.0, normal(r, H), normal(s.Nq, r), normal(r, H), normal(s.Nkv, r),
                                          normal(r, H), normal(s.Nkv, r))
                if case["mlp_adapters"]:
                    ab.alora_register_mlp_adapter(self.ctx, i, layer, r, 1.0, normal(r, H), normal(F, r), normal(r, H), normal(F, r),
                                                  normal(r, F), normal(H, r))

        # block tables: pages handed out in random order; the sharers of a conversation name the same pages up to
        # the page that holds their first new position (its cached rows are theirs after the copy-on-write)
        ps, per = s.page_size, case["sharers"]
        blocks = [-(-(p + n) // ps) for p, n in zip(z.prefix, z.new)]
        common = [p // ps if r % per else 0 for r, p in enumerate(z.prefix)]
        self.max_blocks, self.num_pages = max(blocks), sum(b - k for b, k in zip(blocks, common)) + 3
        order = torch.randperm(self.num_pages, generator=torch.Generator().manual_seed(seed)).to(torch.int32)
        tables, at = torch.zeros(R, self.max_blocks, dtype=torch.int32), 0
        for r in range(R):
            k, own = common[r], blocks[r] - common[r]
            tables[r, :k] = tables[r - r % per, :k]
            tables[r, k:k + own] = order[at:at + own]
            at += own
        ints = lambda v: torch.tensor(v, dtype=torch.int32).cuda()  # noqa: E731
        starts = [0]
        for n in z.new:
            starts.append(starts[-1] + n)
        self.tables, self.qsl = tables.cuda(), ints(starts)
        self.positions = ints([p + i for p, n in zip(z.prefix, z.new) for i in range(n)])
        self.seq_lens = ints([p + n for p, n in zip(z.prefix, z.new)])
        self.a_req = ints([p + min(case["into_chunk"], n) for p, n in zip(z.prefix, z.new)])
        self.ids = ints(z.ids)
        self.pools = [normal(self.num_pages, 2, s.n_kv_heads, ps, s.head_dim, std=1.0) for _ in range(L)]
        self.hidden = normal(z.T, H, std=1.0)
        self.out = torch.empty(z.T, H if stack else s.Nq, device="cuda", dtype=dt)
        torch.cuda.synchronize()   # the adapters' source matrices may go now

    def __del__(self):
        if self.ctx is not None:
            ab.alora_destroy(self.ctx)


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    """One call; the outputs are the attention rows (of a stack: the hidden states) and the page pools with the new K/V rows."""
    s, call = state, state.case["call"]
    if call == "prefill_layer":
        ab.alora_prefill_layer(s.ctx, 0, s.hidden, s.positions, s.a_req, s.ids, s.qsl, s.seq_lens, s.pools[0], s.tables,
                               s.max_blocks, s.num_pages, s.T, s.R, s.out)
    elif call == "decode_step":
        ab.alora_decode_step(s.ctx, 0, s.hidden, s.positions, s.a_req, s.ids, s.seq_lens, s.pools[0], s.tables, s.max_blocks,
                             s.num_pages, s.R, s.out)
    elif call == "full_prefill_layer":
        ab.alora_full_lora_prefill_layer(s.ctx, 0, s.hidden, s.positions, s.ids, s.qsl, s.seq_lens, s.pools[0], s.tables,
                                         s.max_blocks, s.num_pages, s.T, s.R, s.out)
    elif call == "forward_stack":
        ab.alora_forward_stack(s.ctx, ab.MODE_ALORA, s.hidden, s.positions, s.a_req, s.ids, s.qsl, s.seq_lens, s.pools, s.tables,
                               s.max_blocks, s.num_pages, s.T, s.R, s.out)
    else:
        ab.alora_decode_stack(s.ctx, s.hidden, s.positions, s.a_req, s.ids, s.seq_lens, s.pools, s.tables, s.max_blocks,
                              s.num_pages, s.R, s.out)
    return {"out": s.out, "pools": s.pools}
