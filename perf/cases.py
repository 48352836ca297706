"""What is timed: the calls a serving program makes of libdkv, as cases with seeded inputs.

A case names one use of the library and its shape (the fields of ``dkv_config``); the uses are

``pass``    a prompt whose layers' queries, keys and values are all on the GPU is compressed with
            ``dkv_run_prefill_pass``, and its first new token attends to the result (``dkv_decode_attend``)
``lse``     the same where the prefill attention kernel has left the window rows' log-denominators
            (``dkv_run_prefill_pass_lse``)
``layers``  the same call by call, as a program does whose layers become available one after another:
            score, select, gather each layer, update and shrink every m layers
``host``    ``dkv_run_prefill_pass_host``: everything in pinned host memory, compressed buffers back in it
``decode``  one decoding step over a compressed cache, ``per_call`` layers to a call, ``nq`` queries a sample

``prepare`` makes the inputs and the context, ``run`` is one pass over them.
"""
import math

import torch

from paper_2412_14838_b200 import binding as B

#: The shape fields of a case, in the order of ``binding.make_config``.
SHAPE = ("L", "Hq", "Hkv", "D", "Bt", "S", "ws", "pool", "N", "Bl", "m")


def _case(name, use, L, Hq, Hkv, D, Bt, S, ws, pool, N, Bl, m, nq=1, per_call=0):
    c = dict(use=use, L=L, Hq=Hq, Hkv=Hkv, D=D, Bt=Bt, S=S, ws=ws, pool=pool, N=N, Bl=Bl, m=m, nq=nq,
             per_call=per_call or L)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest configuration of the benchmark: a short prompt of a small model, where the time is latency
        _case("pass_tiny", "pass", 4, 8, 2, 64, 1, 1024, 16, 5, 64, 128, 2),
        # one 8K prompt of a 32-layer model with 32/8 heads: the ordinary chat or retrieval request
        _case("pass_8k", "pass", 32, 32, 8, 128, 1, 8192, 32, 7, 128, 512, 4),
        # one 32K document with the large budget: the benchmark's default workload
        _case("pass_32k", "pass", 32, 32, 8, 128, 1, 32768, 32, 7, 512, 2048, 4),
        # a batch of four 16K prompts compressed hard: the most keys of all
        _case("pass_16k_b4", "pass", 32, 32, 8, 128, 4, 16384, 32, 7, 64, 256, 4),
        # 28/4 heads: seven query heads share a KV head, 224 window rows, few KV heads
        _case("pass_16k_g7", "pass", 28, 28, 4, 128, 1, 16384, 32, 7, 128, 512, 4),
        # odd sizes throughout: three prompts padded to 5003, 18/6 heads of 64, window 24, L not a multiple of m
        _case("pass_ragged", "pass", 14, 18, 6, 64, 3, 5003, 24, 5, 100, 330, 4),
        # a 32K prompt with a small budget, log-denominators at hand
        _case("lse_32k", "lse", 32, 32, 8, 128, 1, 32768, 32, 7, 64, 512, 4),
        # compression interleaved with the model's own prefill: every call on its own
        _case("layers_16k", "layers", 32, 32, 8, 128, 1, 16384, 32, 7, 128, 512, 4),
        # caches kept in host memory (offloading): a 4K prompt through the bus and back
        _case("host_4k", "host", 32, 32, 8, 128, 1, 4096, 32, 7, 128, 512, 4),
        # generation after a 32K prompt, layer by layer as a model's forward goes
        _case("decode_layers", "decode", 32, 32, 8, 128, 1, 32768, 32, 7, 512, 2048, 4, 1, 1),
        # generation for four sequences with small caches, all layers in one call
        _case("decode_b4", "decode", 32, 32, 8, 128, 4, 16384, 32, 7, 64, 256, 4, 1, 32),
        # four drafted tokens per step verified against the large cache
        _case("decode_nq4", "decode", 32, 32, 8, 128, 1, 32768, 32, 7, 512, 2048, 4, 4, 32),
    ]


#: The most keys (L * Bt * Hkv * S * D values) a drawn case of each use has: no more than the largest listed one.
_MOST = {"pass": 32 * 4 * 8 * 16384 * 128, "lse": 32 * 8 * 32768 * 128, "layers": 32 * 8 * 16384 * 128,
         "host": 32 * 8 * 4096 * 128, "decode": 32 * 8 * 32768 * 128}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    use = rng.choice(["pass", "pass", "pass", "lse", "layers", "host", "decode", "decode"])
    while True:
        L, Bt, Hkv = _log_int(rng, 4, 32), rng.choice([1, 1, 1, 2, 3, 4]), rng.choice([2, 4, 6, 8])
        D, G = rng.choice([64, 128, 128]), rng.choice([1, 2, 3, 4, 4, 7, 8])
        S, ws = _log_int(rng, 700, 32768), rng.choice([8, 16, 24, 32, 32])
        if L * Bt * Hkv * S * D <= _MOST[use]:
            break
    N = _log_int(rng, 32, max(32, min(512, S // 8)))
    nq = rng.choice([1, 1, 2, 4]) if use == "decode" else 1
    per_call = rng.choice([1, L]) if use == "decode" else L
    return _case("", use, L, G * Hkv, Hkv, D, Bt, S, ws, rng.choice([3, 5, 7]), N, int(N * rng.choice([2.0, 3.3, 4.0])),
                 rng.choice([2, 3, 4, 8]), nq, per_call)


class _Context:
    """The library's context; its memory lives as long as this object."""

    def __init__(self, config):
        self.handle = B.dkv_create(config)

    def __del__(self):
        if getattr(self, "handle", None):
            B.dkv_destroy(self.handle)


class _LayerScores:
    """A layer's scores inside the context, for torch, which holds this object (and with it the context) as long as
    a tensor shows them."""

    def __init__(self, context, layer, shape):
        self.context = context
        self.__cuda_array_interface__ = {"data": (B.dkv_layer_views(context.handle, layer)[0], False), "shape": shape,
                                         "typestr": "<f4", "version": 3}


class State:
    """What a program keeps: the context, its tensors and the lists of per-layer tensors it passes on."""

    def __init__(self, case):
        for f in SHAPE:
            setattr(self, f, case[f])
        self.use, self.nq, self.per_call = case["use"], case["nq"], case["per_call"]
        self.G, self.P = self.Hq // self.Hkv, self.S - self.ws
        self.rows = min(self.Bl, self.P) + self.ws
        self.context = _Context(B.make_config(*(case[f] for f in SHAPE)))
        self.ctx = self.context.handle


def _draw_prompt(s, g, on_layer):
    """Queries of the window, keys and values of every layer, bf16, handed to ``on_layer(l, q, k, v)``.

    Keys are normal with four outlier channels (x8) per head, the first four are attention sinks aligned with
    the mean query, and in every layer another share of them correlates with the queries to another degree, so
    that the layers deserve different budgets."""
    dev = "cuda"
    cut = torch.rand((s.L, 2), generator=g, device=dev).tolist()
    for l in range(s.L):
        kv = (s.Bt, s.Hkv, s.S, s.D)
        k = torch.randn(kv, generator=g, device=dev, dtype=torch.bfloat16)
        v = torch.randn(kv, generator=g, device=dev, dtype=torch.bfloat16)
        mu = torch.randn((s.Bt, s.Hkv, 1, s.D), generator=g, device=dev)
        channels = torch.rand((s.Hkv, s.D), generator=g, device=dev).topk(4, dim=1).indices
        scale = torch.ones((s.Hkv, s.D), device=dev).scatter_(1, channels, 8.0).to(torch.bfloat16)
        k *= scale[None, :, None, :]
        share, c = cut[l][0] * min(0.125, 4096 / s.P), 0.6 * cut[l][1]
        hot = torch.rand((s.Bt, s.Hkv, s.S, 1), generator=g, device=dev) < share
        toward = c * math.sqrt(s.D) * mu / mu.norm(dim=-1, keepdim=True)
        k = torch.where(hot, math.sqrt(1 - c * c) * k + toward.to(torch.bfloat16), k)
        k[:, :, :4] = mu.to(torch.bfloat16)
        q = torch.randn((s.Bt, s.Hq, s.ws, s.D), generator=g, device=dev) + mu.repeat_interleave(s.G, dim=1)
        on_layer(l, q.to(torch.bfloat16), k, v)


def _log_denominators(s, q, k):
    """ln sum exp of the window rows' scaled logits over the keys each row sees, fp32 [Bt, Hq, ws]."""
    logits = torch.matmul(q.float().view(s.Bt, s.Hkv, s.G * s.ws, s.D), k.float().transpose(-1, -2))
    logits = logits.view(s.Bt, s.Hq, s.ws, s.S) / math.sqrt(s.D)
    last = s.P + torch.arange(s.ws, device="cuda")
    logits.masked_fill_(torch.arange(s.S, device="cuda") > last[:, None], -math.inf)
    return torch.logsumexp(logits, dim=-1)


def _budget_buffers(s, **kw):
    """K and V budget buffers [L, Bt, Hkv, rows, D] as 16-bit patterns, and their per-layer tensors."""
    shape = (s.L, s.Bt, s.Hkv, s.rows, s.D)
    s.kb_all, s.vb_all = (torch.zeros(shape, dtype=torch.int16, **kw) for _ in range(2))
    s.kb, s.vb = list(s.kb_all), list(s.vb_all)


def _decode_tensors(s, g):
    """One decoding step's queries (normal plus a common direction) and its fp32 results, all layers."""
    shape = (s.L, s.Bt, s.Hq, s.nq, s.D)
    dq = torch.randn(shape, generator=g, device="cuda") + torch.randn((s.L, s.Bt, s.Hq, 1, s.D), generator=g, device="cuda")
    s.dq_all = dq.to(torch.bfloat16)
    s.attn = torch.zeros(shape, dtype=torch.float32, device="cuda")
    s.dq, s.out = list(s.dq_all), list(s.attn)


def _prepare_resident(s, g):
    s.q = [None] * s.L
    s.k, s.v, s.lse = list(s.q), list(s.q), list(s.q)

    def on_layer(l, q, k, v):
        s.q[l], s.k[l], s.v[l] = q, k, v
        if s.use == "lse":
            s.lse[l] = _log_denominators(s, q, k)

    _draw_prompt(s, g, on_layer)
    _budget_buffers(s, device="cuda")
    _decode_tensors(s, g)
    if s.use == "layers":                                    # the program asks for its own copy of the scores
        s.scores = [torch.zeros((s.Bt, s.Hkv, s.P), dtype=torch.float32, device="cuda") for _ in range(s.L)]
    else:                                                    # the scores stay in the context
        s.scores = [torch.as_tensor(_LayerScores(s.context, l, (s.Bt, s.Hkv, s.P)), device="cuda") for l in range(s.L)]


def _prepare_host(s, g):
    q = torch.empty((s.L, s.Bt, s.Hq, s.ws, s.D), dtype=torch.bfloat16, pin_memory=True)
    k, v = (torch.empty((s.L, s.Bt, s.Hkv, s.S, s.D), dtype=torch.bfloat16, pin_memory=True) for _ in range(2))

    def on_layer(l, *layer):
        for dst, src in zip((q, k, v), layer):
            dst[l].copy_(src, non_blocking=True)

    _draw_prompt(s, g, on_layer)
    torch.cuda.synchronize()
    s.q, s.k, s.v = list(q), list(k), list(v)
    _budget_buffers(s, pin_memory=True)
    s.counts = torch.zeros((s.Bt, s.L), dtype=torch.int32)


def _prepare_cache(s, g):
    """A compressed cache as a prompt leaves it: the budgets come from given scores (log-normal with a spread of
    its own per layer, max-pooled), the rows are random."""
    _budget_buffers(s, device="cuda")
    _decode_tensors(s, g)
    spread = (1.0 + torch.rand((s.L,), generator=g, device="cuda")).tolist()
    for l in range(s.L):
        raw = torch.randn((s.Bt, s.Hkv, s.P), generator=g, device="cuda").mul_(spread[l]).sub_(8.0).exp_()
        B.dkv_set_scores(s.ctx, l, torch.nn.functional.max_pool1d(raw, s.pool, 1, s.pool // 2))
        B.dkv_select_topk(s.ctx, l)
        k, v = (torch.randn((s.Bt, s.Hkv, s.S, s.D), generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(2))
        B.dkv_compact(s.ctx, l, k, v, s.kb[l], s.vb[l])
    B.dkv_rebudget(s.ctx, s.L)
    B.dkv_compact_all(s.ctx, s.L, s.kb, s.vb)


def prepare(case, seed):
    s = State(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    {"pass": _prepare_resident, "lse": _prepare_resident, "layers": _prepare_resident, "host": _prepare_host,
     "decode": _prepare_cache}[s.use](s, g)
    return s


def _first_token(s):
    B.dkv_decode_attend(s.ctx, 0, s.L, s.nq, s.dq, s.kb, s.vb, s.out)
    return {"scores": s.scores, "attn": s.attn}


def run(s):
    if s.use == "pass":
        B.dkv_run_prefill_pass(s.ctx, s.q, s.k, s.v, s.kb, s.vb)
        return _first_token(s)
    if s.use == "lse":
        B.dkv_run_prefill_pass_lse(s.ctx, s.q, s.k, s.v, s.lse, s.kb, s.vb)
        return _first_token(s)
    if s.use == "layers":
        B.dkv_reset(s.ctx)
        for l in range(s.L):
            B.dkv_score(s.ctx, l, s.q[l], s.k[l], s.scores[l])
            B.dkv_select_topk(s.ctx, l)
            B.dkv_compact(s.ctx, l, s.k[l], s.v[l], s.kb[l], s.vb[l])
            if (l + 1) % s.m == 0 or l + 1 == s.L:
                B.dkv_rebudget(s.ctx, l + 1)
                B.dkv_compact_all(s.ctx, l + 1, s.kb[:l + 1], s.vb[:l + 1])
        return _first_token(s)
    if s.use == "host":
        B.dkv_run_prefill_pass_host(s.ctx, s.q, s.k, s.v, s.kb, s.vb, s.counts)
        return {"counts": s.counts, "kb": s.kb_all, "vb": s.vb_all}
    for l in range(0, s.L, s.per_call):
        n = min(s.per_call, s.L - l)
        B.dkv_decode_attend(s.ctx, l, n, s.nq, s.dq[l:l + n], s.kb[l:l + n], s.vb[l:l + n], s.out[l:l + n])
    return {"attn": s.attn}


def work(case):
    """Bytes: q and K read once, the kept rows (N + ws a head and layer on average) of V read and of K and V
    written once, the scores written once; in a decoding step the kept rows, the queries and the results.
    Operations: one contraction of the window rows with the keys, and the decoding step's two."""
    L, Hq, Hkv, D, Bt, S, ws, N, nq = (case[f] for f in ("L", "Hq", "Hkv", "D", "Bt", "S", "ws", "N", "nq"))
    heads, kept = L * Bt * Hkv, min(N, S - ws) + ws
    decode_flops = 4 * L * Bt * Hq * nq * kept * D
    decode_io = L * Bt * Hq * nq * D * (2 + 4)
    if case["use"] == "decode":
        return {"bytes": heads * kept * D * 2 * 2 + decode_io, "flops": decode_flops}
    scoring = heads * (S * D * 2 + kept * D * 2 * 3) + L * Bt * Hq * ws * D * 2
    flops = 2 * L * Bt * Hq * ws * S * D
    if case["use"] == "host":
        return {"bytes": scoring, "flops": flops}
    return {"bytes": scoring + heads * (S - ws) * 4 + decode_io, "flops": flops + decode_flops}


def tolerance(case):
    if case["use"] == "decode":                              # 32-bit sums over rows that are given exactly
        return {"rel": 1e-5, "max": 1e-3}
    if case["use"] == "host":                                # rows are copies; their order follows 32-bit scores,
        return {"rel": 0.0, "differ": 0.01}                  # so that rows whose scores are nearly equal may swap
    return {"rel": 1e-2, "max": 0.5}                         # the same: a near-tie at a cut keeps another row
