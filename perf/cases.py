"""Performance cases of the BalanceKV library: what a program that uses it has it do.

A case is a dict of plain values.  Its ``kind`` names the way the library is used:

``prefill``   a context that serves one request after another: reset, append the prompt's keys and
              values (chunk by chunk, layer by layer), compress, and attend for the first tokens;
``decode``    one token's attention over every layer of an already compressed cache;
``generate``  a turn: load the compressed prefix and its recent window, then token by token the fused
              append + attend step of every layer;
``routed``    Algorithm 1 in full (value-norm buckets and the separate denominator instance), or the
              variant that preserves anti-correlated keys, each with the decode merged over its slots;
``static``    the allocation-free decode over caches that the caller owns;
``host``      prefill and decode steps on host buffers.

Sizes are those of the repository's workloads (one 8B-shaped layer, the 8B-shaped stack, the 14B-shaped
layer with a recent window, the decode sweep of the 32B shape, the tiny fp32 stream) or generic ones.
Timings are those of a serving loop: a context and its inputs exist, a pass is one request (or one token).
"""
from __future__ import annotations

import math

import torch

import paper_2502_07861_b200 as bk

_PREFILL = dict(kind="prefill", batch=1, layers=1, kv_heads=8, group=4, head_dim=128, dtype="bf16", block=1024, levels=2,
                window=0, context=8192, chunk=8192, per_layer=False, center=False, keys="llama", queries=1)
_DECODE = dict(kind="decode", batch=1, layers=1, kv_heads=8, group=4, head_dim=128, dtype="bf16", levels=2, rows=8192, tail=0)
_GENERATE = dict(kind="generate", batch=1, layers=4, kv_heads=8, group=4, head_dim=128, dtype="bf16", block=1024, levels=2,
                 rows=8192, tail=64, steps=16)
_ROUTED = dict(kind="routed", route="buckets", batch=1, kv_heads=8, group=4, head_dim=128, block=1024, levels=2,
               context=16384, buckets=4)
_STATIC = dict(kind="static", streams=16, layers=4, group=4, head_dim=128, dtype="bf16", rows=4096, tail=0, levels=2)
_HOST = dict(kind="host", batch=1, kv_heads=8, group=4, head_dim=128, block=1024, levels=2, context=8192, steps=32)


def listed():
    return [
        # a small model's single head in fp32, streamed in blocks of 256 and asked 16 queries: latency and launches
        dict(_PREFILL, name="tiny_fp32_stream", kv_heads=1, group=1, head_dim=64, dtype="fp32", block=256, levels=1,
             context=1024, chunk=256, keys="outlier2", queries=16),
        # one layer of an 8B-shaped model: a 32k prompt appended at once, compressed 4x, first token
        dict(_PREFILL, name="layer_8b_prefill", context=32768, chunk=32768),
        # half of the 8B-shaped stack, four sequences, two prefill chunks of 8192 with one compress each: the largest
        dict(_PREFILL, name="stack_8b_chunks", batch=4, layers=16, block=2048, context=16384, chunk=8192),
        # layers of a 14B-shaped model, eight sequences, an exact recent window, heavy-tailed keys, a prompt that is
        # no multiple of anything, compressed layer by layer as a forward pass reaches them
        dict(_PREFILL, name="layers_14b_window", batch=8, layers=4, group=5, levels=3, window=128, context=20011,
             chunk=8192, per_layer=True, keys="student_t"),
        # fp32 caches at d = 128 with shorter blocks
        dict(_PREFILL, name="layers_fp32", layers=2, dtype="fp32", block=512, context=8192, chunk=4096, queries=4),
        # small heads (d = 64) with the key mean shift and a block that is no power of two
        dict(_PREFILL, name="small_heads_centered", layers=2, group=8, head_dim=64, block=192, context=8000, chunk=4000,
             center=True, queries=4),
        # a token of a large batch at the 32B shape: two layers of 16384 kept rows for 32 sequences
        dict(_DECODE, name="decode_32b_batch", batch=32, layers=2, group=5, levels=3, rows=16384),
        # a token of a small batch over eight layers, with an odd number of kept rows and a recent window
        dict(_DECODE, name="decode_small_batch", batch=3, layers=8, rows=4611, tail=389),
        # a turn of 16 tokens through four layers of a single 8B-shaped sequence
        dict(_GENERATE, name="generate_8b"),
        # Algorithm 1 in full on a 16k prompt: four value-norm buckets and the denominator instance
        dict(_ROUTED, name="algorithm1_buckets"),
        # decode over the caller's own caches, four layers, 16 streams
        dict(_STATIC, name="static_decode", rows=4096, tail=404),
        # prompt and tokens that live in pinned host memory
        dict(_HOST, name="host_turn"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(["prefill", "prefill", "prefill", "prefill", "decode", "decode", "generate", "routed", "static", "host"])
    if kind == "prefill":
        d, dtype = rng.choice([(128, "bf16")] * 4 + [(64, "bf16"), (128, "fp32"), (64, "fp32")])
        t = rng.choice([128, 256, 512, 1024, 2048, 64 * rng.randint(1, 40)])
        n = max(2 * t, _log(rng, 512, 65536) | rng.randint(0, 1))
        return dict(_PREFILL, batch=rng.randint(1, 8), layers=_log(rng, 1, 16), kv_heads=rng.choice([1, 2, 4, 8, 8, 10]),
                    group=rng.randint(1, 8), head_dim=d, dtype=dtype, block=t, levels=rng.randint(1, 3),
                    window=rng.choice([0, 0, 128, rng.randint(1, 500)]), context=n, chunk=min(n, rng.choice([t, 4096, 8192, n])),
                    per_layer=rng.random() < 0.5, center=rng.random() < 0.2, keys=rng.choice(["llama", "student_t"]),
                    queries=_log(rng, 1, 16))
    if kind == "decode":
        d, dtype = rng.choice([(128, "bf16")] * 4 + [(64, "bf16"), (128, "fp32"), (64, "fp32")])
        return dict(_DECODE, batch=_log(rng, 1, 32), layers=_log(rng, 1, 16), kv_heads=rng.choice([1, 2, 4, 8, 8, 10]),
                    group=rng.randint(1, 8), head_dim=d, dtype=dtype, levels=rng.randint(1, 3), rows=_log(rng, 65, 32768),
                    tail=rng.choice([0, rng.randint(1, 1200)]))
    if kind == "generate":
        return dict(_GENERATE, batch=_log(rng, 1, 16), layers=rng.randint(1, 8), kv_heads=rng.choice([2, 4, 8, 8, 10]),
                    group=rng.randint(1, 8), rows=_log(rng, 256, 16384), tail=rng.randint(0, 1500), steps=_log(rng, 4, 64))
    if kind == "routed":
        t = rng.choice([256, 512, 1024, 2048])
        return dict(_ROUTED, route=rng.choice(["buckets", "preserving"]), batch=rng.randint(1, 4), kv_heads=rng.choice([2, 4, 8]),
                    group=rng.randint(1, 8), block=t, levels=rng.randint(1, 3), context=max(2 * t, _log(rng, 2048, 65536) | 1),
                    buckets=rng.randint(1, 5))
    if kind == "static":
        d, dtype = rng.choice([(128, "bf16"), (128, "bf16"), (64, "bf16"), (128, "fp32"), (64, "fp32")])
        return dict(_STATIC, streams=_log(rng, 1, 256), layers=rng.randint(1, 8), group=rng.randint(1, 8), head_dim=d, dtype=dtype,
                    rows=_log(rng, 65, 16384), tail=rng.randint(0, 1000), levels=rng.randint(0, 3))
    return dict(_HOST, batch=rng.randint(1, 4), group=rng.randint(1, 8), block=rng.choice([256, 512, 1024]),
                context=_log(rng, 2048, 16384), steps=_log(rng, 4, 64))


def _cost_ms(case):
    """Rough time of a pass, to bound the drawn cases by the largest listed one."""
    w = work(case)
    slow = case["kind"] == "prefill" and (case["dtype"] == "fp32" or case["head_dim"] == 64 or case["block"] % 128)
    ms = w["bytes"] / 5e9 + w["flops"] / (1.5e10 if slow else 5e11)
    if case["kind"] == "host":
        ms += _rows(case) * 4 * case["head_dim"] / 5e7
    if case["kind"] == "prefill":                       # launches: an append and a compress per chunk, per layer at worst
        ms += 0.04 * case["layers"] * -(-case["context"] // case["chunk"]) + 0.01 * case["layers"] * case["queries"]
    return ms


def draw(rng):
    while True:
        case = _draw_once(rng)
        if _cost_ms(case) <= 8.0 and _state_bytes(case) <= 20e9:
            return case


# ---------------------------------------------------------------------------------------------- shapes

def _esz(case):
    return 4 if case.get("dtype") == "fp32" else 2


def _rows(case):
    """(key, value) rows of a pass's prompt over all streams."""
    return case["batch"] * case.get("layers", 1) * case["kv_heads"] * case["context"]


def _calls(case):
    """SoftmaxBalance calls per stream of a prompt."""
    blocks = max(0, case["context"] - case.get("window", 0)) // case["block"]
    return sum(blocks >> level for level in range(case["levels"]))


def _kept(case):
    """Rows that a stream keeps of its prompt."""
    blocks, t, left = max(0, case["context"] - case.get("window", 0)) // case["block"], case["block"], case["context"]
    for level in range(case["levels"]):
        left -= (blocks >> level) * (t // 2)
    return left


def _state_bytes(case):
    row = 2 * case["head_dim"] * _esz(case)
    if case["kind"] in ("prefill", "routed", "host"):
        return 3 * _rows(case) * row * (case.get("buckets", 0) + 1 if case["kind"] == "routed" else 1) + 2e9
    streams = case["streams"] if case["kind"] == "static" else case["batch"] * case["kv_heads"]
    return 2 * streams * case["layers"] * (case["rows"] + case["tail"] + 2048) * row


def work(case):
    """Bytes: the prompt's rows read once and the kept ones written once, the attended rows read once, queries and
    outputs.  Flops: the strict lower triangle of both Gram matrices of every call, and attention's two products."""
    d, e, g = case["head_dim"], _esz(case), case["group"]
    row = 2 * d * e
    if case["kind"] in ("prefill", "routed", "host"):
        streams = case["batch"] * case.get("layers", 1) * case["kv_heads"]
        kept, t = _kept(case), case["block"]
        asked = case.get("queries", 1) if case["kind"] != "host" else case["steps"]
        bytes_ = streams * row * (case["context"] + kept + asked * (kept + g))
        flops = streams * (_calls(case) * 2.0 * t * (t - 1) * d + asked * 4.0 * g * kept * d)
        if case["kind"] == "routed" and case["route"] == "buckets":     # the denominator instance: keys in, kept, attended
            bytes_ += streams * row // 2 * (case["context"] + 2 * kept)
            flops += streams * (_calls(case) * 2.0 * t * (t - 1) * d + 2.0 * g * kept * d)
        return {"bytes": bytes_, "flops": flops}
    streams = (case["streams"] if case["kind"] == "static" else case["batch"] * case["kv_heads"]) * case["layers"]
    stored, tokens = case["rows"] + case["tail"], case.get("steps", 1)
    bytes_ = streams * tokens * row * (stored + g)
    if case["kind"] == "generate":
        bytes_ += streams * row * (2 * stored + 2 * tokens)             # the prefix and the turn's rows: read and written
    return {"bytes": bytes_, "flops": streams * tokens * 4.0 * g * stored * d}


def tolerance(case):
    """Decode outputs are rounded to the caches' type.  The kept sets follow coins drawn from the seed: with the
    paper's constant no decision of these inputs hangs on the last bits of a sum."""
    # Seen between the library's two kernel families, other split factors and attention in 64 bits: fp32 6e-7 and at
    # most 8e-6; bf16 3e-4 and at most 0.024 between implementations (1.7e-3 against 64 bits: the final rounding).
    if case.get("dtype") == "fp32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 2e-3, "max": 0.1}


# ---------------------------------------------------------------------------------------------- inputs

def _dtype(case):
    return torch.float32 if case.get("dtype") == "fp32" else torch.bfloat16


def _profile(case, g, heads):
    """Per-head mean and channel scale of the keys: [.., heads, 1, d]."""
    d, recipe = case["head_dim"], case.get("keys", "llama")
    mu = torch.zeros(*heads, 1, d, device="cuda")
    scale = torch.ones(*heads, 1, d, device="cuda")
    if recipe == "outlier2":
        scale[..., torch.randperm(d, device="cuda", generator=g)[:2]] = 8.0
    elif recipe == "llama":
        mu = 0.5 * torch.randn(*heads, 1, d, device="cuda", generator=g)
        hot = torch.rand(*heads, 1, d, device="cuda", generator=g).topk(4, dim=-1).indices
        scale.scatter_(-1, hot, 10.0)
    return mu, scale


def _draw_kv(case, g, shape, profile):
    """Keys and values [.., n, d] as the synthetic recipes have them."""
    mu, scale = profile
    k = torch.randn(*shape, device="cuda", generator=g)
    if case.get("keys") == "student_t":                 # Student-t with 4 degrees of freedom: chi^2_4 = -2 ln(u1 u2)
        u = torch.rand(*shape, device="cuda", generator=g).mul_(torch.rand(*shape, device="cuda", generator=g)).clamp_(min=1e-12)
        k = k / (u.log_().mul_(-0.5)).sqrt_()
    else:
        k = (k + mu) * scale
    v = torch.randn(*shape, device="cuda", generator=g)
    return k.to(_dtype(case)), v.to(_dtype(case))


def _context(case, layers, **kw):
    return bk.Context(n_seqs=case["batch"], n_layers=layers, n_kv_heads=case["kv_heads"],
                      n_q_heads=case["kv_heads"] * case["group"], head_dim=case["head_dim"], dtype=case.get("dtype", "bf16"),
                      levels=case["levels"], seed=11, **kw)


def _queries(case, g, *lead):
    shape = (*lead, case["batch"], case["kv_heads"] * case["group"], case["head_dim"])
    return torch.randn(*shape, device="cuda", generator=g).to(_dtype(case))


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return {"case": case, **globals()["_prepare_" + case["kind"]](case, g)}


def run(state):
    return globals()["_run_" + state["case"]["kind"]](state)


def _asked(q, out):
    """The query and output tensors of every call, taken apart once: [(layer, query, output)]."""
    return [(layer, q[i, layer], out[i, layer]) for i in range(q.shape[0]) for layer in range(q.shape[1])]


def _prepare_prefill(case, g):
    B, H, d, n = case["batch"], case["kv_heads"], case["head_dim"], case["context"]
    ctx = _context(case, case["layers"], block=case["block"], max_tokens=n, max_pending=case["chunk"],
                   recent_window=case["window"], center_keys=int(case["center"]))
    profile = [_profile(case, g, (B, H)) for _ in range(case["layers"])]
    chunks = []
    for first in range(0, n, case["chunk"]):
        rows = min(case["chunk"], n - first)
        chunks.append([_draw_kv(case, g, (B, H, rows, d), profile[layer]) for layer in range(case["layers"])])
    q = _queries(case, g, case["queries"], case["layers"])
    out = torch.empty_like(q)
    return {"ctx": ctx, "chunks": chunks, "asked": _asked(q, out), "out": out}


def _run_prefill(state):
    ctx, case = state["ctx"], state["case"]
    ctx.reset()
    for chunk in state["chunks"]:
        for layer, (k, v) in enumerate(chunk):
            ctx.stream_append_layer(layer, k, v)
            if case["per_layer"]:
                ctx.compress_layer(layer)
        if not case["per_layer"]:
            ctx.compress()
    for layer, q, out in state["asked"]:
        ctx.decode_attn(layer, q, out)
    return {"out": state["out"], "sizes": ctx.level_sizes(0, 0, 0)}


def _load(case, ctx, layer, prefix, recent):
    ctx.cache_load_level(layer, case["levels"], *prefix)
    if recent is not None:
        ctx.stream_append_layer(layer, *recent)


def _caches(case, g):
    """Per layer: the key profile, the compressed prefix, and the recent rows (or None)."""
    B, H, d = case["batch"], case["kv_heads"], case["head_dim"]
    for _ in range(case["layers"]):
        profile = _profile(case, g, (B, H))
        prefix = _draw_kv(case, g, (B, H, case["rows"], d), profile)
        yield profile, prefix, _draw_kv(case, g, (B, H, case["tail"], d), profile) if case["tail"] else None


def _prepare_decode(case, g):
    ctx = _context(case, case["layers"], block=64, max_tokens=(case["rows"] << case["levels"]) + case["tail"],
                   max_pending=max(1, case["tail"]))
    for layer, (_, prefix, recent) in enumerate(_caches(case, g)):
        _load(case, ctx, layer, prefix, recent)
    q = _queries(case, g, 1, case["layers"])
    out = torch.empty_like(q)
    return {"ctx": ctx, "asked": _asked(q, out), "out": out}


def _run_decode(state):
    for layer, q, out in state["asked"]:
        state["ctx"].decode_attn(layer, q, out)
    return state["out"]


def _prepare_generate(case, g):
    L, steps, B, H, d = case["layers"], case["steps"], case["batch"], case["kv_heads"], case["head_dim"]
    ctx = _context(case, L, block=case["block"], max_tokens=(case["rows"] << case["levels"]) + case["tail"] + steps,
                   max_pending=case["tail"] + steps)
    caches, new = [], []
    for profile, prefix, recent in _caches(case, g):
        caches.append((prefix, recent))
        k, v = _draw_kv(case, g, (B, H, steps, d), profile)
        new.append([(k[:, :, i].contiguous(), v[:, :, i].contiguous()) for i in range(steps)])
    q = _queries(case, g, steps, L)
    out = torch.empty_like(q)
    asked = [(layer, qi, *new[layer][i // L], oi) for i, (layer, qi, oi) in enumerate(_asked(q, out))]
    return {"ctx": ctx, "caches": caches, "asked": asked, "out": out}


def _run_generate(state):
    ctx = state["ctx"]
    ctx.reset()
    for layer, (prefix, recent) in enumerate(state["caches"]):
        _load(state["case"], ctx, layer, prefix, recent)
    for layer, q, k, v, out in state["asked"]:
        ctx.stream_step(layer, q, k, v, out)
    return state["out"]


def _prepare_routed(case, g):
    B, H, d, n = case["batch"], case["kv_heads"], case["head_dim"], case["context"]
    slots = case["buckets"] + 1 if case["route"] == "buckets" else 2
    ctx = _context(case, slots, block=case["block"], max_tokens=n)
    k, v = _draw_kv(case, g, (B, H, n, d), _profile(case, g, (B, H)))
    if case["route"] == "buckets":                      # value norms (about 11) spread over the buckets' octaves below 2^4
        spread = torch.rand(B, H, n, 1, device="cuda", generator=g)
        v = (v.float() * torch.exp2(-case["buckets"] * spread)).to(v.dtype)
    return {"ctx": ctx, "k": k, "v": v, "q": _queries(case, g)}


def _run_routed(state):
    ctx, case = state["ctx"], state["case"]
    ctx.reset()
    if case["route"] == "buckets":
        nb = case["buckets"]
        counts = ctx.stream_append_layer_bucketed(0, nb, 4, state["k"], state["v"])
        ctx.stream_append_layer_keys(nb, state["k"])
        ctx.compress()
        out = ctx.decode_attn_merged(list(range(nb)), [nb], state["q"])
    else:
        counts = ctx.stream_append_layer_preserving(0, state["k"], state["v"], -0.1)
        ctx.compress_layer(1)
        out = ctx.decode_attn_merged([0, 1], [0, 1], state["q"])
    return {"out": out, "counts": counts}


def _prepare_static(case, g):
    S, d, n = case["streams"], case["head_dim"], case["rows"] + case["tail"]
    caches = [_draw_kv(case, g, (S, n, d), _profile(case, g, (S,))) for _ in range(case["layers"])]
    q = torch.randn(case["layers"], S, case["group"], d, device="cuda", generator=g).to(_dtype(case))
    out = torch.empty_like(q)
    return {"caches": [(k, v, q[i], out[i]) for i, (k, v) in enumerate(caches)], "out": out}


def _run_static(state):
    case = state["case"]
    for k, v, q, out in state["caches"]:
        bk.decode_attn_static(k, v, case["rows"], case["levels"], q, out=out)
    return state["out"]


def _prepare_host(case, g):
    B, H, d, n, steps = case["batch"], case["kv_heads"], case["head_dim"], case["context"], case["steps"]
    ctx = _context(case, 1, block=case["block"], max_tokens=n + steps)
    profile = _profile(case, g, (B, H))
    pin = lambda x: x.cpu().pin_memory()  # noqa: E731
    k, v = (pin(x) for x in _draw_kv(case, g, (B, H, n, d), profile))
    kn, vn = (pin(x.permute(2, 0, 1, 3).contiguous()) for x in _draw_kv(case, g, (B, H, steps, d), profile))
    q = pin(_queries(case, g, steps))
    out = torch.empty_like(q).pin_memory()
    torch.cuda.synchronize()                            # a server has its staging buffers in place before the first request
    ctx.stream_step_host(0, q[0], kn[0], vn[0], out[0])
    torch.cuda.synchronize()
    return {"ctx": ctx, "k": k, "v": v, "steps": list(zip(q, kn, vn, out)), "out": out}


def _run_host(state):
    ctx = state["ctx"]
    ctx.reset()
    ctx.stream_append_layer_host(0, state["k"], state["v"])
    ctx.compress()
    for q, k, v, out in state["steps"]:
        ctx.stream_step_host(0, q, k, v, out)
    torch.cuda.current_stream().synchronize()           # the turn's outputs are read on the host
    return state["out"]
