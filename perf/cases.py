"""The work that programs built on this library have it do, as cases that can be timed and compared.

A case is one pass of a serving program over the public calls of ``binding.Context``: a batch of requests is composed
from registered packets (``assemble``) and the query tokens are run through every layer (``query_prefill``), as one
batch of a server does it.  Registration is offline and lies in ``prepare``.  ``kind`` says what a pass does:

* ``prefill``   assemble, then one prefill call per layer
* ``ragged``    the same with per-request query lengths (``query_prefill_ragged``)
* ``generate``  assemble, prefill of raw (un-rotated) q and k, then ``steps`` decode steps of one token per request
* ``pruned``    prefill over documents that a KV compressor thinned out per layer and kv head
* ``host``      the documents wait in pinned host memory: evict, assemble (copies them in), prefill
* ``handover``  prefill here, decode in another engine: the composed cache is materialised, attended to, and exported
  with the query's rows, layer by layer

Sizes are those of the repository's own workloads (``inputs.py``) and the ranges around them.
"""
from __future__ import annotations

import random

import torch

from paper_2604_13226_b200 import binding as kvp

_DEFAULTS = dict(kind="prefill", layers=1, hq=32, hkv=8, d=128, dtype="bf16", pairing=0, theta=500000.0, batch=1, docs=5,
                 doc_lo=512, doc_hi=512, pool=0, filler=16, filler_std=1.0, q=64, steps=0, outliers=0, precise=False,
                 lse=False, keep=1.0, layout=1)


def _case(**kw):
    return dict(_DEFAULTS, **kw)


def listed():
    return [
        # the smallest call there is: 4/2 heads of 64, fp32, three short documents, a short question; launches and host time
        _case(name="tiny_f32", hq=4, hkv=2, d=64, dtype="f32", theta=10000.0, docs=3, doc_lo=128, doc_hi=128, filler=8,
              filler_std=0.02, q=32, lse=True),
        # one attention layer of an 8B model for one ordinary question over five passages; latency
        _case(name="question_5x512", docs=5, q=64),
        # a server's step over a stack of layers: four requests draw their ten passages from a common store
        _case(name="stack_10x1024_b4", layers=8, batch=4, docs=10, doc_lo=1024, doc_hi=1024, pool=64, q=128),
        # group of 7 heads, documents of uneven lengths, outlier channels, and the option that keeps their scores exact
        _case(name="uneven_docs_precise", layers=2, hq=28, hkv=4, theta=1000000.0, batch=8, docs=20, doc_lo=256, doc_hi=1024,
              q=256, outliers=2, precise=True),
        # a short question over a very long context (131K tokens): reading the cache is all there is
        _case(name="long_64x2048_q16", docs=64, doc_lo=2048, doc_hi=2048, q=16),
        # long questions over long contexts: the largest pass, bound by arithmetic
        _case(name="long_16x2048_q1024_b4", batch=4, docs=16, doc_lo=2048, doc_hi=2048, q=1024, lse=True),
        # an answer is generated: prefill of the raw question, then token after token over the grown cache
        _case(name="generate_b8", kind="generate", layers=4, batch=8, docs=10, doc_lo=1024, doc_hi=1024, pool=64, q=32, steps=16),
        # a batch as it arrives: questions of different lengths over documents of different lengths
        _case(name="ragged_b8", kind="ragged", layers=4, batch=8, docs=10, doc_lo=200, doc_hi=1200, q=192),
        # documents thinned out to about two fifths, each layer and head keeping its own tokens
        _case(name="pruned_b4", kind="pruned", layers=4, batch=4, docs=10, doc_lo=1024, doc_hi=1024, q=128, keep=0.41),
        # the first question about documents that are still in host memory: the transfer is part of the time to the first token
        _case(name="host_b2", kind="host", layers=4, batch=2, docs=8, doc_lo=512, doc_hi=512, q=64),
        # the composed cache is handed over to another engine after the prefill
        _case(name="handover_b2", kind="handover", layers=2, batch=2, docs=10, doc_lo=700, doc_hi=1024, q=64),
        # heads of 64, as smaller models have them, bf16
        _case(name="heads64_8x1024_b4", layers=2, d=64, batch=4, docs=8, doc_lo=1024, doc_hi=1024, q=128),
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], spread evenly over its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


#: Most flops of a drawn case: those of its kind's listed ones.
_MOST = {"small": 6e10, "d128": 2e12}


def draw(rng):
    what = rng.choice(["f32", "f32", "heads64", "heads64", "question", "stack", "uneven", "long", "long", "generate", "generate", "ragged",
                       "pruned", "host", "handover"])
    heads = rng.choice([(32, 8), (32, 8), (28, 4)])
    while True:
        c = dict(layout=rng.randrange(1 << 30), hq=heads[0], hkv=heads[1], pairing=rng.choice([0, 0, 0, 1]), lse=rng.random() < 0.3)
        most = _MOST["d128"]
        if what in ("f32", "heads64"):
            h = rng.choice([(4, 2), (8, 2), (32, 8), (14, 2)])
            c.update(hq=h[0], hkv=h[1], d=64 if what == "heads64" else rng.choice([64, 128]), dtype="f32" if what == "f32" else "bf16",
                     theta=10000.0, batch=_log(rng, 1, 4), docs=_log(rng, 1, 12), filler=rng.choice([0, 8, 16]), q=_log(rng, 1, 256),
                     layers=rng.choice([1, 2]))
            lo, hi, most = 64, 1024, _MOST["small"]
        elif what == "question":
            c.update(docs=_log(rng, 1, 10), q=_log(rng, 1, 128), filler=rng.choice([0, 8, 16, 16, 20]))
            lo, hi = 64, 1024
        elif what == "stack":
            c.update(layers=rng.randint(2, 8), batch=rng.randint(1, 8), docs=_log(rng, 2, 16), pool=64, q=_log(rng, 16, 256))
            lo, hi = 256, 1024
        elif what == "uneven":
            c.update(layers=2, batch=rng.randint(1, 8), docs=_log(rng, 4, 20), q=_log(rng, 16, 256), outliers=2, precise=rng.random() < 0.7)
            lo, hi = 100, 1024
        elif what == "long":
            c.update(batch=rng.choice([1, 2, 4]), docs=_log(rng, 2, 64), q=_log(rng, 8, 1024))
            lo, hi = 1024, 2048
        elif what == "generate":
            c.update(kind="generate", layers=rng.randint(1, 4), batch=_log(rng, 1, 12), docs=_log(rng, 2, 12), q=_log(rng, 4, 128),
                     steps=rng.randint(4, 16))
            lo, hi = 256, 1024
        elif what == "ragged":
            c.update(kind="ragged", layers=rng.randint(1, 4), batch=rng.randint(2, 8), docs=_log(rng, 2, 12), q=_log(rng, 16, 256))
            lo, hi = 100, 1200
        elif what == "pruned":
            c.update(kind="pruned", layers=rng.randint(1, 4), batch=rng.randint(1, 4), docs=_log(rng, 2, 12), q=_log(rng, 8, 192),
                     keep=round(rng.uniform(0.2, 0.8), 2))
            lo, hi = 256, 1024
        elif what == "host":
            c.update(kind="host", layers=rng.randint(1, 4), batch=rng.randint(1, 2), docs=_log(rng, 2, 8), q=_log(rng, 8, 128))
            lo, hi = 128, 512
        else:
            c.update(kind="handover", layers=rng.randint(1, 2), batch=rng.randint(1, 3), docs=_log(rng, 2, 10), q=_log(rng, 8, 128))
            lo, hi = 200, 1024
        a, b = sorted((_log(rng, lo, hi), _log(rng, lo, hi)))
        c.update(doc_lo=a, doc_hi=b)
        c = _case(**c)
        w = work(c)
        if w["flops"] <= most and w["bytes"] <= 2.2e9 * (8 if c["kind"] == "generate" else 1):
            return c


def _sizes(case):
    """Document lengths, the requests' document lists, kept rows and query lengths: from the case alone."""
    rng = random.Random(case["layout"])
    n_docs = case["pool"] or case["batch"] * case["docs"]
    lens = [rng.randint(case["doc_lo"], case["doc_hi"]) for _ in range(n_docs)]
    if case["pool"]:
        items = [rng.sample(range(n_docs), case["docs"]) for _ in range(case["batch"])]
    else:
        items = [list(range(b * case["docs"], (b + 1) * case["docs"])) for b in range(case["batch"])]
    used = sorted({p for it in items for p in it})                 # only documents that some request names are held
    number = {p: i for i, p in enumerate(used)}
    lens = [lens[p] for p in used]
    items = [[number[p] for p in it] for it in items]
    planes = case["layers"] * case["hkv"]
    kept = None
    if case["kind"] == "pruned":
        kept = []
        for n in lens:
            rows = []
            for _ in range(case["layers"]):
                per_layer = case["keep"] * rng.uniform(0.7, 1.3)
                rows += [max(1, min(n, round(n * per_layer * rng.uniform(0.6, 1.0)))) for _ in range(case["hkv"])]
            kept.append(rows)
    q_lens = [rng.randint(1, case["q"]) for _ in range(case["batch"])] if case["kind"] == "ragged" else [case["q"]] * case["batch"]
    return lens, items, kept, q_lens, planes


def work(case):
    lens, items, kept, q_lens, planes = _sizes(case)
    e = 2 if case["dtype"] == "bf16" else 4
    row = 2 * case["d"] * e                                        # K and V of one token in one plane (layer, kv head)
    fill = 2 * case["filler"]
    if kept is None:
        doc_rows = [n * planes for n in lens]
    else:
        doc_rows = [sum(r) for r in kept]
    prefix_rows = [sum(doc_rows[p] + fill * planes for p in it) for it in items]       # over all planes
    prefix_bytes = (sum(doc_rows) + fill * planes) * row
    L, hq, hkv, d = case["layers"], case["hq"], case["hkv"], case["d"]
    per_token = L * ((2 * hq + 4 * hkv) * d * e + (4 * hq if case["lse"] else 0))      # q, k, v read; output and cache rows written
    flops, new = 0.0, 0
    group = hq // hkv
    for rows, n in zip(prefix_rows, q_lens):
        flops += 4.0 * d * group * (n * rows + planes * n * (n + 1) / 2)
        new += n
    nbytes = prefix_bytes + new * per_token
    if case["kind"] == "generate":                                 # each step reads the whole cache again, shared documents once
        for s in range(case["steps"]):
            flops += sum(4.0 * d * group * (rows + planes * (case["q"] + s + 1)) for rows in prefix_rows)
            nbytes += prefix_bytes + case["batch"] * ((case["q"] + s) * planes * row + per_token)
    if case["kind"] == "handover":                                 # the exported cache, each request its own
        nbytes += (sum(prefix_rows) + new * planes) * row
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # bf16: probabilities and the rotated operand of q.k are rounded to 8 bits; fp32: sums of 32-bit products
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2, "max": 0.1}


class _State:
    pass


def prepare(case, seed):
    lens, items, kept, q_lens, planes = _sizes(case)
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    L, B, hq, hkv, d, F = case["layers"], case["batch"], case["hq"], case["hkv"], case["d"], case["filler"]

    def normal(*dims):
        return torch.randn(dims, generator=gen, device=dev, dtype=dt)

    s = _State()
    s.case, s.q_lens = case, q_lens
    total_q = case["q"] + case["steps"]
    prefix = [sum(lens[p] + 2 * F for p in it) for it in items]
    staged = sum(prefix) if case["kind"] == "handover" else sum(2 * F * len(it) for it in items)
    s.ctx = kvp.Context(L, hq, hkv, d, case["dtype"], rope_theta=case["theta"], rope_pairing=case["pairing"],
                        pool_tokens=sum(lens) + 2 * F + 8, max_packets=len(lens), max_adapters=1, max_batch=B,
                        max_slots=sum(len(it) for it in items), max_prefix_tokens=max(prefix), max_query_tokens=total_q,
                        max_ws_rows=staged + B * total_q + 8, device=torch.cuda.current_device(),
                        max_compressed=len(lens) if kept else 0)
    scale = None
    if case["outliers"]:                                           # the same loud channels in every document
        at = torch.rand((L, 1, hkv, d), generator=gen, device=dev).topk(case["outliers"], dim=-1).indices
        scale = torch.ones((L, 1, hkv, d), device=dev, dtype=dt).scatter_(-1, at, 8.0)
    s.host = []
    for i, n in enumerate(lens):
        if kept:
            rows = sum(kept[i])
            s.ctx.register_packet_compressed(normal(rows, d), normal(rows, d), n, 0, kept[i])
        elif case["kind"] == "host":
            k, v = (normal(L, hkv, n, d).cpu().pin_memory() for _ in range(2))
            s.host.append((k, v))
            s.ctx.register_packet_host(k, v, n, 0)
        else:
            k, v = normal(L, n, hkv, d), normal(L, n, hkv, d)
            if scale is not None:
                k, v = k * scale, v * scale
            s.ctx.register_packet(k, v, n, 0)
    if F:
        hk, hv, tk, tv = (normal(L, F, hkv, d) * case["filler_std"] for _ in range(4))
        s.ctx.register_adapter(hk, hv, F, 0, tk, tv, F, 0)
    s.items = [[(p, 0 if F else -1) for p in it] for it in items]
    s.prefix = prefix

    # each layer's projections of the query tokens, and where their results go
    def calls(n_calls, q_len):
        got = []
        for _ in range(n_calls):
            lse = torch.zeros((B, hq, q_len), device=dev, dtype=torch.float32) if case["lse"] else None
            got.append((normal(B, q_len, hq, d), normal(B, q_len, hkv, d), normal(B, q_len, hkv, d),
                        torch.zeros((B, q_len, hq, d), device=dev, dtype=dt), lse))
        return got

    s.prompt = calls(L, case["q"])
    # a step's tokens of all layers lie together
    s.steps = []
    if case["steps"]:
        T = case["steps"]
        q, k, v = normal(T, L, B, 1, hq, d), normal(T, L, B, 1, hkv, d), normal(T, L, B, 1, hkv, d)
        s.step_out = torch.zeros((T, L, B, 1, hq, d), device=dev, dtype=dt)
        s.steps = [[(q[t, l], k[t, l], v[t, l], s.step_out[t, l]) for l in range(L)] for t in range(T)]
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx = s.case, s.ctx
    kind, q_len = case["kind"], case["q"]
    if kind == "host":
        for p in range(len(s.host)):
            ctx.evict_packet(p)
    aid, prefix = ctx.assemble(s.items, kvp.REBASE | (kvp.MATERIALIZE if kind == "handover" else 0))
    if kind == "ragged":
        for l, (q, k, v, out, lse) in enumerate(s.prompt):
            ctx.query_prefill_ragged(aid, l, q, k, v, q_len, s.q_lens, out, lse)
    else:
        flags = (kvp.ROPE_QUERY if kind == "generate" else 0) | (kvp.PRECISE_QK if case["precise"] else 0)
        for l, (q, k, v, out, lse) in enumerate(s.prompt):
            ctx.query_prefill(aid, l, q, k, v, q_len, out, lse, flags)
    got = {"out": [c[3] for c in s.prompt], "lse": [c[4] for c in s.prompt]}
    if kind == "generate":
        for step in s.steps:
            for l, (q, k, v, out) in enumerate(step):
                ctx.query_prefill(aid, l, q, k, v, 1, out, None, kvp.CONTINUE | kvp.ROPE_QUERY)
        got["step_out"] = s.step_out
    if kind == "handover":
        got["cache"] = [[ctx.export_cache(aid, l, b, prefix[b], q_len) for b in range(case["batch"])] for l in range(case["layers"])]
    return got
