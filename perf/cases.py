"""The work whose speed counts: calls of the public entry points at the sizes users bring.

A case is a dict of plain values.  ``listed()`` names twelve, ``draw(rng)`` gives more of the
same ranges; ``prepare`` makes what a program holds before the call (device tensors, the
descriptor, the workspace), ``run`` is the call.  Every retained row of K and V is a bit copy and
every index a whole number, so those outputs are returned as integers.

Inputs.  The rows of an observation window are neighbouring tokens, so the queries of a head share
most of their direction; keys carry a few outlier channels (one in a hundred, scaled by eight);
priors mark the first tokens of structural code lines (lines of geometric length, mean 12), or the
tokens of the spans that the planner selects, or grade every token between 0 and 1.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_10235_b200 import binding as cc
from paper_2604_10235_b200 import inputs as gen
from paper_2604_10235_b200.api import LayerCompressor, LayerSpec

HEAD_DIM = 128
POOLS = {"none": cc.CC_POOL_NONE, "max": cc.CC_POOL_MAX, "avg": cc.CC_POOL_AVG}
#: (query heads, KV heads) of the configurations in inputs.py
HEADS = ((8, 2), (32, 8), (28, 4))


def _text(values):
    return ",".join(str(int(v)) for v in values)


def _ints(text):
    return tuple(int(v) for v in text.split(","))


def _case(name, op, heads, window, lens, budgets, pool="max", pool_size=7, **more):
    """One compression case; the keywords left out keep the values a plain call has."""
    c = {"name": name, "op": op, "heads_q": heads[0], "heads_kv": heads[1], "window": window,
         "lens": _text(lens), "budgets": _text(budgets), "pool": pool, "pool_size": pool_size,
         "chunk": 1, "page_size": 0, "prior": "lines", "p_structural": 0.29, "beta": 0.0,
         "force": True, "span_ratio": 0.0, "causal": False, "nearest": False, "layers": 1,
         "v_in_place": False, "overlap": False}
    c.update(more)
    return c


def listed():
    w = gen.workloads()
    ragged = w["ragged_paged"]
    # thirty-two chunks of at most 4096 tokens, budgets spread by the planner's multipliers
    rng = np.random.Generator(np.random.PCG64(5005))
    chunk_lens = rng.integers(128, 4097, size=32)
    chunk_budgets = np.floor(chunk_lens * 0.4 * rng.uniform(0.5, 1.5, size=32))
    return [
        # one short prompt on a small model: four launches, so latency and host time
        _case("tiny", "layer", (8, 2), 32, (2048,), (512,)),
        # one layer of a long prompt, token-major K/V as attention leaves it after prefill
        _case("llama3_8b", "layer", (32, 8), 64, (32768,), (2048,)),
        # a longer prompt, 448 query rows per KV head, many structural tokens
        _case("qwen25_coder_7b", "layer", (28, 4), 64, (65536,), (4096,), p_structural=0.6529),
        # whole chunks of ten tokens kept or dropped together
        _case("chunk10", "layer", (32, 8), 64, (32768,), (2048,), pool="none", pool_size=1, chunk=10),
        # the layer of a served batch in a paged cache: the largest work of one call
        _case("ragged_paged", "layer", (32, 8), 64, ragged.lens, ragged.budgets, page_size=16),
        # the paper's own setting: retrieved chunks as one batch, planned spans, capped protection
        _case("paper_chunks", "layer", (32, 8), 128, chunk_lens, chunk_budgets, pool="avg", pool_size=5,
              prior="spans", span_ratio=0.5),
        # the window inside the prompt (causal), an odd length, graded priors added to the scores
        _case("causal_graded", "layer", (28, 4), 64, (10007,), (1500,), pool="avg", pool_size=5,
              prior="graded", beta=0.01, force=False, causal=True),
        # the budget left by the protected tokens goes to their neighbours
        _case("nearest_fill", "layer", (32, 8), 64, (32768,), (4096,), nearest=True),
        # a retrieved chunk of a request, all layers of the model in one call
        _case("all_layers", "layers", (32, 8), 128, (4096,), (1638,), pool="avg", pool_size=5,
              prior="spans", span_ratio=0.5, layers=32),
        # a prompt whose K/V were offloaded: copied in from page-locked memory and results back out
        _case("offloaded", "host", (32, 8), 64, (32768,), (3276,), v_in_place=True, overlap=True),
        # choosing the chunks worth keeping: 32 candidates, 64 query tokens, bf16 logits
        _ppl_case("chunk_scoring", 32, 64, 128256, "bf16", 8),
        # the same with f32 logits and a vocabulary whose rows do not start on 16-byte boundaries
        _ppl_case("chunk_scoring_odd", 48, 16, 50257, "f32", 12),
    ]


def _ppl_case(name, chunks, tokens, vocab, dtype, keep):
    return {"name": name, "op": "ppl", "chunks": chunks, "tokens": tokens, "vocab": vocab,
            "dtype": dtype, "keep": keep}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: lengths and budgets spread over their logarithm, odd ones among them."""
    kind = rng.choices(("single", "batch", "chunked", "nearest", "layers", "host", "ppl"),
                       (30, 20, 10, 10, 10, 5, 15))[0]
    if kind == "ppl":
        vocab = rng.choice((32000, 32003, 50257, 128256, 151936, _log_int(rng, 8000, 160000)))
        rows = _log_int(rng, 16, 2048 * 128256 // vocab)
        tokens = min(_log_int(rng, 4, 128), rows)
        dtype = rng.choice(("bf16", "bf16", "f32"))
        chunks = max(1, min(512, rows // tokens // (2 if dtype == "f32" else 1)))
        c = _ppl_case("", chunks, tokens, vocab, dtype, max(1, chunks // rng.choice((2, 4))))
        del c["name"]
        return c
    heads = rng.choice(HEADS)
    group = heads[0] // heads[1]
    window = rng.choice([w for w in (16, 32, 50, 64, 100, 128) if w * group <= 512])
    pool, size = rng.choice((("max", 7), ("avg", 5), ("max", 5), ("avg", 3)))
    more = {}
    ratio = math.exp(rng.uniform(math.log(0.03), math.log(0.6)))
    if kind == "batch":
        lens = [_log_int(rng, 200, 65536) for _ in range(rng.choice((2, 5, 8, 16, 32)))]
        more["page_size"] = rng.choice((0, 16, 16, 32, 64))
    else:
        lens = [_log_int(rng, 1000, {"layers": 8192, "host": 32768}.get(kind, 131072))]
    if kind == "layers":
        more["layers"] = rng.choice((16, 28, 32))
    if kind == "host":
        more["v_in_place"] = more["overlap"] = rng.random() < 0.5
        if not more["v_in_place"]:
            lens = [max(1000, n // 2) for n in lens]
    # no more multiplications and copies than the largest listed case has
    room = 290000 * 8 // heads[1] * min(1.0, 256 / (group * window)) / (0.91 + 0.9 * ratio)
    room = int(room / more.get("layers", 1))
    if sum(lens) > room:
        lens = [max(200, n * room // sum(lens)) for n in lens]
    budgets = [max(1, int(n * ratio)) for n in lens]
    prior, force, beta = rng.choice((("lines", True, 0.0), ("lines", True, 0.0), ("spans", True, 0.0),
                                     ("graded", False, 0.01)))
    more.update(prior=prior, force=force, beta=beta, p_structural=rng.choice((0.2176, 0.29, 0.6529)))
    if prior == "spans":
        more["span_ratio"] = 0.5
    if kind in ("single", "batch"):
        more["causal"] = rng.random() < 0.25
    if kind == "chunked":
        pool, size, more["chunk"] = "none", 1, rng.choice((4, 10, 16, 33))
    if kind == "nearest":
        more.update(nearest=True, prior="lines", force=True, beta=0.0, span_ratio=0.0)
    op = {"layers": "layers", "host": "host"}.get(kind, "layer")
    c = _case("", op, heads, window, lens, budgets, pool, size, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------------------- inputs
def _line_starts(rng, n):
    """First tokens of the lines of a text of n tokens and the lines' labels (gen.LABELS)."""
    lengths = rng.geometric(1.0 / 12.0, size=n // 6 + 16)
    starts = np.concatenate([[0], np.cumsum(lengths)])
    starts = starts[starts < n]
    return starts, rng.random(len(starts))


def _prior(case, seed):
    """The prior of every sequence, back to back (f32)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for n, budget in zip(_ints(case["lens"]), _ints(case["budgets"])):
        starts, kind = _line_starts(rng, n)
        structural = starts[kind < case["p_structural"]]
        p = np.zeros(n, dtype=np.float32)
        if case["prior"] == "lines":
            for k in range(3):
                p[np.minimum(structural + k, n - 1)] = 1.0
        elif case["prior"] == "graded":
            p[:] = np.repeat(rng.random(len(starts)).astype(np.float32), np.diff(np.append(starts, n)))
        else:
            ends = np.minimum(structural + rng.integers(6, 41, size=len(structural)), n)
            score = 0.14 + 0.24 * rng.random(len(structural))
            p, _ = cc.cc_select_spans(structural, ends, score, rng.random(len(structural)) < 0.03, n,
                                      budget, 0.5, 16)
        out.append(p)
    return np.concatenate(out)


def _tensors(case, seed, rows):
    """Q window, K and V on the device; ``rows`` K/V rows."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    hq, hkv, w, s = case["heads_q"], case["heads_kv"], case["window"], len(_ints(case["lens"]))

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)

    shared = normal(s, 1, hkv, 1, HEAD_DIM) * 0.5 + normal(s, 1, hkv, hq // hkv, HEAD_DIM) * 0.5
    q = (shared.reshape(s, 1, hq, HEAD_DIM) + normal(s, w, hq, HEAD_DIM) * 0.7).contiguous()
    k, v = normal(rows, hkv, HEAD_DIM), normal(rows, hkv, HEAD_DIM)
    outliers = torch.randint(0, HEAD_DIM, (hkv, 2), generator=g, device="cuda")
    scale = torch.ones(hkv, HEAD_DIM, device="cuda", dtype=torch.bfloat16).scatter_(1, outliers, 8.0)
    return q, k.mul_(scale), v


def _desc_args(case):
    return dict(pool_kind=POOLS[case["pool"]], pool_size=case["pool_size"], chunk_size=case["chunk"],
                alpha=1.0, beta=case["beta"], force_threshold=0.5 if case["force"] else math.inf,
                span_ratio=case["span_ratio"], span_min=16, page_size=case["page_size"],
                causal=case["causal"],
                fill_mode=cc.CC_FILL_NEAREST if case["nearest"] else cc.CC_FILL_ATTENTION)


_CTX = []


def _context():
    """A program keeps one library context per thread."""
    if not _CTX:
        _CTX.append(cc.Context(0))
    return _CTX[0]


def _bits(t):
    return t.view(torch.int16)


def prepare(case, seed):
    return {"layer": _prepare_layer, "layers": _prepare_layers, "host": _prepare_host,
            "ppl": _prepare_ppl}[case["op"]](case, seed)


def _prepare_layer(case, seed):
    ctx, lens, budgets = _context(), _ints(case["lens"]), _ints(case["budgets"])
    ps, hkv, s = case["page_size"], case["heads_kv"], len(lens)
    kw, rows, st = _desc_args(case), sum(lens), {"op": "layer", "ctx": ctx}
    if ps:
        # a shuffled page table over the lower pages of the pool; the compacted cache goes to the
        # upper ones, in shuffled order as a free list hands them out
        pages = [-(-n // ps) for n in lens]
        fresh_counts = [-(-min(b, n) // ps) for b, n in zip(budgets, lens)]
        used, fresh = sum(pages), sum(fresh_counts)
        rng = np.random.Generator(np.random.PCG64(seed))
        ids = rng.permutation(used).astype(np.int32)
        table = np.full((s, max(pages)), -1, dtype=np.int32)
        at = 0
        for i, c in enumerate(pages):
            table[i, :c] = ids[at:at + c]
            at += c
        st["free_pages"] = torch.from_numpy(used + rng.permutation(fresh).astype(np.int32)).cuda()
        st["out_page_table"] = torch.empty((s, max(fresh_counts)), dtype=torch.int32, device="cuda")
        kw.update(page_table=torch.from_numpy(table).cuda(), pool_pages=used + fresh,
                  out_page_table_stride=max(fresh_counts))
        rows = (used + fresh) * ps
    if s > 1 or ps:
        st["desc"] = cc.Desc(case["heads_q"], hkv, case["window"], seq_lens=lens, budgets=budgets, **kw)
    else:
        st["desc"] = cc.Desc(case["heads_q"], hkv, case["window"], n=lens[0], budget=budgets[0], **kw)
    st["q"], st["k"], st["v"] = _tensors(case, seed, rows)
    st["prior"] = torch.from_numpy(_prior(case, seed)).cuda()
    if ps:
        st["k_out"], st["v_out"] = st["k"], st["v"]
        first = used * ps
    else:
        st["k_out"] = torch.empty((sum(budgets), hkv, HEAD_DIM), dtype=torch.bfloat16, device="cuda")
        st["v_out"] = torch.empty_like(st["k_out"])
        first = 0
    st["idx"] = torch.empty((hkv, sum(budgets)), dtype=torch.int32, device="cuda")
    st["count"] = torch.empty((s, hkv), dtype=torch.int32, device="cuda")
    st["ws"] = ctx.workspace(st["desc"])
    st["out"] = {"k": _bits(st["k_out"][first:]), "v": _bits(st["v_out"][first:]), "idx": st["idx"],
                 "count": st["count"]}
    if ps:
        st["out"]["page_table"] = st["out_page_table"]
    return st


def _prepare_layers(case, seed):
    ctx, n, b, hkv = _context(), _ints(case["lens"])[0], _ints(case["budgets"])[0], case["heads_kv"]
    layers = case["layers"]
    st = {"op": "layers", "ctx": ctx,
          "desc": cc.Desc(case["heads_q"], hkv, case["window"], n=n, budget=b, **_desc_args(case))}
    made = [_tensors(case, seed * 64 + i, n) for i in range(layers)]
    st["q"], st["k"], st["v"] = ([m[j] for m in made] for j in range(3))
    st["prior"] = torch.from_numpy(_prior(case, seed)).cuda()
    k_out, v_out = (torch.empty((layers, b, hkv, HEAD_DIM), dtype=torch.bfloat16, device="cuda")
                    for _ in range(2))
    idx = torch.empty((layers, hkv, b), dtype=torch.int32, device="cuda")
    count = torch.empty((layers, 1, hkv), dtype=torch.int32, device="cuda")
    st["k_out"], st["v_out"], st["idx"], st["count"] = (list(t) for t in (k_out, v_out, idx, count))
    st["ws"] = ctx.workspace(st["desc"])
    st["out"] = {"k": _bits(k_out), "v": _bits(v_out), "idx": idx, "count": count}
    return st


def _prepare_host(case, seed):
    spec = LayerSpec(case["heads_q"], case["heads_kv"], case["window"], _ints(case["lens"]),
                     _ints(case["budgets"]), **_desc_args(case))
    tensors = _tensors(case, seed, sum(spec.lens))
    host = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in tensors]
    comp = LayerCompressor(_context(), spec)
    return {"op": "host", "comp": comp, "host": host, "v_in_place": case["v_in_place"],
            "overlap": case["overlap"], "prior": torch.from_numpy(_prior(case, seed)).pin_memory()}


def _prepare_ppl(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    chunks, tokens, vocab = case["chunks"], case["tokens"], case["vocab"]
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    x = torch.randn((chunks, tokens, vocab), generator=g, device="cuda", dtype=dtype).mul_(2.0)
    targets = torch.randint(0, vocab, (tokens,), generator=g, device="cuda", dtype=torch.int32)
    # the better a chunk explains the query, the more its logits favour the query's tokens
    lift = torch.rand((chunks, 1), generator=g, device="cuda") * 12.0
    at = targets.long().view(1, tokens, 1).expand(chunks, tokens, 1)
    x.scatter_add_(2, at, lift.view(chunks, 1, 1).expand(chunks, tokens, 1).to(dtype))
    return {"op": "ppl", "ctx": _context(), "logits": x, "targets": targets, "keep": case["keep"],
            "nll": torch.empty((chunks, tokens), device="cuda"),
            "score": torch.empty((chunks,), device="cuda"),
            "chosen": torch.empty((case["keep"],), dtype=torch.int32, device="cuda")}


# ---------------------------------------------------------------------------------- run
def run(st):
    op = st["op"]
    if op == "layer":
        cc.cc_compress_layer(st["ctx"], st["desc"], st["q"], st["k"], st["v"], st["prior"], st["k_out"],
                             st["v_out"], st["idx"], st["count"], st.get("free_pages"),
                             st.get("out_page_table"), ws=st["ws"])
        return st["out"]
    if op == "layers":
        cc.cc_compress_layers(st["ctx"], st["desc"], st["q"], st["k"], st["v"], st["prior"], st["k_out"],
                              st["v_out"], st["idx"], st["count"], ws=st["ws"])
        return st["out"]
    if op == "host":
        out = st["comp"].run_host(*st["host"], st["prior"], v_in_place=st["v_in_place"],
                                  overlap_readback=st["overlap"])
        return {"k": _bits(out["k_out"]), "v": _bits(out["v_out"]), "idx": out["idx"],
                "count": out["count"]}
    cc.cc_ppl_chunk_scores(st["ctx"], st["logits"], st["targets"], st["nll"], st["score"])
    cc.cc_select_chunks(st["ctx"], st["score"], st["keep"], st["chosen"])
    return {"nll": st["nll"], "score": st["score"], "chosen": st["chosen"]}


def work(case):
    """Bytes read and written once, and multiply-adds, of one pass."""
    if case["op"] == "ppl":
        values = case["chunks"] * case["tokens"] * case["vocab"]
        size = 2 if case["dtype"] == "bf16" else 4
        return {"bytes": float(values * size + 4 * case["chunks"] * case["tokens"]), "flops": 3.0 * values}
    lens, budgets = _ints(case["lens"]), _ints(case["budgets"])
    hkv, row = case["heads_kv"], HEAD_DIM * 2
    keep = sum(min(b, n) for b, n in zip(budgets, lens))
    per_layer = 4.0 * keep * hkv * row + 4.0 * keep * hkv
    flops = 0.0
    if not case["nearest"]:
        per_layer += sum(lens) * hkv * row + len(lens) * case["window"] * case["heads_q"] * row
        flops = 2.0 * case["window"] * case["heads_q"] * HEAD_DIM * sum(lens)
    return {"bytes": case["layers"] * per_layer + 4.0 * sum(lens), "flops": case["layers"] * flops}


def tolerance(case):
    if case["op"] == "ppl":
        return {"rel": 1e-5, "max": 1e-4}
    # whole numbers throughout; scores rounded otherwise in the last places of f32 may swap two
    # tokens at the cut-off, which moves the entries between them by one
    return {"rel": 1e-5, "differ": 0.01}
