"""The work whose speed counts: calls of the library's public entry points as a serving program makes
them, over the sizes of the named workloads (`workloads.CONFIGS`), of the tests and of the benchmark.

A case is a dict of plain values; its "op" names the entry point:
  prune       Pruner.prune, the fused path (Eq. 10 to the compacted buffer)
  staged      Pruner.score, .select and .compact one after the other: a program that looks at scores
              and energies between the stages
  score       Pruner.score alone
  static      query_score_static, the entry point of callers that may not allocate
  correct     correct, gating and residual correction over the vocabulary
  candidates  branch_candidates, the bonus-branch tokens of every drafted position

Inputs are the seeded synthetic stand-ins of `paper_2605_02218_b200/workloads.py`: rank-R Gaussian
mixtures (or tiles, or video frames that repeat) with log-normal token norms, half of the query
elements correlated with visual tokens, a stack of late hidden states, logits of two models that
mostly agree.  The request sizes of a ragged batch belong to the case ("sizes": the seed they are drawn
from), the contents to the seed given to `prepare`.
"""
import math
import random

import numpy as np
import torch

from paper_2605_02218_b200 import api, workloads

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
VOCAB = 151674            # vocabulary of the correction benchmark and tests


def _case(name, op, **kw):
    return dict({"name": name, "op": op}, **kw)


def listed():
    return [
        # one request, float32 features, one relevance head: the smallest call of an interactive program
        # (time to first token; launches and latency count)
        _case("prune_one_f32", "prune", dtype="f32", batch=1, n_lo=576, n_hi=576, t_lo=32, t_hi=32, d=1024, heads=1,
              rank=32, clusters=8, kind="mixture", keep=64, ratio=0.0, act=4, sizes=0),
        # one request with the token count of the paper's own system, 768 visual tokens kept down to 64
        _case("prune_one_bf16", "prune", dtype="bf16", batch=1, n_lo=768, n_hi=768, t_lo=32, t_hi=32, d=2048, heads=16,
              rank=64, clusters=8, kind="mixture", keep=64, ratio=0.0, act=4, sizes=0),
        # an ordinary serving batch of standard-resolution images
        _case("prune_batch", "prune", dtype="bf16", batch=16, n_lo=576, n_hi=576, t_lo=64, t_hi=64, d=2048, heads=16,
              rank=64, clusters=8, kind="mixture", keep=0, ratio=0.25, act=4, sizes=0),
        # high-resolution images cut into five tiles each, a wide model
        _case("prune_tiles", "prune", dtype="bf16", batch=32, n_lo=2880, n_hi=2880, t_lo=128, t_hi=128, d=4096, heads=32,
              rank=128, clusters=5, kind="tiles", keep=0, ratio=0.10, act=4, sizes=0),
        # dynamic-resolution images: ragged token and query counts in one packed batch
        _case("prune_ragged", "prune", dtype="bf16", batch=64, n_lo=256, n_hi=4096, t_lo=16, t_hi=256, d=1536, heads=12,
              rank=64, clusters=8, kind="mixture", keep=0, ratio=0.20, act=4, sizes=3),
        # video: 16384 tokens a request, consecutive frames nearly alike (the largest case)
        _case("prune_video", "prune", dtype="bf16", batch=8, n_lo=16384, n_hi=16384, t_lo=64, t_hi=64, d=3584, heads=28,
              rank=64, clusters=8, kind="video", keep=1024, ratio=0.0, act=4, sizes=0),
        # the stages called one by one on a small float32 batch of odd sizes
        _case("staged_f32_ragged", "staged", dtype="f32", batch=5, n_lo=140, n_hi=1100, t_lo=3, t_hi=70, d=520, heads=3,
              rank=16, clusters=8, kind="mixture", keep=0, ratio=0.25, act=4, sizes=7),
        # Eq. 10 on the embeddings as they are (no projection heads): both scores and their fusion
        _case("score_identity", "score", dtype="bf16", batch=16, n_lo=400, n_hi=729, t_lo=9, t_hi=64, d=2048, heads=0,
              rank=64, clusters=8, kind="mixture", keep=0, ratio=0.25, act=4, sizes=5),
        # the same score from inside a loop whose memory pool is handed out
        _case("static_score", "static", dtype="bf16", batch=4, n_lo=576, n_hi=576, t_lo=32, t_hi=32, d=1024, heads=0,
              rank=32, clusters=8, kind="mixture", keep=0, ratio=0.25, act=0, sizes=0),
        # the positions of one drafted block: what a single session corrects at a time
        _case("correct_block", "correct", dtype="f16", rows=8, vocab=VOCAB),
        # the positions of many sessions in one call
        _case("correct_many", "correct", dtype="f16", rows=1024, vocab=VOCAB),
        # bonus-branch candidates of the drafted blocks of four sessions
        _case("candidates", "candidates", dtype="f16", rows=32, vocab=VOCAB, fan=8, rho=0.6, block=8),
    ]


# No drawn case does more work than the largest listed one (131072 tokens of 3584 features, 28 heads).
_MOST_FLOPS, _MOST_BYTES = 2.5e12, 4.0e9


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: entry points by how often a program calls them, sizes spread
    over their logarithm, most of them odd."""
    what = rng.random()
    if what < 0.20:
        return dict(op="correct", dtype=rng.choice(["f16", "f16", "bf16", "f32"]), rows=_log_int(rng, 1, 512),
                    vocab=rng.choice([VOCAB, _log_int(rng, 30000, 200000)]))
    if what < 0.30:
        return dict(op="candidates", dtype=rng.choice(["f16", "f16", "bf16", "f32"]), rows=_log_int(rng, 1, 256),
                    vocab=rng.choice([VOCAB, _log_int(rng, 30000, 200000)]), fan=rng.randint(2, 16),
                    rho=rng.choice([0.5, 0.6, 0.8]), block=rng.randint(4, 12))
    op = "static" if what < 0.36 else "score" if what < 0.46 else "staged" if what < 0.56 else "prune"
    heads = 0 if op == "static" else rng.choice([0, 0, 1, 8, 12]) if op == "score" else rng.choice([1, 2, 3, 8, 12, 16, 28, 32])
    c = dict(op=op, dtype="f32" if rng.random() < 0.2 else "bf16", batch=_log_int(rng, 1, 64),
             n_lo=0, n_hi=_log_int(rng, 256, 16384), t_lo=0, t_hi=_log_int(rng, 16, 256),
             d=8 * _log_int(rng, 64, 512), heads=heads, rank=rng.choice([16, 32, 64, 128]), clusters=rng.randint(4, 10),
             kind=rng.choice(["mixture", "mixture", "tiles", "video"]), keep=0, ratio=rng.choice([0.0625, 0.1, 0.2, 0.25, 0.3]),
             act=0 if op == "static" else rng.choice([2, 4, 4, 6]), sizes=rng.randint(1, 10 ** 6))
    ragged = rng.random() < 0.6
    c["n_lo"] = max(64, c["n_hi"] // rng.randint(2, 8)) if ragged else c["n_hi"]
    c["t_lo"] = max(3, c["t_hi"] // rng.randint(2, 8)) if ragged else c["t_hi"]
    if op == "static":
        c["batch"] = min(c["batch"], max(1, api.STATIC_MAX_QUERY_ELEMS // (c["t_hi"] * c["d"])))
    # the identity embedding scores every token against every query element at full width
    most = (_MOST_FLOPS, _MOST_BYTES) if heads else (1.0e11, 1.0e9)
    while True:
        w = work(c)
        if w["flops"] <= most[0] and w["bytes"] <= most[1]:
            return c
        if c["batch"] > 1:
            c["batch"] = max(1, c["batch"] * 2 // 3)
        else:
            c["n_hi"] = c["n_hi"] * 2 // 3
            c["n_lo"] = min(c["n_lo"], c["n_hi"])


def _sizes(case):
    r = random.Random(case["sizes"])
    n = [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case["batch"])]
    t = [r.randint(case["t_lo"], case["t_hi"]) for _ in range(case["batch"])]
    return n, t


def _keeps(case, n):
    return [min(case["keep"], v) if case["keep"] else workloads.keep_from_ratio(v, case["ratio"]) for v in n]


def prepare(case, seed):
    dev = "cuda:0"
    if case["op"] in ("correct", "candidates"):
        data = workloads.make_logits(seed=seed, rows=case["rows"], vocab=case["vocab"], dtype=DTYPES[case["dtype"]], device=dev)
        st = dict(op=case["op"], data=data)
        if case["op"] == "candidates":
            st["fan"] = [api.fanout(case["fan"], case["rho"], j % case["block"]) for j in range(case["rows"])]
        return st
    n, t = _sizes(case)
    wl = workloads.make_workload(case["op"], seed=seed, dtype=DTYPES[case["dtype"]], batch=case["batch"], sizes=(n, t),
                                 d=case["d"], n_heads=case["heads"], rank=case["rank"], n_clusters=case["clusters"],
                                 kind=case["kind"], keep=_keeps(case, n), act_layers=case["act"], device=dev)
    st = dict(op=case["op"], wl=wl)
    if case["op"] == "static":
        st["out"] = torch.empty(wl.total_vis, dtype=torch.float32, device=dev)
    else:
        st["pruner"] = api.Pruner.for_workload(wl)
        st["call"] = st["pruner"].marshal(wl)
    return st


def run(state):
    op = state["op"]
    if op == "prune":
        return state["pruner"].prune(state["call"])
    if op == "score":
        return state["pruner"].score(state["call"])
    if op == "staged":
        pr, m = state["pruner"], state["call"]
        s_query, s_act, s_fused = pr.score(m)
        keep_idx, keep_off, presel, presel_off, energy = pr.select(m, s_fused)
        out, pos = pr.compact(m, keep_idx, keep_off)
        return dict(s_query=s_query, s_act=s_act, s_fused=s_fused, keep_idx=keep_idx, keep_off=keep_off, presel=presel,
                    presel_off=presel_off, energy=energy, out=out, pos=pos)
    if op == "static":
        wl = state["wl"]
        return api.query_score_static(wl.X, wl.Q, wl.vis_offsets, wl.txt_offsets, out=state["out"])
    d = state["data"]
    if op == "correct":
        return api.correct(d["z_draft"], d["z_target"], d["uniforms"], 0.02, d["drafted"], vocab=d["vocab"])
    return api.branch_candidates(d["z_draft"], state["fan"], d["drafted"], vocab=d["vocab"])


def work(case):
    """Every input read once, every output written once; the products of Eq. 10 (projection and cosines),
    of the Gram matrix (its symmetric half) and of four multiplications by it with r + 16 vectors."""
    if case["op"] in ("correct", "candidates"):
        e = 4 if case["dtype"] == "f32" else 2
        entries = float(case["rows"]) * case["vocab"]
        if case["op"] == "correct":
            return {"bytes": 2 * entries * e + 28.0 * case["rows"], "flops": 12 * entries}
        return {"bytes": entries * e, "flops": entries}
    n, t = _sizes(case)
    d, heads, act = case["d"], case["heads"], case["act"]
    e = 4 if case["dtype"] == "f32" else 2
    width = heads * 128 if heads else d
    rows, queries = float(sum(n)), float(sum(t))
    flops = 2.0 * width * sum(a * b for a, b in zip(n, t)) + (2.0 * (rows + queries) * d * width if heads else 0.0)
    size = (rows + queries) * d * e + (2.0 * width * d * e if heads else 0.0)
    if act:
        size += (act + 1) * rows * d * e
        flops += 3.0 * act * rows * d
    if case["op"] == "static":
        return {"bytes": size + 4 * rows, "flops": flops}
    if case["op"] in ("score", "staged"):
        size += 12 * rows
    if case["op"] in ("prune", "staged"):
        for v, k in zip(n, _keeps(case, n)):
            m = min(v, 2 * k)
            if k < m:
                r = max(1, min(-(-k // 2), 128, m - 1, d - 1))
                flops += float(m) * m * d + 4 * 2.0 * m * m * (r + 16)
            size += k * (d * e + 4.0)
            if case["op"] == "staged":
                size += 8.0 * m + 4.0 * k
    return {"bytes": size, "flops": flops}


def tolerance(case):
    if case["op"] == "candidates":
        return "exact"
    if case["op"] in ("score", "static") and not case["heads"]:
        return {"rel": 1e-5}                                  # float32 sums over at most 4096 features
    if case["op"] == "score":
        return {"rel": 1e-5 if case["dtype"] == "bf16" else 3e-5}   # float32 operands in three bf16 terms, about 2^-17
    if case["op"] == "correct":
        return {"rel": 1e-5, "differ": 0.005}                 # float32 softmax sums; a draw at a step of the distribution
    if case["op"] == "staged":
        return {"rel": 1e-4, "differ": 0.005}                 # energies of the truncated SVD: operands of 16 mantissa bits
    return {"rel": 1e-2, "differ": 0.005}                     # bit copies of the kept rows; near ties at the cut
