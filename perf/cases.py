"""What is timed: the calls that a program around this library makes for a prompt.

A case is one kind of call at one size:

  score    importance of every prompt key (`Session.score`), with or without the log-sum-exp
           that the caller's prefill attention may have kept
  select   search for the ratio under the budget and compaction (`Session.search`,
           `Session.compact`), from given scores, so that every result is exact
  decode   tokens generated against a compressed cache (`Session.decode`), either all layers in one
           call or layer by layer as a model does, whose next layer's query depends on this
           layer's output

Shapes are the repository's configurations (their layers, heads, head sizes, prompt lengths, budgets
and batches) and generic ones around them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_03409_b200 import workloads as wl
from paper_2412_03409_b200.session import Session

DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}


def _score(name, B, L, H, D, N, dtype="bf16", lse=False):
    return {"name": name, "kind": "score", "B": B, "L": L, "H": H, "D": D, "N": N, "dtype": dtype, "lse": lse}


def _select(name, B, L, H, D, N, ratio, dtype="bf16"):
    return {"name": name, "kind": "select", "B": B, "L": L, "H": H, "D": D, "N": N, "dtype": dtype, "ratio": ratio}


def _decode(name, B, L, H, D, N, ratio, tokens, layerwise=False, convs=1, evict=0, dtype="bf16"):
    return {"name": name, "kind": "decode", "B": B, "L": L, "H": H, "D": D, "N": N, "dtype": dtype, "ratio": ratio,
            "tokens": tokens, "layerwise": layerwise, "convs": convs, "evict": evict}


def listed():
    return [
        # the smallest call: a unit test's or a toy model's prompt in fp32, all launch latency
        _score("score_tiny_fp32", 1, 4, 4, 64, 128, dtype="fp32"),
        # fp32 users (checking another implementation, small research models), a ragged prompt
        _score("score_fp32_ragged", 1, 8, 16, 128, 777, dtype="fp32"),
        # one image prompt of a chat: the latency a user waits for before the first token
        _score("score_7b_b1", 1, 32, 32, 128, 640),
        # a batch of multi-image prompts whose prefill attention kept its log-sum-exp
        _score("score_13b_b2_lse", 2, 40, 40, 128, 2048, lse=True),
        # a long high-resolution prompt: scoring is most of the compression
        _score("score_long_b1", 1, 32, 32, 128, 16384),
        # selection and compaction of one chat prompt
        _select("select_7b_b1", 1, 32, 32, 128, 640, 0.2),
        # the same for two long prompts
        _select("select_long_b2", 2, 32, 32, 128, 16384, 0.05),
        # a chat server's single-prompt decoding; four conversations served in turn
        _decode("decode_7b_b1", 1, 32, 32, 128, 640, 0.2, tokens=8, convs=4),
        # the same from inside a model: one call per layer
        _decode("decode_7b_b1_layerwise", 1, 32, 32, 128, 640, 0.2, tokens=2, layerwise=True, convs=4),
        # a batch with decode-time pruning on: long answers that keep their proportion of the cache
        _decode("decode_7b_b16_pruned", 16, 32, 32, 128, 640, 0.2, tokens=12, evict=4),
        # a batch of multi-image prompts, one call per layer
        _decode("decode_13b_b8_layerwise", 8, 40, 40, 128, 2048, 0.2, tokens=2, layerwise=True),
        # long prompts in one call: the largest caches
        _decode("decode_long_b4", 4, 32, 32, 128, 16384, 0.05, tokens=4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _model(rng):
    """Layers, heads, head size: the two configured models' and smaller generic ones."""
    return rng.choice([(32, 32, 128), (32, 32, 128), (40, 40, 128), (24, 16, 64), (28, 24, 128), (16, 8, 64)])


_SCORE_MAX = 32 * 32 * 16384 * 16385 * 128          # the long listed case
_SCORE32_MAX = 8 * 16 * 777 * 778 * 128             # the ragged fp32 case
_KV_MAX = 2 * 32 * 32 * 16384 * 128                 # prompt elements of K of the listed selection
_CACHE_MAX = 4 * 32 * 32 * 128 * int(0.05 * 16384)  # cache elements of K of the listed long decode


def draw(rng):
    kind = rng.choice(["score", "score", "select", "decode", "decode", "decode"])
    while True:
        if kind == "score":
            if rng.random() < 0.25:
                c = _score("", rng.choice([1, 1, 2]), _log_int(rng, 2, 12), _log_int(rng, 2, 16), rng.choice([64, 128]),
                           _log_int(rng, 64, 1500), "fp32", rng.random() < 0.25)
                ok = c["B"] * c["L"] * c["H"] * c["N"] * (c["N"] + 1) * c["D"] <= _SCORE32_MAX
            else:
                L, H, D = _model(rng)
                c = _score("", _log_int(rng, 1, 16), L, H, D, _log_int(rng, 64, 16384), "bf16", rng.random() < 0.3)
                ok = (c["B"] * L * H * c["N"] * (c["N"] + 1) * D <= _SCORE_MAX
                      and c["B"] * L * H * c["N"] * D <= 32 * 32 * 16384 * 128)
        elif kind == "select":
            L, H, D = _model(rng)
            c = _select("", _log_int(rng, 1, 16), L, H, D, _log_int(rng, 128, 16384), round(rng.uniform(0.05, 0.5), 3),
                        rng.choice(["bf16", "bf16", "bf16", "fp32"]))
            ok = c["B"] * L * H * c["N"] * D * (2 if c["dtype"] == "fp32" else 1) <= _KV_MAX and \
                c["N"] * c["ratio"] >= 8 and \
                c["B"] * L * H * c["N"] * D * c["ratio"] * (2 if c["dtype"] == "fp32" else 1) <= _KV_MAX * 0.05
        else:
            L, H, D = _model(rng)
            layerwise = rng.random() < 0.5
            evict = 0 if layerwise else rng.choice([0, 0, 4])
            c = _decode("", _log_int(rng, 1, 16), L, H, D, _log_int(rng, 64, 16384), round(rng.uniform(0.05, 0.5), 3),
                        tokens=12 if evict else (2 if layerwise else 4), layerwise=layerwise, evict=evict,
                        dtype=rng.choice(["bf16", "bf16", "bf16", "fp32"]))
            ok = c["N"] * c["ratio"] >= 8 and c["B"] * L * H * c["N"] * D <= _KV_MAX and \
                c["B"] * L * H * D * c["N"] * c["ratio"] * (2 if c["dtype"] == "fp32" else 1) * \
                c["tokens"] / 4 <= _CACHE_MAX
            # several conversations in turn when one cache is small enough to stay in L2
            if ok and c["B"] * L * H * D * c["N"] * c["ratio"] * 4 < 1 << 27 and not evict:
                c["convs"] = 4
        if ok:
            c.pop("name")
            return c


def _budget_rows(c):
    return int(math.floor(c["ratio"] * c["L"] * c["N"] + 1e-9))


def _layer_factors(c, seed):
    """How sharply each layer attends: log-uniform, as the prompts of the configurations have it."""
    rng = np.random.default_rng(seed * 7919 + 17)
    return np.exp(rng.uniform(math.log(0.5), math.log(4.0), size=(c["B"], c["L"])))


def _normal(shape, dtype, gen):
    """Standard normal tensor [B, L, ...], a layer at a time to bound the fp32 temporary."""
    out = torch.empty(shape, dtype=dtype, device="cuda")
    for b in range(shape[0]):
        for l in range(shape[1]):
            out[b, l] = torch.randn(shape[2:], generator=gen, device="cuda")
    return out


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * seed + 11)
    return g


def _session(c, decode_cap=0):
    return Session(c["B"], c["L"], c["H"], c["D"], c["N"], DTYPES[c["dtype"]],
                   np.full(c["L"], 1.0 / math.sqrt(c["D"]), np.float32), decode_cap=decode_cap,
                   max_budget_rows=_budget_rows(c) if "ratio" in c else c["L"], evict_distance=c.get("evict", 0))


def _scores(c, seed):
    s = np.stack([wl.synthetic_scores(c["L"], c["N"], 1000 * seed + b) for b in range(c["B"])])
    return torch.from_numpy(s).cuda()


def _prepare_score(c, seed):
    B, L, H, N, D = c["B"], c["L"], c["H"], c["N"], c["D"]
    g = _gen(seed)
    dt = DTYPES[c["dtype"]]
    s = _session(c)
    q = _normal((B, L, H, N, D), dt, g)
    k = torch.empty((B, L, H, N, D), dtype=dt, device="cuda")
    f = _layer_factors(c, seed)
    # text positions at both ends keep unit keys, image positions carry the layer's factor
    lo, hi = N // 20, N - N // 10
    for b in range(B):
        for l in range(L):
            x = torch.randn((H, N, D), generator=g, device="cuda")
            x[:, lo:hi] *= float(f[b, l])
            k[b, l] = x
    lse = None
    if c["lse"]:  # what a prefill attention kernel of the caller returns beside its output
        lse = torch.empty((B, L, H, N), dtype=torch.float32, device="cuda")
        mask = torch.ones((N, N), dtype=torch.bool, device="cuda").triu(1)
        step = max(1, (1 << 28) // (N * N))
        for b in range(B):
            for l in range(L):
                for h in range(0, H, step):
                    x = torch.matmul(q[b, l, h:h + step].float(), k[b, l, h:h + step].float().transpose(-1, -2))
                    x *= 1.0 / math.sqrt(D)
                    lse[b, l, h:h + step] = torch.logsumexp(x.masked_fill_(mask, -math.inf), dim=-1)
    return {"kind": "score", "s": s, "q": q, "k": k, "lse": lse}


def _prepare_select(c, seed):
    B, L, H, N, D = c["B"], c["L"], c["H"], c["N"], c["D"]
    g = _gen(seed)
    dt = DTYPES[c["dtype"]]
    s = _session(c)
    s.kept.zero_()      # entries past a layer's length are never written
    s.cache.k.zero_()   # and neither are rows the budget leaves over
    s.cache.v.zero_()
    return {"kind": "select", "s": s, "budget": _budget_rows(c), "scores": _scores(c, seed),
            "k": _normal((B, L, H, N, D), dt, g), "v": _normal((B, L, H, N, D), dt, g)}


def _prepare_decode(c, seed):
    B, L, H, N, D = c["B"], c["L"], c["H"], c["N"], c["D"]
    dt = DTYPES[c["dtype"]]
    T = c["tokens"]
    convs = []
    for i in range(c["convs"]):
        g = _gen(seed * 16 + i)
        s = _session(c, decode_cap=T)
        s.cache.k.zero_()
        s.cache.v.zero_()
        s.search(_budget_rows(c), scores=_scores(c, seed * 16 + i))
        s.compact(_normal((B, L, H, N, D), dt, g), _normal((B, L, H, N, D), dt, g))
        tok = [[torch.randn((B, L, H, D), generator=g, device="cuda").to(dt) for _ in range(3)] for _ in range(T)]
        outs = [torch.zeros((B, L, H, D), dtype=dt, device="cuda") for _ in range(T)]
        # the compressed prompt's state, to which another answer to the same prompt goes back
        keep = [x.clone() for x in _growing(s.cache)]
        convs.append({"s": s, "tok": tok, "outs": outs, "keep": keep})
    torch.cuda.synchronize()
    return {"kind": "decode", "convs": convs, "layers": L, "layerwise": c["layerwise"], "tokens": T}


def _growing(cache):
    """What decoding changes besides the rows: lengths, and with pruning the tokens' places."""
    return [cache.len] + ([cache.gen, cache.slot_ring] if cache.evict_distance > 0 else [])


def prepare(case, seed):
    return {"score": _prepare_score, "select": _prepare_select, "decode": _prepare_decode}[case["kind"]](case, seed)


def run(state):
    kind = state["kind"]
    if kind == "score":
        return {"scores": state["s"].score(state["q"], state["k"], lse=state["lse"])}
    if kind == "select":
        s = state["s"]
        s.search(state["budget"], scores=state["scores"])
        s.compact(state["k"], state["v"])
        return {"order": s.order, "cum": s.cum, "len": s.len, "p": s.p, "iters": s.iters, "kept": s.kept,
                "k": s.cache.k, "v": s.cache.v, "row_offset": s.cache.row_offset, "cache_len": s.cache.len,
                "cap": s.cache.cap, "status": s.status}
    # another answer to every conversation's prompt: back to the compressed prompt, then token by token
    convs = state["convs"]
    for c in convs:
        for x, x0 in zip(_growing(c["s"].cache), c["keep"]):
            x.copy_(x0)
    for t in range(state["tokens"]):
        for c in convs:
            q, k_new, v_new = c["tok"][t]
            if state["layerwise"]:
                for l in range(state["layers"]):
                    c["s"].decode(q, k_new, v_new, out=c["outs"][t], layer_begin=l, layer_end=l + 1)
            else:
                c["s"].decode(q, k_new, v_new, out=c["outs"][t])
    return [{"out": c["outs"], "k": c["s"].cache.k, "v": c["s"].cache.v, "state": _growing(c["s"].cache),
             "status": c["s"].status} for c in convs]


def work(case):
    c = case
    B, L, H, N, D = c["B"], c["L"], c["H"], c["N"], c["D"]
    es = 4 if c["dtype"] == "fp32" else 2
    row = H * D * es
    if c["kind"] == "score":
        # Q and K (and the log-sum-exp) read, scores written; the causal half of one Q K^T
        return {"bytes": B * L * (2 * N * row + (4 * H * N if c["lse"] else 0) + 4 * N), "flops": B * L * H * N * (N + 1) * D}
    rows = B * _budget_rows(c)
    if c["kind"] == "select":
        # scores in; order, sums, retained lists out; the retained rows of K and V in and out
        return {"bytes": B * L * N * (4 + 4 + 8) + 4 * rows + 4 * rows * row, "flops": 0}
    total, kept = 0, rows
    for t in range(c["tokens"]):
        grow = c["ratio"] * B * L if c["evict"] and t >= c["evict"] else B * L
        kept += grow
        # every cached row but the new one read, the new K and V rows read and written, q in, out out
        total += 2 * (kept - B * L) * row + 6 * B * L * row
    return {"bytes": int(c["convs"] * total), "flops": int(c["convs"] * c["tokens"] * 4 * kept * H * D)}


def tolerance(case):
    """Four times what the path differs by from itself in 64 bits: scores 2e-7 at 2048 tokens (5e-7 allowed for at
    16384), fp32 decode outputs 2e-7 at 150 rows and likewise, bf16 decode outputs 1.65e-3 (their own rounding)."""
    if case["kind"] == "select":
        return "exact"
    if case["kind"] == "score" or case["dtype"] == "fp32":
        return {"rel": 2e-6}
    return {"rel": 6.5e-3}
