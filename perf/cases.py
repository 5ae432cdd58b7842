"""The work whose speed counts: whole calls of the package's public entry points, at the sizes of the
configurations, tests and benchmark of this repository.

Six kinds of call, as a generation makes them:
  cascade   csd_cascade_generate: prompt in, tokens out (host to host), greedy, one neural draft and Max-Gram
  review    csd_review_forward over a committed cache: the target's review of k+1 rows, the draft's decode
  tree      csd_review_forward_tree and csd_tree_accept_greedy: candidates at the first position and a lead chain
  batch     csd_review_forward_batch: blocks of several sequences in one pass over the weights
  prompt    csd_prefill of a prompt (or csd_encoder_forward and the start token), then the review of one row
  accept    csd_spec_accept on given logits: rows of one block each, sampled

Weights are random at the named shapes, from the case's seed.  Two variations, both plain in `_weights`:
the decoder-only models of "cascade" and "tree" are made confident (see `_confident`), so that the greedy
tokens are decided by wide margins, as a trained model's mostly are, and drafts are accepted as often as
trained drafts; the encoder-decoder shape, whose scores are not scaled by the head dimension, gets the
standard deviation 0.005 at which its scores are of unit size.
"""
import math

import numpy as np
import torch

import workloads
from paper_2312_11462_b200 import binding as b

# The weights of a decoder-only cascade: drafts that agree with the target on this share of the vocabulary.
AGREE = 0.7
EMBED_STD = 4.0
CASCADES = {
    "tiny": ("tiny_target", "tiny_draft"),
    "llama7b": ("llama7b", "draft68m"),
}


def listed():
    return [
        # a whole generation with the smallest models: latency of launches and of the host loop
        {"name": "cascade_tiny", "kind": "cascade", "models": "tiny", "prompt": 32, "new": 64, "k": 4},
        # the flagship: 7B-shaped target, 68M-shaped draft, Max-Gram, four drafts a review
        {"name": "cascade_7b", "kind": "cascade", "models": "llama7b", "prompt": 128, "new": 96, "k": 4},
        # one decode step of the draft model
        {"name": "review_draft_m1", "kind": "review", "model": "draft68m", "rows": 1, "cache": 203},
        # the target's review of four drafts, short cache
        {"name": "review_7b_m5", "kind": "review", "model": "llama7b", "rows": 5, "cache": 128},
        # the longest block over a long cache
        {"name": "review_7b_long_m17", "kind": "review", "model": "llama7b", "rows": 17, "cache": 2048},
        # the decoder of the encoder-decoder target: self- and cross-attention
        {"name": "review_t5xxl_m4", "kind": "review", "model": "t5xxl", "rows": 4, "cache": 61, "source": 256},
        # tree attention: eight candidates at the first position, the lead continued by a chain of three
        {"name": "tree_7b_m12", "kind": "tree", "model": "llama7b", "width": 8, "depth": 3, "cache": 300},
        # three sequences served together, ragged blocks and caches
        {"name": "batch_7b_3x", "kind": "batch", "model": "llama7b", "blocks": "5,3,5", "caches": "128,77,301"},
        # a long prompt of the target
        {"name": "prompt_7b_1000", "kind": "prompt", "model": "llama7b", "tokens": 1000},
        # a source text through the encoder, the start token through the decoder
        {"name": "prompt_t5xxl_256", "kind": "prompt", "model": "t5xxl", "tokens": 256},
        # the accept call of one sequence
        {"name": "accept_1x4_v32000", "kind": "accept", "rows": 1, "k": 4, "vocab": 32000, "sigma": 0.5},
        # the accept call of a large batch over a large vocabulary: streams its logits
        {"name": "accept_64x16_v128256", "kind": "accept", "rows": 64, "k": 16, "vocab": 128256, "sigma": 0.5},
    ]


def _between(rng, lo, hi):
    """A whole number from lo to hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cascade", "review", "review", "review", "tree", "batch", "prompt", "prompt", "accept", "accept"])
    if kind == "cascade":
        if rng.random() < 0.5:
            return {"kind": kind, "models": "tiny", "prompt": _between(rng, 8, 64), "new": _between(rng, 8, 64), "k": rng.randint(2, 5)}
        return {"kind": kind, "models": "llama7b", "prompt": _between(rng, 16, 250), "new": _between(rng, 8, 64), "k": rng.randint(2, 6)}
    if kind == "review":
        model = rng.choice(["draft68m", "llama7b", "llama7b", "t5xxl"])
        case = {"kind": kind, "model": model, "rows": rng.randint(1, 17)}
        if model == "t5xxl":
            return dict(case, cache=_between(rng, 1, 170), source=_between(rng, 8, 256))
        return dict(case, cache=_between(rng, 16, 2500 if model == "llama7b" else 430))
    if kind == "tree":
        return {"kind": kind, "model": "llama7b", "width": rng.randint(2, 8), "depth": rng.randint(1, 8), "cache": _between(rng, 16, 2000)}
    if kind == "batch":
        n = rng.randint(2, 4)
        return {"kind": kind, "model": "llama7b", "blocks": ",".join(str(rng.randint(1, 16 // n)) for _ in range(n)),
                "caches": ",".join(str(_between(rng, 16, 1500)) for _ in range(n))}
    if kind == "prompt":
        if rng.random() < 0.3:
            return {"kind": kind, "model": "t5xxl", "tokens": _between(rng, 20, 256)}
        return {"kind": kind, "model": "llama7b", "tokens": _between(rng, 20, 1500)}
    vocab = rng.choice([4096, 32000, 32128, 128256, _between(rng, 500, 128256)])
    return {"kind": kind, "rows": _between(rng, 1, 64), "k": rng.randint(1, 16), "vocab": vocab, "sigma": rng.choice([0.1, 0.5, 2.0])}


def _shape(name, positions):
    s = workloads.SHAPES[name]
    return s if positions <= s.max_seq else workloads.with_max_seq(s, positions)


def _tokens(vocab, n, seed):
    return torch.from_numpy(workloads.make_prompt(vocab, n, seed)).cuda()


def _seeds(seed):
    """Seeds of the parts of a state, all from the case's own."""
    return [int(x) for x in np.random.default_rng(seed).integers(0, 1 << 31, 8)]


def _weights(shape, seed):
    return workloads.make_weights(shape, seed, "cuda", std=0.005 if shape.arch == workloads.ARCH_T5 else 0.02)


def _confident(shape, seed, follows):
    """Random weights whose head knows what follows each token: token t's embedding is large enough to show
    in the residual rows after all layers, and the head's row of follows[t] points along it."""
    blob = workloads.make_weights(shape, seed, "cuda")
    at = {name: (off, shp) for name, off, shp in workloads.blob_layout(shape)[0]}
    part = lambda name: blob[at[name][0]:at[name][0] + at[name][1][0] * at[name][1][1]].view(at[name][1])  # noqa: E731
    embed, head = part("embed"), part("lm_head")
    embed.mul_(EMBED_STD / 0.02)
    head[follows] = embed * (0.02 / EMBED_STD)
    return blob


def _follows(vocab, seed):
    """A permutation: follows[t] is the token that comes after t."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randperm(vocab, generator=g, device="cuda")


def _text(follows, n, seed):
    """A prompt in which about half of the tokens follow from the one before."""
    f = follows.cpu().numpy()
    rng = np.random.default_rng(seed)
    out = [int(rng.integers(0, len(f)))]
    while len(out) < n:
        out.append(int(f[out[-1]]) if rng.random() < 0.5 else int(rng.integers(0, len(f))))
    return np.asarray(out, dtype=np.int32)


def _source(model, n, seed):
    if model.shape.arch == workloads.ARCH_T5:
        model.csd_encoder_forward(_tokens(model.shape.vocab, n, seed))


def prepare(case, seed):
    s = _seeds(seed)
    kind = case["kind"]
    if kind == "accept":
        t, d, tok = workloads.accept_case(case["rows"], case["k"], case["vocab"], case["sigma"], s[0], device="cuda")
        out = tuple(torch.empty(case["rows"], dtype=torch.int32, device="cuda") for _ in range(2))
        ws = b.csd_spec_accept_workspace(case["rows"], case["k"], case["vocab"], "cuda")
        return {"kind": kind, "target": t, "draft": d, "tokens": tok, "seed": s[1], "ws": ws, "out": out}
    if kind == "cascade":
        ts, ds = (workloads.SHAPES[n] for n in CASCADES[case["models"]])
        follows = _follows(ts.vocab, s[0])
        # the draft is right about AGREE of the tokens, the bigram table about a third
        g = torch.Generator(device="cuda")
        g.manual_seed(s[1])
        right = torch.rand(ts.vocab, generator=g, device="cuda")
        other = torch.randint(0, ts.vocab, (ts.vocab,), generator=g, device="cuda")
        shuffled = follows.clone()
        wrong = right >= AGREE
        shuffled[wrong] = follows[wrong].flip(0)
        bigram = torch.where(right < 0.3, follows, other).to(torch.int32)
        models = [b.Model(ts, _confident(ts, s[2], follows)), b.Model(ds, _confident(ds, s[3], shuffled))]
        k = case["k"]
        return {"kind": kind, "prompt": _text(follows, case["prompt"], s[4]), "new": case["new"],
                "cascade": b.Cascade(models, [[k, 0], [0, k]], k, bigram, case["prompt"])}
    if kind == "tree":
        m = 1 + case["width"] + case["depth"]
        shape = _shape(case["model"], case["cache"] + m)
        follows = _follows(shape.vocab, s[0])
        model = b.Model(shape, _confident(shape, s[1], follows))
        f = follows.cpu().numpy()
        toks = workloads.make_prompt(shape.vocab, m, s[2])
        toks[1] = f[toks[0]]                        # the first candidate is right, so is the chain below it but for its last token
        parent = [-1] + [0] * case["width"]
        for i in range(case["depth"]):
            at = 1 + case["width"] + i
            parent.append(1 if i == 0 else at - 1)
            if i + 1 < case["depth"]:
                toks[at] = f[toks[parent[at]]]
        model.csd_prefill(_tokens(shape.vocab, case["cache"], s[3]), 0)
        return {"kind": kind, "model": model, "block": torch.from_numpy(toks).cuda(), "parent": parent, "cache": case["cache"]}
    if kind == "batch":
        rows, caches = ([int(x) for x in case[n].split(",")] for n in ("blocks", "caches"))
        shape = _shape(case["model"], max(c + r for c, r in zip(caches, rows)))
        blob = _weights(shape, s[0])
        models = [b.Model(shape, blob) for _ in rows]
        for i, (m, c) in enumerate(zip(models, caches)):
            m.csd_prefill(_tokens(shape.vocab, c, s[1] + i), 0)
        return {"kind": kind, "models": models, "blocks": [_tokens(shape.vocab, r, s[2] + i) for i, r in enumerate(rows)], "caches": caches}
    if kind == "prompt":
        shape = _shape(case["model"], case["tokens"])
        model = b.Model(shape, _weights(shape, s[0]))
        return {"kind": kind, "model": model, "tokens": _tokens(shape.vocab, case["tokens"], s[1]),
                "start": torch.zeros(1, dtype=torch.int32, device="cuda"), "logits": torch.empty(1, shape.vocab, device="cuda")}
    shape = _shape(case["model"], case["cache"] + case["rows"])
    model = b.Model(shape, _weights(shape, s[0]))
    _source(model, case.get("source", 0), s[1])
    model.csd_prefill(_tokens(shape.vocab, case["cache"], s[2]), 0)
    return {"kind": kind, "model": model, "block": _tokens(shape.vocab, case["rows"], s[3]), "cache": case["cache"],
            "logits": torch.empty(case["rows"], shape.vocab, device="cuda")}


def run(state):
    kind = state["kind"]
    if kind == "accept":
        return b.csd_spec_accept(state["target"], state["draft"], state["tokens"], 1.0, seed=state["seed"],
                                 workspace=state["ws"], out=state["out"])
    if kind == "cascade":
        tokens, stats = state["cascade"].csd_cascade_generate(state["prompt"], state["prompt"], state["new"])
        return {"tokens": tokens, "accepted": stats["accepted"], "drafted": stats["drafted"], "reviews": stats["reviews"]}
    if kind == "tree":
        logits = state["model"].csd_review_forward_tree(state["block"], state["parent"], state["cache"])
        tokens, path, valid = b.csd_tree_accept_greedy(logits, state["block"], state["parent"])
        return {"logits": logits, "tokens": tokens, "path": path, "valid": valid}
    if kind == "batch":
        return b.csd_review_forward_batch(state["models"], state["blocks"], state["caches"])
    if kind == "prompt":
        model, tokens = state["model"], state["tokens"]
        if model.shape.arch == workloads.ARCH_T5:
            model.csd_encoder_forward(tokens)
            return model.csd_review_forward(state["start"], 0, state["logits"])
        n = tokens.numel() - 1
        model.csd_prefill(tokens[:n], 0)
        return model.csd_review_forward(tokens[n:], n, state["logits"])
    return state["model"].csd_review_forward(state["block"], state["cache"], state["logits"])


def _sizes(name):
    """Parameters of a decoder pass (embedding table aside: it is only gathered from), of the head alone, of
    the encoder with the cross-attention projections of its output, and K/V elements per cached position."""
    s = workloads.SHAPES[name]
    size = {n: int(np.prod(shp)) for n, _, shp in workloads.blob_layout(s)[0] if n != "embed"}
    encoder = sum(v for n, v in size.items() if n[0] == "e" or n.endswith((".xk", ".xv")))
    return sum(size.values()) - encoder, size["lm_head"], encoder, 2 * s.n_layers * s.d_inner


def _pass(name, rows, cache, head_rows, source=0):
    """Bytes and operations of one pass of `rows` rows behind `cache` positions, the last head_rows of them through the head."""
    body, head, _, kv = _sizes(name)
    pairs = rows * (cache + source) + rows * (rows + 1) // 2             # (row, key) pairs
    weights = body if head_rows else body - head
    return {"bytes": 2.0 * weights + 2.0 * kv * (cache + source + rows) + 4.0 * workloads.SHAPES[name].vocab * head_rows,
            "flops": 2.0 * (body - head) * rows + 2.0 * head * head_rows + 2.0 * kv * pairs}


def _sum(*parts):
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "accept":
        r, k, v = case["rows"], case["k"], case["vocab"]
        return {"bytes": 4.0 * r * (v * (2 * k + 1) + k + 2), "flops": 4.0 * r * v * (2 * k + 1)}
    if kind == "prompt":
        n = case["tokens"]
        if case["model"] == "t5xxl":
            enc = _sizes("t5xxl")[2]
            s = workloads.SHAPES["t5xxl"]
            return _sum(_pass("t5xxl", 1, 0, 1, n), {"bytes": 2.0 * enc, "flops": 2.0 * enc * n + 4.0 * s.n_enc_layers * s.d_inner * n * n})
        return _pass(case["model"], n, 0, 1)
    if kind == "cascade":
        # the fewest passes: every review accepts all of its k tokens; the draft's and the target's prompt in one pass each
        target, draft = CASCADES[case["models"]]
        p, k, new = case["prompt"], case["k"], case["new"]
        reviews = -(-new // (k + 1))
        parts = []
        for name, n in ((target, reviews), (draft, reviews)):
            one = _pass(name, k + 1, p, k + 1)
            parts += [_pass(name, p, 0, 0), {m: v * n for m, v in one.items()}]
        return _sum(*parts)
    if kind == "tree":
        m = 1 + case["width"] + case["depth"]
        return _pass(case["model"], m, case["cache"], m)
    if kind == "batch":
        rows, caches = ([int(x) for x in case[n].split(",")] for n in ("blocks", "caches"))
        one = _pass(case["model"], sum(rows), 0, sum(rows))
        kv = _sizes(case["model"])[3]
        return _sum(one, {"bytes": 2.0 * kv * sum(caches), "flops": 2.0 * kv * sum(r * c for r, c in zip(rows, caches))})
    return _pass(case["model"], case["rows"], case["cache"], case["rows"], case.get("source", 0))


def tolerance(case):
    kind = case["kind"]
    if kind == "cascade":
        return "exact"
    if kind == "accept":
        return {"rel": 0.0, "differ": 0.01}        # whole numbers; a draft at the edge of acceptance may fall either way
    # Four times the distance between this package's two independent sets of kernels (tensor cores, CUDA cores) on
    # the same weights, caches made by each.  Both round K and V to bf16 before the cache; a last-bit difference
    # upstream moves some entries to the neighbouring bf16 value, and the layers above see that: the distance grows
    # with the depth (2 layers 4e-5; 24 layers 4.5e-4 after a decoder, 1.6e-3 after encoder and decoder; 32 layers
    # 2.2e-3 to 4.1e-3; 7e-4 on the confident weights, whose residual rows the embedding dominates).
    if case["model"] == "draft68m":
        return {"rel": 1.6e-4}
    if case["model"] == "t5xxl":
        return {"rel": 2e-3 if kind == "review" else 6.5e-3}
    return {"rel": 3e-3 if kind == "tree" else 1.6e-2}
