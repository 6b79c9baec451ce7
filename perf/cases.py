"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values; ``listed`` names twelve of them, ``draw`` makes more of the same ranges.  ``prepare``
builds what a program has in hand before the call, ``run`` is one pass through the public entry points.

Kinds
  step      one decoding step from host integers: prompt-lookup retrieval, ``Model.step_host``, window refill
  tree      one verification step of resident trees (one or several sequences): ``verify_step`` with its logits,
            ``node_topk`` where the template has siblings, ``accept``, ``compact_kv``
  prefill   a prompt into an empty cache: ``Model.prefill``
  generate  a whole request: prefill, then ``Model.decode_device`` for a number of steps
  ops       op level, for programs that bring their own decoder: ``tree_attention`` and ``argmax_accept``

The models are random but behave like trained ones where that matters to a decoder: the LM head is the embedding table
under ten permutations of decreasing weight, so that every position has a clear next token and clear runners-up (drafts
can then be planted, and tokens do not hang on the last bit of a logit).  Projections are N(0, 0.02), those that write to
the residual stream scaled by 1 / sqrt(2 * layers), the embedding N(0, 1), norm gains 1.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2406_17404_b200 as trj

# the decoder shapes of this repository's configurations
MODELS = {
    "tiny": dict(n_layers=2, d_model=256, n_heads=4, head_dim=64, d_ff=688, vocab=1024, dtype="f32", n_kv_heads=4,
                 rope_theta=10000.0),
    "llama7b": dict(n_layers=32, d_model=4096, n_heads=32, head_dim=128, d_ff=11008, vocab=32000, dtype="bf16",
                    n_kv_heads=32, rope_theta=10000.0),
    "llama3_8b": dict(n_layers=32, d_model=4096, n_heads=32, head_dim=128, d_ff=14336, vocab=128256, dtype="bf16",
                      n_kv_heads=8, rope_theta=500000.0),
}
CANDIDATES = [1.0, 0.7, 0.63, 0.57, 0.52, 0.48, 0.44, 0.41, 0.38, 0.36]   # weights of the ten permutations


def listed():
    return [
        # the smallest decoder in fp32 (the parity configuration): latency of launches and of the host
        {"name": "step_tiny_f32", "kind": "step", "model": "tiny", "prefix": 64, "window": 4, "branches": 2, "branch_len": 3},
        # the smallest step of a 7B decoder: a Jacobi window of 4 without retrieval, an early position
        {"name": "step_7b_window4", "kind": "step", "model": "llama7b", "prefix": 137, "window": 4, "branches": 0, "branch_len": 0},
        # the step that the benchmark is quoted on: 32 drafts (window 5, nine retrieved 3-grams) after 512 tokens
        {"name": "step_7b_32drafts", "kind": "step", "model": "llama7b", "prefix": 512, "window": 5, "branches": 9, "branch_len": 3},
        # the paper-sized template: 63 nodes with top-10 siblings, a retrieval path of 5 and the root
        {"name": "template_7b_69rows", "kind": "tree", "model": "llama7b", "batch": 1, "prefix_lo": 1023, "prefix_hi": 1023,
         "rows_lo": 69, "rows_hi": 69, "depth": 5, "top_k": 10, "layout": 1},
        # grouped-query attention and a 128 256-way vocabulary, far into a conversation
        {"name": "tree_8b_prefix4000", "kind": "tree", "model": "llama3_8b", "batch": 1, "prefix_lo": 4000, "prefix_hi": 4000,
         "rows_lo": 33, "rows_hi": 33, "depth": 6, "top_k": 0, "layout": 2},
        # a server's batch: eight sequences of unequal length, trees of unequal size
        {"name": "batch8_7b", "kind": "tree", "model": "llama7b", "batch": 8, "prefix_lo": 200, "prefix_hi": 1000,
         "rows_lo": 16, "rows_hi": 64, "depth": 6, "top_k": 0, "layout": 3},
        # a short odd prompt, where the weights' stream still counts, and the longest one, which is all tensor cores
        {"name": "prefill_8b_333", "kind": "prefill", "model": "llama3_8b", "tokens": 333},
        {"name": "prefill_7b_2048", "kind": "prefill", "model": "llama7b", "tokens": 2048},
        # one request from prompt to answer without the host between steps
        {"name": "generate_7b", "kind": "generate", "model": "llama7b", "tokens": 200, "window": 5, "branches": 9, "branch_len": 3, "steps": 12},
        # op level: a 64-row tree over 1024 keys with its arg-max and acceptance; a long context; a ragged batch
        {"name": "ops_1024_64rows", "kind": "ops", "batch": 1, "kv_heads": 32, "prefix_lo": 1024, "prefix_hi": 1024, "rows_lo": 64,
         "rows_hi": 64, "depth": 6, "vocab": 32000, "logits": "bf16", "layout": 4},
        {"name": "ops_8192_128rows", "kind": "ops", "batch": 1, "kv_heads": 32, "prefix_lo": 8192, "prefix_hi": 8192, "rows_lo": 128,
         "rows_hi": 128, "depth": 8, "vocab": 0, "logits": "bf16", "layout": 5},
        {"name": "ops_batch8_ragged", "kind": "ops", "batch": 8, "kv_heads": 32, "prefix_lo": 256, "prefix_hi": 4096, "rows_lo": 16,
         "rows_hi": 64, "depth": 6, "vocab": 32000, "logits": "bf16", "layout": 6},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "tree", "batch", "prefill", "generate", "ops"])
    if kind == "step":
        model = rng.choice(["tiny", "llama7b", "llama7b"])
        r, length = rng.randint(0, 9), rng.randint(1, 5)
        return {"kind": "step", "model": model, "prefix": _log(rng, 48, 512 if model == "tiny" else 2048), "window": rng.randint(1, 8),
                "branches": r, "branch_len": length if r else 0}
    if kind == "tree":
        model = rng.choice(["llama7b", "llama3_8b"])
        s = _log(rng, 64, 4096 if model == "llama7b" else 8192)
        m = rng.randint(8, 128)
        return {"kind": "tree", "model": model, "batch": 1, "prefix_lo": s, "prefix_hi": s, "rows_lo": m, "rows_hi": m,
                "depth": rng.randint(3, 7), "top_k": rng.choice([0, 4, 10]), "layout": rng.randint(0, 1 << 20)}
    if kind == "batch":
        lo = rng.randint(64, 512)
        return {"kind": "tree", "model": rng.choice(["llama7b", "llama3_8b"]), "batch": rng.randint(2, 12), "prefix_lo": lo,
                "prefix_hi": rng.randint(lo, 1024), "rows_lo": rng.randint(5, 16), "rows_hi": rng.randint(24, 64), "depth": 4,
                "top_k": 0, "layout": rng.randint(0, 1 << 20)}
    if kind == "prefill":
        model = rng.choice(["llama7b", "llama3_8b"])
        return {"kind": "prefill", "model": model, "tokens": _log(rng, 16, 2047 if model == "llama7b" else 1800)}
    if kind == "generate":
        return {"kind": "generate", "model": "llama7b", "tokens": _log(rng, 64, 512), "window": rng.randint(3, 6),
                "branches": rng.randint(2, 9), "branch_len": rng.randint(2, 4), "steps": rng.randint(4, 12)}
    many = rng.random() < 0.5
    lo = _log(rng, 256, 4096) if many else _log(rng, 128, 8192)
    m = rng.randint(16, 64) if many else rng.randint(8, 128)
    return {"kind": "ops", "batch": rng.randint(2, 8) if many else 1, "kv_heads": rng.choice([32, 8]), "prefix_lo": lo,
            "prefix_hi": rng.randint(lo, 4096) if many else lo, "rows_lo": 8 if many else m, "rows_hi": m, "depth": 5,
            "vocab": rng.choice([0, 32000, 128256]), "logits": rng.choice(["bf16", "f32"]), "layout": rng.randint(0, 1 << 20)}


# ------------------------------------------------------------------------------------------------ inputs
def _cfg(name):
    return SimpleNamespace(rms_eps=1e-5, **MODELS[name])


def _sizes(case):
    """(prefix lengths, tree sizes) of the batch: part of the case, not of the seed."""
    r = random.Random(case["layout"])
    n = case["batch"]
    return ([r.randint(case["prefix_lo"], case["prefix_hi"]) for _ in range(n)],
            [r.randint(case["rows_lo"], case["rows_hi"]) for _ in range(n)])


def _tree(r, m, depth):
    """Parent pointers of a random tree: a chain of the stated depth first, then children of shallower rows."""
    parent, deep = [-1], [0]
    for i in range(1, m):
        p = i - 1 if i <= depth else r.choice([j for j in range(i) if deep[j] < depth])
        parent.append(p)
        deep.append(deep[p] + 1)
    return np.asarray(parent, np.int32)


def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


def _trees(case, next_token, roots, seed):
    """The batch's trees on the device.  A row's token is its parent's next token with probability 0.6 (acceptance as
    with good drafts), else uniform.  ``next_token`` [rows before it, token] -> the prediction of a row."""
    r, shape = random.Random(seed * 7919 + 17), random.Random(case["layout"] + 1)
    tokens, parents, depths, ancs, off = [], [], [], [], [0]
    for b, m in enumerate(_sizes(case)[1]):
        parent = _tree(shape, m, min(case["depth"], m - 1))
        depth, anc = trj.tree_from_parents(parent)
        tok = [roots[b]]
        for i in range(1, m):
            want = next_token(off[-1] + int(parent[i]), tok[parent[i]])
            tok.append(want if r.random() < 0.6 else r.randrange(case.get("vocab") or 1000))
        tokens += tok
        parents.append(parent)
        depths.append(depth)
        ancs.append(anc)
        off.append(off[-1] + m)
    return SimpleNamespace(tokens=_i32(tokens), parent=_i32(np.concatenate(parents)), depth=_i32(np.concatenate(depths)),
                           anc=torch.from_numpy(np.concatenate(ancs).view(np.int64)).cuda(), row_off=_i32(off))


def _model(name, seed, max_batch, max_seq, max_rows):
    """(model, next-token table): weights drawn on the device, see the head of this file."""
    c = _cfg(name)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dt = torch.bfloat16 if c.dtype == "bf16" else torch.float32

    def mat(rows, cols, std=0.02):
        return torch.randn(rows, cols, generator=g, device="cuda", dtype=dt).mul_(std)
    d, f, hd, kv = c.d_model, c.d_ff, c.n_heads * c.head_dim, c.n_kv_heads * c.head_dim
    back = 0.02 / math.sqrt(2 * c.n_layers)
    one = torch.ones(d, device="cuda")
    layers = [{"attn_norm": one, "wqkv": mat(hd + 2 * kv, d), "wo": mat(d, hd, back), "mlp_norm": one,
               "w_gate_up": mat(2 * f, d), "w_down": mat(d, f, back)} for _ in range(c.n_layers)]
    embed = mat(c.vocab, d, 1.0)
    head = torch.zeros(c.vocab, d, device="cuda")
    nxt = None
    for weight in CANDIDATES:
        perm = torch.randperm(c.vocab, generator=g, device="cuda")
        head.index_add_(0, perm, embed.float(), alpha=0.02 * weight)      # token t's candidate is perm[t]
        nxt = perm if nxt is None else nxt
    glob = {"embed": embed, "lm_head": head.to(dt), "final_norm": one}
    model = trj.Model(c, layers, glob, max_batch=max_batch, max_seq=max_seq, max_rows=max_rows)
    return model, nxt.cpu().numpy()


def _prompt(r, n, vocab, nxt):
    """n tokens: noise with, in the middle, a copy of the continuation that has every third token or so wrong, as text
    that repeats itself gives prompt lookup good, partly good and bad drafts.  Returns (tokens, first new token)."""
    toks = np.array([r.randrange(vocab) for _ in range(n)], np.int32)
    at, t = n // 4, int(toks[-1])
    for i in range(at, at + n // 2):
        toks[i] = t if i < at + 3 or r.random() < 0.7 else r.randrange(vocab)
        t = int(nxt[t])
    return toks, int(nxt[int(toks[-1])])


def prepare(case, seed):
    r = random.Random(seed * 104729 + 5)
    kind = case["kind"]
    if kind == "ops":
        return _prepare_ops(case, seed, r)
    c = _cfg(case["model"])
    if kind == "step":
        rows = 1 + case["window"] + case["branches"] * case["branch_len"]
        model, nxt = _model(case["model"], seed, 1, case["prefix"] + rows + 64, max(rows, 32))
        toks, root = _prompt(r, case["prefix"], c.vocab, nxt)
        model.prefill(_i32(toks))
        return SimpleNamespace(kind=kind, case=case, model=model, context=np.append(toks, np.int32(root)), root=root,
                               window=np.array([r.randrange(c.vocab) for _ in range(case["window"])], np.int32),
                               draws=np.array([r.randrange(1 << 31) for _ in range(rows)], np.int64), length=model.seq_len.clone(),
                               rows=rows, max_len=case["prefix"] + rows,
                               k=model.k_cache[:, :, :, :case["prefix"] + rows], v=model.v_cache[:, :, :, :case["prefix"] + rows])
    if kind == "tree":
        lens, rows = _sizes(case)
        longest = max(s + m for s, m in zip(lens, rows))
        model, nxt = _model(case["model"], seed, case["batch"], longest + 8, max(rows + [32]))
        roots = []
        for b, s in enumerate(lens):
            toks, root = _prompt(r, s, c.vocab, nxt)
            model.prefill(_i32(toks), b)
            roots.append(root)
        trees = _trees(dict(case, vocab=c.vocab), lambda row, tok: int(nxt[tok]), roots, seed)
        wrote = [cache[:, b, :, s:s + m] for cache in (model.k_cache, model.v_cache) for b, (s, m) in enumerate(zip(lens, rows))]
        return SimpleNamespace(kind=kind, case=case, model=model, trees=trees, length=model.seq_len.clone(), rows=sum(rows),
                               max_rows=max(rows), max_len=longest, wrote=wrote)
    if kind == "prefill":
        model, nxt = _model(case["model"], seed, 1, case["tokens"] + 64, 128)
        toks, _ = _prompt(r, case["tokens"], c.vocab, nxt)
        n = case["tokens"]
        return SimpleNamespace(kind=kind, case=case, model=model, tokens=_i32(toks), k=model.k_cache[:, :, :, :n], v=model.v_cache[:, :, :, :n])
    assert kind == "generate", kind
    n, rows = case["tokens"], 1 + case["window"] + case["branches"] * case["branch_len"]
    most = n + 1 + case["steps"] * (max(case["window"], case["branch_len"]) + 1)
    model, nxt = _model(case["model"], seed, 1, most + rows, 128)
    toks, _ = _prompt(r, n, c.vocab, nxt)
    context = np.zeros(most, np.int32)
    context[:n] = toks
    return SimpleNamespace(kind=kind, case=case, model=model, tokens=_i32(toks), context=_i32(context), n_ctx=_i32([0]), n_ctx0=_i32([n + 1]),
                           window=_i32([0] * case["window"]), window0=_i32([r.randrange(c.vocab) for _ in range(case["window"])]),
                           draws=torch.tensor([[r.randrange(1 << 31) for _ in range(rows - 1)] for _ in range(case["steps"])], device="cuda"),
                           k_log=_i32([0] * case["steps"]))


def _prepare_ops(case, seed, r):
    lens, rows = _sizes(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    heads, d, total = 32, 128, sum(rows)
    longest = max(s + m for s, m in zip(lens, rows))

    def normal(*shape, dtype=torch.bfloat16):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)
    s = SimpleNamespace(kind="ops", case=case, q=normal(total, heads, d), seq_len=_i32(lens), max_rows=max(rows), max_len=longest,
                        k=normal(case["batch"], case["kv_heads"], longest, d), v=normal(case["batch"], case["kv_heads"], longest, d), logits=None)
    best = [0] * total
    if case["vocab"]:
        s.logits = normal(total, case["vocab"], dtype=torch.bfloat16 if case["logits"] == "bf16" else torch.float32)
        best = s.logits.float().argmax(1).tolist()
        s.accept_ws = torch.zeros(trj.argmax_accept_workspace(total, case["batch"]), dtype=torch.uint8, device="cuda")
    s.trees = _trees(case, lambda row, tok: best[row], [r.randrange(1000) for _ in rows], seed)
    s.attn_ws = torch.empty(trj.tree_attention_workspace(total, case["batch"], heads, d, longest), dtype=torch.uint8, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    if s.kind == "step":
        return _run_step(s)
    if s.kind == "tree":
        return _run_tree(s)
    if s.kind == "ops":
        t = s.trees
        out = trj.tree_attention(s.q, s.k, s.v, s.seq_len, t.row_off, t.anc, max_rows=s.max_rows, max_len=s.max_len, workspace=s.attn_ws)
        if s.logits is None:
            return out
        return out, trj.argmax_accept(s.logits, t.tokens, t.parent, t.depth, t.row_off, workspace=s.accept_ws)
    m = s.model
    m.seq_len.zero_()
    first = m.prefill(s.tokens)
    if s.kind == "prefill":
        return {"first": first, "k": s.k, "v": s.v, "length": m.seq_len}
    n = s.case["tokens"]
    s.context[n:n + 1].copy_(first)
    s.n_ctx.copy_(s.n_ctx0)
    s.window.copy_(s.window0)
    m.decode_device(s.context, s.n_ctx, n + 1, s.window, s.case["branches"], s.case["branch_len"], s.draws, s.case["steps"], s.k_log)
    return {"context": s.context, "accepted": s.k_log, "k": m.k_cache, "v": m.v_cache, "length": m.seq_len, "n_ctx": s.n_ctx, "window": s.window}


def _run_step(s):
    c, m = s.case, s.model
    m.seq_len.copy_(s.length)                                # back to the prompt's end, so that a pass can be repeated
    branches = trj.retrieve(s.context, c["branches"], c["branch_len"], s.draws[c["window"]:]) if c["branches"] else []
    got = m.step_host(s.root, s.window, branches, s.max_len)
    path = got["path"]
    context = np.concatenate([s.context, got["tokens"][path[1:]], [got["bonus"]]])
    window = trj.refill_window(got["parent"], got["node_argmax"], int(path[-1]), c["window"], context, s.draws[:c["window"]])
    return {"tokens": got["tokens"], "predicted": got["node_argmax"], "accepted": got["k_acc"], "bonus": got["bonus"], "best": int(path[-1]),
            "window": window, "k": s.k, "v": s.v, "length": m.seq_len}


def _run_tree(s):
    m, t = s.model, s.trees
    m.seq_len.copy_(s.length)
    got = m.verify_step(t.tokens, t.parent, t.depth, t.anc, t.row_off, max_rows=s.max_rows, max_len=s.max_len, want_logits=True)
    top = m.node_topk(s.rows, s.case["top_k"]) if s.case["top_k"] else None
    acc = m.accept(t.tokens, t.parent, t.depth, t.row_off, got["node_argmax"])
    m.compact_kv(acc["k_acc"], acc["path"], batch=s.case["batch"])
    return {"logits": got["logits"], "predicted": got["node_argmax"], "top": top, "accepted": acc, "wrote": s.wrote, "length": m.seq_len}


# ------------------------------------------------------------------------------------------------ cost and comparison
def _forward(model, lens, rows, head_rows, logits_out):
    """Bytes and operations of one forward: weights and cached K/V read, new K/V and logits written; row i of a tree sees
    the prefix and about half of the tree."""
    c = _cfg(model)
    es = 2 if c.dtype == "bf16" else 4
    hd, kv = c.n_heads * c.head_dim, c.n_kv_heads * c.head_dim
    layer = c.d_model * (hd + 2 * kv) + hd * c.d_model + 3 * c.d_model * c.d_ff
    head = c.vocab * c.d_model if head_rows else 0
    m = sum(rows)
    nbytes = es * (c.n_layers * layer + head + m * c.d_model) + 2 * es * c.n_layers * kv * sum(s + r for s, r in zip(lens, rows))
    nbytes += 4 * c.vocab * m if logits_out else 0
    flops = 2.0 * (m * c.n_layers * layer + head_rows * head) + 4.0 * c.n_layers * hd * sum(r * (s + r / 2) for s, r in zip(lens, rows))
    return float(nbytes), flops


def work(case):
    if case["kind"] == "ops":
        lens, rows = _sizes(case)
        keys = sum(s + m for s, m in zip(lens, rows))
        nbytes = 2 * 2 * case["kv_heads"] * 128 * keys + 2 * 2 * 32 * 128 * sum(rows)
        nbytes += sum(rows) * case["vocab"] * (2 if case["logits"] == "bf16" else 4)
        return {"bytes": nbytes, "flops": 4 * 32 * 128 * sum(m * (s + m / 2) for s, m in zip(lens, rows))}
    if case["kind"] == "tree":
        lens, rows = _sizes(case)
        b, f = _forward(case["model"], lens, rows, sum(rows), True)
    elif case["kind"] == "step":
        rows = 1 + case["window"] + case["branches"] * case["branch_len"]
        b, f = _forward(case["model"], [case["prefix"]], [rows], rows, False)
    else:
        b, f = _forward(case["model"], [0], [case["tokens"]], 1, False)
        if case["kind"] == "generate":
            rows = 1 + case["window"] + case["branches"] * case["branch_len"]
            for i in range(case["steps"]):
                sb, sf = _forward(case["model"], [case["tokens"] + 3 * i], [rows], rows, False)
                b, f = b + sb, f + sf
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["kind"] == "ops":
        # bf16 probabilities and outputs: 2.3e-3 and 0.015 against fp64 on all three listed shapes; ids and paths are exact
        return {"rel": 0.01, "max": 0.06}
    if MODELS[case["model"]]["dtype"] == "f32":
        return {"rel": 1e-5}                                 # fp32 sums of up to 688 products
    # Activations reach the projections as bf16 pairs, q and the cache are bf16.  Scoring the same rows in another split or
    # chunking: logits 5e-5, K/V 4.6e-4 with single elements one bf16 step (0.0078) apart; top-K ids may swap on near ties.
    return {"rel": 2e-3, "max": 0.03, "differ": 0.01}
