"""Workloads by which the speed of this framework is measured, with the ranges they stand for.

A case is a dict of plain values; ``kind`` says which public calls one pass makes:

``verify``      one verify step at temperature 0: clv_tree_attn, clv_accept_argmax,
                clv_accept_walk_commit (the sequence of ``step.VerifyStep.run``)
``sample``      one verify step at temperature 1: clv_tree_attn, clv_accept_sample, clv_kv_commit
``model``       the verify step of all layers of a model (the sequence of
                ``step.ModelVerifyStep.run``): the tree from its interval labels, clv_tree_attn per
                layer, clv_lm_head_argmax, clv_accept_walk, clv_kv_commit_layers
``host``        one verify step whose inputs and results are pinned host buffers
                (clv_verify_step_host)
``lm_head``     clv_lm_head_argmax alone: the greedy choice for a batch of final hidden states
``draft_head``  clv_draft_head_step: one head of the drafter for a few rows
``token_tree``  clv_build_token_tree: speculated sequences merged into draft trees

The sizes are those of the repository's workloads C1-C5 and of its benchmark, plus odd and ragged
ones.  Inputs are drawn on the GPU from the seed: Q, K, V ~ N(0, 1) as in ``workloads.generate``,
random trees with distinct siblings, and logits with one clear winner per node, which is a drafted
child's token for 60 % of the nodes, so that the walk accepts drafts as it does with a useful drafter.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2408_00264_b200 import binding as clv
from paper_2408_00264_b200 import workloads

D = workloads.HEAD_DIM
PAGE = workloads.PAGE_SIZE
HIDDEN = 4096

# the largest listed sizes: a drawn case stays below them
MAX_KV_ROWS = 8 * 8 * 32768          # batch x kv heads x context
MAX_SCORES = 8 * 32 * 128 * 32768    # batch x query heads x nodes x context
MAX_LOGITS = 1024 * 128256           # rows x vocabulary


def _verify(name, batch, nodes, hq, hkv, ctx_lo, ctx_hi, depth, vocab, paged=False, kind="verify", **more):
    return dict(name=name, kind=kind, batch=batch, nodes=nodes, hq=hq, hkv=hkv, ctx_lo=ctx_lo, ctx_hi=ctx_hi,
                depth=depth, vocab=vocab, paged=paged, **more)


def listed():
    return [
        # one user, short context, small tree, as many KV heads as query heads: latency and launches
        _verify("verify_mha_b1_short", 1, 16, 32, 32, 512, 512, 4, 32000),
        # one user in the middle of a conversation: the case the paper's evaluation is made of
        _verify("verify_mha_b1", 1, 64, 32, 32, 2048, 2048, 6, 32000),
        # a few users, grouped heads, large vocabulary: the benchmark's default workload
        _verify("verify_gqa_b4", 4, 64, 32, 8, 4096, 4096, 6, 128256),
        # batched serving: ragged contexts in a paged cache
        _verify("verify_paged_b32", 32, 32, 32, 8, 561, 8180, 5, 128256, paged=True),
        # long contexts and the largest tree: attention is a dense contraction
        _verify("verify_long_b8", 8, 128, 32, 8, 32768, 32768, 8, 128256),
        # sampling instead of greedy decoding; odd sizes everywhere (group of 7 heads, ragged contexts)
        _verify("sample_ragged_b5", 5, 27, 28, 4, 301, 3011, 5, 50257, kind="sample"),
        # one user, all layers of a model, the LM head fused with the greedy choice
        _verify("model_mha_b1", 1, 60, 32, 32, 1500, 1500, 6, 32000, kind="model", layers=32),
        # the same for a few users: the whole target side of a decode iteration
        _verify("model_gqa_b4", 4, 64, 32, 8, 4096, 4096, 6, 128256, kind="model", layers=32),
        # an engine that keeps activations on the host hands the step over in pinned buffers
        _verify("host_mha_b1", 1, 64, 32, 32, 2048, 2048, 6, 32000, kind="host"),
        # greedy choice for every node of a full batch of trees: compute bound
        dict(name="lm_head_1024", kind="lm_head", rows=1024, hidden=HIDDEN, vocab=128256),
        # one step of the drafter for four sequences: a stream over its weights
        dict(name="draft_head_b4", kind="draft_head", rows=4, hidden=HIDDEN, heads=32, vocab=128256, k_top=8),
        # draft trees of four sequences from 32 speculations each: the smallest call
        dict(name="token_tree_b4", kind="token_tree", batch=4, cand=32, length=6, nodes=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["verify", "verify", "verify", "sample", "model", "host", "lm_head", "draft_head", "token_tree"])
    if kind == "token_tree":
        return dict(kind=kind, batch=_log(rng, 1, 64), cand=rng.randint(2, 128), length=rng.randint(2, 12), nodes=128)
    if kind == "lm_head":
        vocab = _log(rng, 16000, 128256)
        return dict(kind=kind, rows=_log(rng, 1, 1024), hidden=64 * rng.randint(16, 64), vocab=vocab)
    if kind == "draft_head":
        return dict(kind=kind, rows=_log(rng, 1, 64), hidden=512 * rng.randint(2, 8), heads=rng.choice([16, 32]),
                    vocab=_log(rng, 16000, 128256), k_top=rng.randint(1, 16))
    hq, hkv = rng.choice([(32, 32), (32, 8), (32, 8), (28, 4), (40, 8), (64, 8), (16, 16), (24, 8)])
    nodes = rng.randint(4, 128)
    hi = _log(rng, 200, 32768)
    lo = hi if rng.random() < 0.4 else max(64, int(hi * rng.uniform(0.1, 0.9)))
    vocab = _log(rng, 16000, 128256)
    layers = rng.randint(4, 32) if kind == "model" else 1
    most = min(MAX_KV_ROWS // (hkv * hi * layers), MAX_SCORES // (hq * nodes * hi * layers), MAX_LOGITS // (nodes * vocab), 48)
    if kind == "host":   # the logits cross the host's link: a few users at most
        most = min(most, 4)
    while most < 1:      # too much for one sequence: a shorter context
        hi, lo = hi // 2, max(64, lo // 2)
        most = min(MAX_KV_ROWS // (hkv * hi * layers), MAX_SCORES // (hq * nodes * hi * layers))
    c = dict(kind=kind, batch=_log(rng, 1, most), nodes=nodes, hq=hq, hkv=hkv, ctx_lo=min(lo, hi), ctx_hi=hi,
             depth=rng.randint(3, 10), vocab=vocab, paged=kind != "host" and rng.random() < 0.5)
    if kind == "model":
        c["layers"] = layers
    return c


# ------------------------------------------------------------------------------------- inputs
def _contexts(case):
    """Context lengths of a batch, evenly spread over the case's range (their order is seeded)."""
    return np.linspace(case["ctx_lo"], case["ctx_hi"], case["batch"]).astype(np.int32)


def _trees(case, rng):
    """Draft trees, their tokens (distinct among siblings) and the target's choice per node."""
    B, N, V = case["batch"], case["nodes"], case["vocab"]
    parent, tokens, winner = (np.empty((B, N), dtype=np.int32) for _ in range(3))
    for b in range(B):
        parent[b] = workloads.tree_random(N, case["depth"], rng)
        tokens[b] = rng.permutation(V)[:N] if V < 4 * N else rng.choice(V, size=N, replace=False, shuffle=False)
        kids = [[] for _ in range(N)]
        for i in range(1, N):
            kids[parent[b, i]].append(i)
        for i in range(N):
            if kids[i] and rng.random() < 0.6:
                winner[b, i] = tokens[b, kids[i][rng.integers(0, len(kids[i]))]]
            else:
                winner[b, i] = rng.integers(0, V)
    return parent, tokens, winner


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _normal(gen, *shape):
    return torch.randn(*shape, dtype=torch.bfloat16, device="cuda", generator=gen)


def _peaked_logits(gen, rows, vocab, winner, std, lift):
    """bf16 logits N(0, std^2), the winner of each row raised to the row's maximum + lift."""
    ld = (vocab + 7) // 8 * 8
    lg = _normal(gen, rows, ld).mul_(std)
    at = _dev(winner.reshape(-1).astype(np.int64)).unsqueeze(1)
    lg.scatter_(1, at, lg[:, :vocab].amax(1, keepdim=True) + lift)
    return lg, ld


def _lm_head_inputs(gen, rows, hidden, vocab, winner):
    """Vocabulary matrix N(0, 1/hidden) and hidden states whose winner's logit leads by about 12."""
    weight = _normal(gen, vocab, hidden).mul_(hidden ** -0.5)
    at = _dev(winner.reshape(-1).astype(np.int64))
    return _normal(gen, rows, hidden) + 12.0 * weight[at], weight


def _prepare_attention(case, rng, gen):
    B, N, hq, hkv = case["batch"], case["nodes"], case["hq"], case["hkv"]
    layers = case.get("layers", 1)
    s = SimpleNamespace(kind=case["kind"], layers=layers)
    ctx = rng.permutation(_contexts(case)).astype(np.int32)
    parent, tokens, winner = _trees(case, rng)
    path_cap = case["depth"] + 1
    s.q, s.k_tree, s.v_tree = _normal(gen, layers, B, N, hq, D), _normal(gen, layers, B, N, hkv, D), _normal(gen, layers, B, N, hkv, D)
    s.block_table = None
    if case["paged"]:
        need = [(int(n) + N + PAGE - 1) // PAGE for n in ctx]
        pages = sum(need) + (sum(need) + 7) // 8
        table, order, at = np.full((B, max(need)), -1, dtype=np.int32), rng.permutation(pages), 0
        for b, n in enumerate(need):
            table[b, :n] = order[at:at + n]
            at += n
        s.block_table = _dev(table)
        rows = (pages, PAGE)
    else:
        rows = (B, int(ctx.max()) + N)
    s.k_cache, s.v_cache = _normal(gen, layers, *rows, hkv, D), _normal(gen, layers, *rows, hkv, D)
    s.parent, s.tokens, s.ctx_len = _dev(parent), _dev(tokens), _dev(ctx)
    s.max_ctx, s.scale, s.winner, s.path_cap = int(ctx.max()), D ** -0.5, winner, path_cap
    s.shape = clv.make_shape(B, N, hq, hkv, case["vocab"], path_cap)
    s.caches = [clv.make_cache(s.k_cache[l], s.v_cache[l], s.block_table) for l in range(layers)]
    s.workspace = clv.new_workspace(s.shape, s.caches[0], s.max_ctx)
    i32 = dict(dtype=torch.int32, device="cuda")
    s.out = torch.empty_like(s.q)
    s.ids, s.accept_len, s.accept_idx = torch.empty(B, N, **i32), torch.empty(B, **i32), torch.empty(B, path_cap, **i32)
    s.next_token, s.ctx_out, s.status = torch.empty(B, **i32), torch.empty(B, **i32), torch.zeros(4 + layers, B, **i32)
    s.statuses = list(s.status[:3])
    return s


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    i32 = dict(dtype=torch.int32, device="cuda")

    if kind == "token_tree":
        B, C, L, N = case["batch"], case["cand"], case["length"], case["nodes"]
        root, cand, lens = workloads.make_candidates(B, C, L, 6, seed=seed)
        # a tree that outgrew its slots would be refused: shorten until the prefixes fit
        for b in range(B):
            while len({tuple(cand[b, c, :d]) for c in range(C) for d in range(1, lens[b, c] + 1)}) >= N:
                lens[b] = np.minimum(lens[b], lens[b].max() - 1)
        return SimpleNamespace(kind=kind, ins=tuple(_dev(a) for a in (root, cand, lens)),
                               outs=tuple(torch.zeros(n, **i32) for n in ((B, N), (B, N), (B,), (B, C, L), (B,))))

    if kind == "lm_head":
        rows, vocab = case["rows"], case["vocab"]
        hidden, weight = _lm_head_inputs(gen, rows, case["hidden"], vocab, rng.integers(0, vocab, rows))
        return SimpleNamespace(kind=kind, hidden=hidden, weight=weight, ids=torch.zeros(rows, **i32),
                               status=torch.zeros(1, **i32),
                               workspace=clv.new_workspace(clv.make_shape(1, 1, 1, 1, vocab=8), None, 0))

    if kind == "draft_head":
        return _prepare_draft_head(case, rng, gen)

    s = _prepare_attention(case, rng, gen)
    B, N, V = case["batch"], case["nodes"], case["vocab"]
    if kind == "model":
        s.hidden, s.weight = _lm_head_inputs(gen, B * N, HIDDEN, V, s.winner)
        s.tin, s.tout = torch.empty_like(s.parent), torch.empty_like(s.parent)
        clv.clv_tree_to_intervals(s.parent, s.tin, s.tout, s.status[0])
        # a model holds its layers' tensors one by one
        s.per_layer = list(zip(s.caches, s.q, s.k_tree, s.v_tree, s.out, s.status[4:]))
        s.tree_status, s.head_status, s.walk_status, s.commit_status = s.status[:4]
        s.flat_ids, s.cache_stride, s.tree_stride = s.ids.view(-1), s.k_cache[0].numel(), s.k_tree[0].numel()
    else:
        # temperature 1: logits as wide as a language model's, so that a few tokens hold the mass
        std, lift = (3.0, 3.0) if kind == "sample" else (1.0, 0.5)
        s.logits, s.ld = _peaked_logits(gen, B * N, V, s.winner, std, lift)
        s.lse = torch.empty(B, N, case["hq"], dtype=torch.float32, device="cuda")
    if kind == "sample":
        s.uniforms = _dev(workloads.make_uniforms(B, N, seed=seed))
    if kind == "host":
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
        s.host_in = [pin(t) for t in (s.q, s.k_tree, s.v_tree, s.parent, s.tokens, s.logits)]
        s.host_out = [torch.zeros(t.shape, dtype=t.dtype).pin_memory()
                      for t in (s.out, s.ids, s.accept_len, s.accept_idx, s.next_token, s.status[:3])]
        s.inputs = clv.ClvHostInputs(*[t.data_ptr() for t in s.host_in], s.ld)
        s.outputs = clv.ClvHostOutputs(*[t.data_ptr() for t in s.host_out])
        s.staging = torch.empty(clv.clv_staging_bytes(s.shape, s.ld), dtype=torch.uint8, device="cuda")
        s.ctx_start = s.ctx_len.clone()
        del s.q, s.k_tree, s.v_tree, s.logits, s.out, s.lse
    return s


def _prepare_draft_head(case, rng, gen):
    rows, H, V, k = case["rows"], case["hidden"], case["vocab"], case["k_top"]
    inv = H ** -0.5
    w = {"n_heads": case["heads"],
         "norm1": 1.0 + 0.1 * _normal(gen, H), "norm2": 1.0 + 0.1 * _normal(gen, H),
         "wq": _normal(gen, H, H) * inv, "wk": _normal(gen, H, H) * inv, "wv": _normal(gen, H, H) * inv,
         "bq": 0.1 * _normal(gen, H), "bk": 0.1 * _normal(gen, H), "bv": 0.1 * _normal(gen, H),
         "wfc": _normal(gen, H, 2 * H) * (inv * 0.5 ** 0.5), "bfc": 0.1 * _normal(gen, H),
         "lm_head": _normal(gen, V, H).mul_(inv)}
    h, e = _normal(gen, rows, H), _normal(gen, rows, H)
    # A trained head's proposals stand out: k rows of the vocabulary point along each row's final
    # state with graded lengths (logits about 15.5, 15, 14.5, ... where the others reach about 4.5).
    f = {n: t.float() for n, t in w.items() if torch.is_tensor(t) and n != "lm_head"}
    norm = lambda x, g: x * torch.rsqrt(x.square().mean(1, keepdim=True) + 1e-5) * g  # noqa: E731
    ef = e.float()
    q = norm(h.float(), f["norm1"]) @ f["wq"].T + f["bq"]
    key, v = ef @ f["wk"].T + f["bk"], ef @ f["wv"].T + f["bv"]
    heads = (rows, case["heads"], H // case["heads"])
    gate = torch.nn.functional.cosine_similarity(q.view(heads), key.view(heads), dim=2, eps=1e-8).unsqueeze(2)
    a = (h.float().view(heads) + v.view(heads) * gate).view(rows, H)
    u = norm(torch.cat([a, ef], 1) @ f["wfc"].T + f["bfc"], f["norm2"])
    ids = _dev(rng.choice(V, size=(rows, k), replace=False))
    goal = 15.5 - 0.5 * torch.arange(k, device="cuda", dtype=torch.float32)
    plant = (u / u.square().sum(1, keepdim=True)).unsqueeze(1) * goal.view(1, k, 1)
    w["lm_head"][ids.view(-1)] = plant.view(rows * k, H).to(torch.bfloat16)
    i32 = dict(dtype=torch.int32, device="cuda")
    return SimpleNamespace(kind="draft_head", weights=w, head=clv.make_draft_head(w), h=h, e=e, k_top=k,
                           hidden_out=torch.empty_like(h), ids=torch.zeros(rows, k, **i32),
                           top=torch.zeros(rows, k, dtype=torch.float32, device="cuda"), status=torch.zeros(5, **i32),
                           workspace=clv.new_draft_head_workspace(rows, H, V))


# ------------------------------------------------------------------------------------- one pass
def run(s):
    if s.kind == "token_tree":
        clv.clv_build_token_tree(*s.ins, *s.outs)
        return s.outs
    if s.kind == "lm_head":
        clv.clv_lm_head_argmax(s.hidden, s.weight, s.ids, s.status, s.workspace)
        return s.ids, s.status
    if s.kind == "draft_head":
        clv.clv_draft_head_step(s.head, s.h, s.e, s.k_top, s.hidden_out, s.ids, s.top, s.status, s.workspace)
        return s.hidden_out, s.ids, s.top, s.status
    cache = s.caches[0]
    if s.kind == "host":
        s.ctx_len.copy_(s.ctx_start)   # the call advances ctx_len in place: back to the pass's own contexts
        clv.clv_verify_step_host(s.shape, cache, s.inputs, s.outputs, s.ctx_len, s.max_ctx, s.scale, s.staging, s.workspace)
        return s.host_out, s.ctx_len, s.k_cache, s.v_cache
    path = (s.accept_len, s.accept_idx, s.next_token)
    if s.kind == "model":
        clv.clv_tree_from_intervals(s.tin, s.tout, s.parent, s.tree_status)
        for layer_cache, q, k_tree, v_tree, out, status in s.per_layer:
            clv.clv_tree_attn(s.shape, layer_cache, q, k_tree, v_tree, s.parent, s.ctx_len, s.max_ctx, s.scale, out, None,
                              status, s.workspace)
        clv.clv_lm_head_argmax(s.hidden, s.weight, s.flat_ids, s.head_status, s.workspace)
        clv.clv_accept_walk(s.shape, s.parent, s.tokens, s.ids, *path, s.walk_status)
        clv.clv_kv_commit_layers(s.shape, cache, s.layers, s.cache_stride, s.k_tree, s.v_tree, s.tree_stride, s.accept_idx,
                                 s.accept_len, s.ctx_len, s.ctx_out, s.commit_status)
        return s.out, s.ids, path, s.ctx_out, s.status, s.parent, s.k_cache, s.v_cache
    attn_status, accept_status, commit_status = s.statuses
    clv.clv_tree_attn(s.shape, cache, s.q, s.k_tree, s.v_tree, s.parent, s.ctx_len, s.max_ctx, s.scale, s.out, s.lse,
                      attn_status, s.workspace)
    if s.kind == "sample":
        clv.clv_accept_sample(s.shape, s.logits, s.ld, s.parent, s.tokens, s.uniforms, 1.0, *path, accept_status, s.workspace)
        clv.clv_kv_commit(s.shape, cache, s.k_tree, s.v_tree, s.accept_idx, s.accept_len, s.ctx_len, s.ctx_out, commit_status)
        return s.out, s.lse, path, s.ctx_out, s.status, s.k_cache, s.v_cache
    clv.clv_accept_argmax(s.shape, s.logits, s.ld, s.ids, s.workspace)
    clv.clv_accept_walk_commit(s.shape, cache, s.parent, s.tokens, s.ids, s.k_tree, s.v_tree, s.ctx_len, *path, s.ctx_out,
                               accept_status, commit_status)
    return s.out, s.lse, s.ids, path, s.ctx_out, s.status, s.k_cache, s.v_cache


# ------------------------------------------------------------------------------------- what a pass needs
def work(case):
    kind = case["kind"]
    if kind == "token_tree":
        words = case["batch"] * (2 * case["cand"] * case["length"] + case["cand"] + 2 * case["nodes"] + 3)
        return {"bytes": 4 * words, "flops": 0}
    if kind == "lm_head":
        R, H, V = case["rows"], case["hidden"], case["vocab"]
        return {"bytes": 2 * (V + R) * H + 4 * R, "flops": 2 * R * H * V}
    if kind == "draft_head":
        R, H, V = case["rows"], case["hidden"], case["vocab"]
        weights = 5 * H * H + V * H
        return {"bytes": 2 * weights + 2 * 3 * R * H + 2 * 6 * H + 8 * R * case["k_top"], "flops": 2 * R * weights}
    B, N, hq, hkv, V = case["batch"], case["nodes"], case["hq"], case["hkv"], case["vocab"]
    layers, keys = case.get("layers", 1), int(_contexts(case).sum())
    attn = 2 * D * (2 * hkv * (keys + B * N) + 2 * hq * B * N)   # cached and tree K/V, Q and output
    flops = 4 * D * hq * N * (keys + B * N)
    if kind == "model":
        return {"bytes": layers * attn + 2 * (V + B * N) * HIDDEN, "flops": layers * flops + 2 * B * N * HIDDEN * V}
    return {"bytes": attn + 2 * B * N * V, "flops": flops}


def tolerance(case):
    if case["kind"] in ("token_tree", "lm_head"):   # whole numbers; the winners are clear
        return "exact"
    # bf16 products and results; ids, paths and cache rows are exact
    return {"rel": 1e-2, "max": 0.1}
