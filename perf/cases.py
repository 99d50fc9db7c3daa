"""The calls whose speed counts: what a program that decodes with this library has it do, over the sizes it meets.

Five kinds of pass, each through the public entry points of ``paper_2604_02047_b200.binding``:

``step``     one ``verify_step`` / ``verify_step_gqa``: attention of the tree, top-k, acceptance walk, compaction.
``cycle``    one ``verify_step_harvest``: what a decoding cycle calls, the step plus the update of the adjacency table.
``model``    a whole model's verification pass out of the four single calls: the tree attention of every layer, then the
             top-k of the logits, the walk, and the compaction of every layer's cache.
``prefill``  ``harvest`` of a prompt's logits rows into the adjacency table.
``host``     one ``verify_step_host``: inputs and results in pinned host memory.

Head counts, tree sizes, vocabularies and prefix lengths are those of the repository's workloads and tests (32, 40 and 52
heads, 32 query heads over 8 key/value heads; trees of 16 to 128 nodes; 32 000 and 128 256 vocabulary entries; prefixes
of 512 to 16 384 tokens), with odd sizes between them.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2604_02047_b200 import binding, synth

D = 128
SCALE = 1.0 / math.sqrt(D)


def case(op, S, H, Hkv, B, ctx, V, k, *, layers=1, counts=False, name=None):
    """``ctx`` = (lo, hi): every sequence's prefix length lies in that range.  ``counts``: the trees have fewer than B
    nodes (n_nodes is passed), and one sequence of the batch has left it.  ``prefill``: S * B rows of logits."""
    c = dict(op=op, S=S, H=H, Hkv=Hkv, B=B, ctx_lo=ctx[0], ctx_hi=ctx[1], V=V, k=k, layers=layers, counts=counts)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a short prompt and a small tree: a draft's first steps, where launches and latency are all there is
        case("step", 1, 32, 32, 16, (512, 512), 32000, 8, name="step_small"),
        # one layer's step of an interactive session, by model size
        case("step", 1, 32, 32, 80, (2048, 2048), 32000, 8, name="step_32h_2k"),
        case("step", 1, 40, 40, 80, (4096, 4096), 32000, 8, name="step_40h_4k"),
        case("step", 1, 52, 52, 128, (8192, 8192), 32000, 8, name="step_52h_8k"),
        # a serving batch of long, ragged prefixes: the largest pass
        case("step", 16, 32, 32, 64, (1024, 16384), 32000, 8, name="step_batch16"),
        # grouped-query heads and a large vocabulary, a small serving batch
        case("step", 4, 32, 8, 32, (4096, 16384), 128256, 8, name="step_gqa_batch4"),
        # the decoding cycle of one grouped-query session with a tree of 60 nodes and 10 candidates a node
        case("cycle", 1, 32, 8, 60, (3001, 3001), 128256, 10, name="cycle_gqa_60"),
        # the decoding cycle of a batch whose trees have different sizes and of which one sequence has finished
        case("cycle", 8, 32, 32, 60, (333, 6000), 32000, 10, counts=True, name="cycle_ragged8"),
        # a whole model's pass through the single calls, multi-head and grouped-query
        case("model", 1, 32, 32, 60, (1531, 1531), 32000, 10, layers=32, name="model_32h"),
        case("model", 2, 32, 8, 61, (1000, 5000), 128256, 10, layers=32, name="model_gqa"),
        # the table's update from a prompt
        case("prefill", 1, 1, 1, 1500, (0, 0), 32000, 10, name="prefill_1500"),
        # the end-to-end call on host buffers
        case("host", 1, 40, 40, 80, (4096, 4096), 32000, 8, name="host_40h_4k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MOST = {"bytes": 2.2e9, "flops": 1.4e11}   # of a drawn case: below the largest listed ones


def draw(rng):
    op = rng.choice(["step", "step", "step", "cycle", "cycle", "model", "model", "prefill", "host"])
    V = rng.choice([32000, 32000, 128256, 8 * _log(rng, 2000, 16000)])
    k = rng.choice([8, 8, 10, rng.randint(1, 16)])
    if op == "prefill":
        return case(op, 1, 1, 1, _log(rng, 40, 2000), (0, 0), V, k)
    H, Hkv = rng.choice([(32, 32), (40, 40), (52, 52), (32, 8), (32, 8), (16, 2)])
    if op == "host" and rng.random() < 0.5:
        H, Hkv = 32, 8
    B = rng.choice([16, 32, 60, 64, 80, 128, rng.randint(5, 128), rng.randint(5, 128)])
    layers = _log(rng, 4, 40) if op == "model" else 1
    S = rng.choice([1, 1, 1, 2, 4, _log(rng, 2, 16)]) if op != "host" else rng.choice([1, 1, 4])
    hi = _log(rng, 300, 16384)
    lo = hi if S == 1 or rng.random() < 0.3 else max(1, int(hi * rng.uniform(0.1, 0.9)))
    counts = S > 1 and op == "cycle" and rng.random() < 0.6
    c = case(op, S, H, Hkv, B, (lo, hi), V, k, layers=layers, counts=counts)
    while any(work(c)[x] > MOST[x] for x in MOST):
        if c["layers"] > 1:
            c["layers"] = c["layers"] * 3 // 4
        else:
            c["ctx_lo"], c["ctx_hi"] = c["ctx_lo"] * 3 // 4 + 1, c["ctx_hi"] * 3 // 4 + 1
    return c


# ------------------------------------------------------------------------------------------------ shapes of a case
def _shapes(c):
    """Prefix lengths and node counts of the case's sequences (part of the case, not of the seed)."""
    r = random.Random("%d %d %d %d" % (c["S"], c["B"], c["ctx_lo"], c["ctx_hi"]))
    ctx = [r.randint(c["ctx_lo"], c["ctx_hi"]) for _ in range(c["S"])]
    nodes = [c["B"]] * c["S"]
    if c["counts"]:
        nodes = [r.randint(max(1, c["B"] // 3), c["B"]) for _ in range(c["S"])]
        nodes[r.randrange(c["S"])] = 0
    return ctx, nodes


def work(c):
    rows, V = c["S"] * c["B"], c["V"]
    if c["op"] == "prefill":
        return {"bytes": rows * V * 2, "flops": 0}
    ctx, nodes = _shapes(c)
    live = [(x, n) for x, n in zip(ctx, nodes) if n]
    kv = sum(2 * (x + n) * c["Hkv"] * D * 2 for x, n in live)
    qo = sum(2 * n * c["H"] * D * 2 for _, n in live)
    flops = sum(4 * n * (x + n) * D * c["H"] for x, n in live)
    return {"bytes": c["layers"] * (kv + qo) + sum(nodes) * V * 2, "flops": c["layers"] * flops}


def tolerance(c):
    """Against the same attention in 64 bits the outputs are off by 2.1e-3 to 2.4e-3 (2-norm) and 7e-3 to 1.3e-2 (largest): P
    and the output are rounded to bf16.  Four times that is allowed.  The table's scores and the log-sum-exp are 32-bit
    sums (measured 7e-7).  Identifiers, lengths and moved cache rows are exact in every case."""
    if c["op"] == "prefill":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    return {"rel": 0.01, "max": 0.05, "differ": 0.0}


# ------------------------------------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=None)
def _context():
    """The process's context: every request of a program goes through the same one."""
    return binding.Goose(max_S=16, max_B=128, max_H=64)


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)


def _int32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


def _trees(c, rs):
    """Spine trees with distinct sibling tokens, and which nodes the model will agree with."""
    S, B, V = c["S"], c["B"], c["V"]
    parent, tok, agree = np.empty((S, B), np.int32), np.empty((S, B), np.int32), np.zeros((S, B), bool)
    for s in range(S):
        n_spine = int(rs.integers(min(4, B), min(24, B) + 1))
        parent[s], spine = synth.spine_tree(rs, B, n_spine, 3)
        tok[s] = synth.distinct_sibling_tokens(rs, parent[s], V)
        agree[s] = rs.random(B) < np.where(spine, rs.uniform(0.5, 0.95), 0.15)
        agree[s, 0] = False
    return parent, tok, agree


def prepare(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rs = np.random.default_rng(seed)
    S, H, Hkv, B, V, k, L = (c[x] for x in ("S", "H", "Hkv", "B", "V", "k", "layers"))
    st = dict(case=c, goose=_context(), k=k)
    if c["op"] == "prefill":
        st["logits"] = _normal(g, B, V)
        st["row_tok"] = _int32(rs.integers(0, V, B))
        st["adj_ids"] = torch.full((V, k), -1, dtype=torch.int32, device="cuda")
        st["adj_scores"] = torch.zeros((V, k), dtype=torch.float32, device="cuda")
        return st
    ctx, nodes = _shapes(c)
    parent, tok, agree = _trees(c, rs)
    used = np.array(ctx, np.int64) + B
    total = int(used.sum())
    st["row_off"] = torch.from_numpy(np.concatenate([[0], np.cumsum(used)[:-1]]).astype(np.int64)).cuda()
    st["ctx_len"], st["parent"], st["tok"] = _int32(np.array(ctx)), _int32(parent), _int32(tok)
    st["n_nodes"] = _int32(np.array(nodes)) if c["counts"] else None
    K, Vc, q = _normal(g, L, total, Hkv, D), _normal(g, L, total, Hkv, D), _normal(g, L, S, B, H, D)
    st["caches"] = [K, Vc]                         # of all layers; below, each layer's own
    st["layers"] = list(zip(q, K, Vc))
    logits = _normal(g, S * B, V)
    s_at, i_at = np.nonzero(agree)
    rows = torch.from_numpy(s_at * B + parent[s_at, i_at]).cuda()
    logits[rows, torch.from_numpy(tok[s_at, i_at].astype(np.int64)).cuda()] += 10.0
    st["logits"] = logits
    if c["op"] == "model":
        st["out"] = torch.zeros_like(q)
        st["layers"] = list(zip(q, K, Vc, st["out"]))
    elif c["op"] == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        at = torch.cat([torch.arange(B, device="cuda") + int(o) + x for o, x in zip(st["row_off"].tolist(), ctx)])
        st["h_in"] = dict(h_q=pin(q[0]), h_k_new=pin(K[0][at].view(S, B, Hkv, D)), h_v_new=pin(Vc[0][at].view(S, B, Hkv, D)),
                          h_row_off=pin(st["row_off"]), h_ctx_len=pin(st["ctx_len"]), h_parent=pin(st["parent"]),
                          h_draft_tok=pin(st["tok"]), h_logits=pin(logits))
        st["h_out"] = {n: torch.zeros(t.shape, dtype=t.dtype).pin_memory() for n, t in st["goose"].alloc_step_outputs(S, B, H, D, k).items()}
        del st["logits"]
    else:
        # rows of nodes that do not exist are not written: they keep what the program put there
        st["outs"] = {n: t.zero_() for n, t in st["goose"].alloc_step_outputs(S, B, H, D, k).items()}
        if c["op"] == "cycle":
            st["outs"]["row_lse"] = torch.zeros(S * B, dtype=torch.float32, device="cuda")
            st["adj_ids"] = torch.full((V, k), -1, dtype=torch.int32, device="cuda")
            st["adj_scores"] = torch.zeros((V, k), dtype=torch.float32, device="cuda")
    return st


# ------------------------------------------------------------------------------------------------ one pass
def run(st):
    c, g = st["case"], st["goose"]
    grouped = c["H"] != c["Hkv"]
    if c["op"] == "step":
        q, kc, vc = st["layers"][0]
        step = g.verify_step_gqa if grouped else g.verify_step
        step(q, kc, vc, st["row_off"], st["ctx_len"], st["parent"], st["tok"], st["logits"], st["k"], SCALE, outs=st["outs"],
             n_nodes=st["n_nodes"])
        return [st["outs"], st["caches"]]
    if c["op"] == "cycle":
        q, kc, vc = st["layers"][0]
        g.verify_step_harvest(q, kc, vc, st["row_off"], st["ctx_len"], st["parent"], st["tok"], st["logits"], st["k"], SCALE,
                              st["adj_ids"], st["adj_scores"], outs=st["outs"], n_nodes=st["n_nodes"])
        return [st["outs"], st["caches"], st["adj_ids"], st["adj_scores"]]
    if c["op"] == "model":
        attn = g.tree_attn_gqa if grouped else g.tree_attn
        for q, kc, vc, out in st["layers"]:
            attn(q, kc, vc, st["row_off"], st["ctx_len"], st["parent"], SCALE, out=out)
        argmax, ids, vals = g.node_topk(st["logits"], st["k"])
        path, accept_len, bonus = g.accept(st["tok"], st["parent"], argmax.view(c["S"], c["B"]))
        for q, kc, vc, out in st["layers"]:
            new_ctx = g.kv_compact(kc, vc, st["row_off"], st["ctx_len"], path, accept_len)
        return [st["out"], argmax, ids, vals, path, accept_len, bonus, new_ctx, st["caches"]]
    if c["op"] == "prefill":
        return [g.harvest(st["logits"], st["k"], st["row_tok"], st["adj_ids"], st["adj_scores"]), st["adj_ids"], st["adj_scores"]]
    q, kc, vc = st["layers"][0]
    call = g.verify_step_host_gqa if grouped else g.verify_step_host
    call(kc, vc, k=st["k"], scale=SCALE, h_outs=st["h_out"], **st["h_in"])
    return [st["h_out"], st["caches"]]


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _attention(q, K, V, row0, ctx, n, parent):
    """Nodes 0..n-1 of one sequence over its ctx prefix rows and, of its tree rows, a node's ancestors and itself."""
    sees = torch.zeros(n, n, dtype=torch.bool)
    for i in range(n):
        if i:
            sees[i] = sees[parent[i]]
        sees[i, i] = True
    sees = torch.cat([torch.ones(n, ctx, dtype=torch.bool), sees], 1).to(q.device)
    group = q.shape[1] // K.shape[1]
    out = torch.empty(n, q.shape[1], D, dtype=torch.float64, device=q.device)
    for hk in range(K.shape[1]):
        keys, values = (t[row0:row0 + ctx + n, hk].double() for t in (K, V))
        for h in range(hk * group, (hk + 1) * group):
            p = (SCALE * (q[:n, h].double() @ keys.T)).masked_fill_(~sees, -math.inf)
            out[:, h] = torch.softmax(p, 1) @ values
    return out


def exact(c, seed):
    """The attention's output, the k largest logits of each row, the rows' log-sum-exp and the table's scores."""
    st = prepare(c, seed)
    k, V = c["k"], c["V"]
    logits = (st["h_in"]["h_logits"].cuda() if c["op"] == "host" else st["logits"]).double()
    ids = torch.sort(logits, dim=1, descending=True, stable=True)[1][:, :k] if c["op"] in ("cycle", "prefill") else None
    top = torch.topk(logits, k, dim=1)[0]
    lse = torch.logsumexp(logits, 1)
    if c["op"] == "prefill":
        tokens, nodes = st["row_tok"].tolist(), [c["B"]]
    else:
        ctx, nodes = _shapes(c)
        tokens, parent, offsets = st["tok"].view(-1).tolist(), st["parent"].tolist(), st["row_off"].tolist()
        out = torch.zeros(c["layers"], c["S"], c["B"], c["H"], D, dtype=torch.float64, device="cuda")
        for layer in range(c["layers"]):
            q, K, Vc = st["layers"][layer][:3]
            for s, n in enumerate(nodes):
                if n:
                    out[layer, s, :n] = _attention(q[s], K, Vc, offsets[s], ctx[s], n, parent[s])
    if c["op"] == "model":
        return [out, None, None, top, None, None, None, None, None]
    live = torch.tensor([i < n for n in nodes for i in range(c["B"])], device="cuda")   # nothing is written of other rows
    top, lse = top * live[:, None], lse * live
    if c["op"] in ("step", "host"):
        return [dict(out=out[0], topk_vals=top), None]
    scores = torch.zeros(V, k, dtype=torch.float64, device="cuda")
    for row, token in enumerate(tokens):                       # of several rows with one token the last one stands
        if live[row] and 0 <= token < V:
            scores[token] = torch.exp(logits[row, ids[row]] - lse[row])
    if c["op"] == "prefill":
        return [[None, None, top, lse], None, scores]
    return [dict(out=out[0], topk_vals=top, row_lse=lse), None, None, scores]
