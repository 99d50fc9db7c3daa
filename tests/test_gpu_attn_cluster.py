"""GPU parity of the attention kernel's cluster form (one sequence, a thread-block cluster per head): every row against the
oracle with the usual bars, over fewer tiles than CTAs of a cluster, as many, one more, tiles cut at the edges of the tree,
trees of all sizes, grouped heads, node counts, an invalid tree; and the whole step, whose top-k runs beside it."""
import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth
from test_gpu_chained_steps import _run_chain
from test_gpu_parity import ATTN_TOL, LSE_TOL, attn_row_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goose():
    from paper_2604_02047_b200 import binding, build
    build.build()
    g = binding.Goose(max_S=2, max_B=128, max_H=64)
    yield g
    g.close()


def _inputs(rng, H, Hkv, B, ctx, q_gain=1.0, **kw):
    tree = synth.spine_tree(rng, B, max(1, B // 4), 3)[0] if B > 1 else synth.chain_tree(1)
    return synth.make_inputs(1, H, B, [ctx], [tree], Hkv=Hkv, seed=int(rng.integers(1 << 30)), q_gain=q_gain, **kw)


def _attn(goose, x, n_nodes=None, parent=None):
    from paper_2604_02047_b200 import binding
    d = binding.to_device(x)
    nn = None if n_nodes is None else torch.tensor([n_nodes], dtype=torch.int32, device="cuda")
    out = torch.full_like(d["q"], 7.0)
    lse = torch.full(d["q"].shape[:3], 7.0, device="cuda")
    par = d["parent"] if parent is None else torch.from_numpy(parent).cuda()
    before = goose.launch_count()
    goose.tree_attn_gqa(d["q"], d["k_cache"], d["v_cache"], d["row_off"], d["ctx_len"], par, x.scale, out=out, lse=lse, n_nodes=nn)
    torch.cuda.synchronize()
    assert goose.launch_count() == before + 1, "these sizes are meant for the cluster form (no merge kernel)"
    return out.float().cpu().numpy().astype(np.float64), lse.cpu().numpy(), int(goose.last_status(1)[0])


# heads of the work list: 32 (clusters of 4) and 40 (clusters of 3); grouped, with one M tile to eight: 20 or 40, 8 to 32, 2 to 16
@pytest.mark.parametrize("H,Hkv", [(32, 32), (40, 40), (40, 20), (32, 8), (16, 2)])
@pytest.mark.parametrize("ctx,B", [(0, 1), (0, 128), (1, 16), (112, 16), (113, 16), (127, 1), (128, 60), (300, 64), (383, 33),
                                   (449, 60), (512, 80), (900, 128)])
def test_cluster_shapes(goose, oracle, H, Hkv, ctx, B):
    rng = np.random.default_rng([H, Hkv, ctx, B])
    x = _inputs(rng, H, Hkv, B, ctx, q_gain=float(rng.choice([1.0, 6.0])), V=8, with_logits=False)
    ref, ref_lse = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)
    out, lse, status = _attn(goose, x)
    assert status == 0 and attn_row_err(out, ref).max() <= ATTN_TOL and np.abs(lse - ref_lse).max() <= LSE_TOL
    again, lse2, _ = _attn(goose, x)
    assert np.array_equal(out, again) and np.array_equal(lse, lse2)


@pytest.mark.parametrize("n", [0, 1, 17, 59])
def test_cluster_node_counts(goose, oracle, n):
    rng = np.random.default_rng(n)
    x = _inputs(rng, 32, 32, 60, 400, V=8, with_logits=False)
    ref, ref_lse = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)
    out, lse, status = _attn(goose, x, n_nodes=n)
    assert status == 0 and np.all(out[:, n:] == 7.0) and np.all(lse[:, n:] == 7.0)
    if n:                                                      # a node sees the prefix and its ancestors: rows < n stand
        assert attn_row_err(out[:, :n], ref[:, :n]).max() <= ATTN_TOL and np.abs(lse[:, :n] - ref_lse[:, :n]).max() <= LSE_TOL


@pytest.mark.parametrize("ctx", [20, 700])
def test_cluster_invalid_tree(goose, ctx):
    rng = np.random.default_rng(ctx)
    x = _inputs(rng, 40, 40, 20, ctx, V=8, with_logits=False)
    parent = x.parent.copy()
    parent[0, 7] = 9
    out, _, status = _attn(goose, x, parent=parent)
    assert status == 1 and np.all(out == 0.0)


@pytest.mark.parametrize("H,Hkv,B,V", [(32, 32, 16, 32000), (32, 32, 80, 32000), (32, 32, 128, 32000), (32, 32, 60, 70000),
                                       (52, 52, 60, 32000), (32, 8, 60, 70000), (16, 2, 100, 32000)])
def test_step_with_clusters(goose, oracle, H, Hkv, B, V):
    """Rows that fit beside the clusters (all, or several a CTA) and rows that do not: integers exact, caches exact."""
    from paper_2604_02047_b200 import binding
    rng = np.random.default_rng([B, V])
    x = _inputs(rng, H, Hkv, B, 600, V=V, k=8)
    d = binding.to_device(x)
    got = goose.verify_step_gqa(d["q"], d["k_cache"], d["v_cache"], d["row_off"], d["ctx_len"], d["parent"], d["draft_tok"],
                                d["logits"], 8, x.scale)
    torch.cuda.synchronize()
    am, ids, vals = oracle.node_topk(x.logits, 8)
    path, alen, bonus = oracle.accept(x.draft_tok, x.parent, am.reshape(1, B))
    assert np.array_equal(got["argmax"].cpu().numpy(), am) and np.array_equal(got["topk_ids"].cpu().numpy(), ids)
    assert np.array_equal(got["path"].cpu().numpy(), path) and got["accept_len"].tolist() == alen.tolist()
    assert got["bonus"].tolist() == bonus.tolist() and got["new_ctx_len"].tolist() == [600 + 1 + int(alen[0])]
    ref, _ = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)
    assert attn_row_err(got["out"].float().cpu().numpy().astype(np.float64), ref).max() <= ATTN_TOL
    r0 = int(x.row_off[0]) + 600
    for cache, before in ((d["k_cache"], x.k_cache), (d["v_cache"], x.v_cache)):
        rows = binding.bf16_to_bits(cache)
        for j in range(int(alen[0]) + 1):
            assert np.array_equal(rows[r0 + j], before[r0 + int(path[0, j])])
    assert int(goose.last_status(1)[0]) == 0


@pytest.mark.parametrize("H,B", [(32, 16), (40, 24)])
def test_steps_back_to_back(goose, oracle, H, B):
    """Three steps of one sequence without synchronisation in between, chains accepted whole and random trees: the top-k
    beside the clusters writes its results before it waits for the attention."""
    _run_chain(goose, oracle, 1, H, B, 4096, 4, [500], lambda t, s: synth.chain_tree(B), seed=70, full_accept=True, prewrite=True)
    rng = np.random.default_rng(H)
    _run_chain(goose, oracle, 1, H, B, 32000, 8, [300], lambda t, s: synth.spine_tree(rng, B, 8, 3)[0], seed=80, full_accept=False,
               prewrite=False)


@pytest.mark.parametrize("H,Hkv,B,ctx,V", [(32, 32, 80, 600, 32000), (40, 40, 80, 900, 32000), (52, 52, 60, 300, 32000), (32, 8, 60, 900, 70000)])
def test_cycles_back_to_back(goose, oracle, H, Hkv, B, ctx, V):
    """Four steps with harvest into one table, on clusters that take 64 to 86 % of the SMs: each against the oracle when waited
    for, and the same four enqueued at once leave the same bits everywhere."""
    from paper_2604_02047_b200 import binding
    rng = np.random.default_rng([H, Hkv, B])
    xs = [_inputs(rng, H, Hkv, B, ctx, V=V, k=8) for _ in range(4)]

    def run(wait):
        ids, scores = torch.full((V, 8), -1, dtype=torch.int32, device="cuda"), torch.zeros((V, 8), device="cuda")
        ds = [binding.to_device(x) for x in xs]
        outs = [goose.alloc_step_outputs(1, B, H, 128, 8) for _ in xs]
        torch.cuda.synchronize()
        for d, o in zip(ds, outs):
            goose.verify_step_harvest(d["q"], d["k_cache"], d["v_cache"], d["row_off"], d["ctx_len"], d["parent"], d["draft_tok"],
                                      d["logits"], 8, xs[0].scale, ids, scores, outs=o)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return outs, [d[n] for d in ds for n in ("k_cache", "v_cache")] + [ids, scores]

    outs, kept = run(True)
    for x, o in zip(xs, outs):
        am, top, _ = oracle.node_topk(x.logits, 8)
        path, alen, bonus = oracle.accept(x.draft_tok, x.parent, am.reshape(1, B))
        assert np.array_equal(o["topk_ids"].cpu().numpy(), top) and np.array_equal(o["path"].cpu().numpy(), path)
        assert o["accept_len"].tolist() == alen.tolist() and o["bonus"].tolist() == bonus.tolist()
        ref, _ = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)
        assert attn_row_err(o["out"].float().cpu().numpy().astype(np.float64), ref).max() <= ATTN_TOL
    for _ in range(3):
        again, kept2 = run(False)
        for o, p in zip(outs, again):
            assert all(torch.equal(o[n], p[n]) for n in ("out", "argmax", "topk_ids", "topk_vals", "path", "accept_len", "bonus", "new_ctx_len", "row_lse"))
        assert all(torch.equal(a, b) for a, b in zip(kept, kept2))
    assert int(goose.last_status(1)[0]) == 0
