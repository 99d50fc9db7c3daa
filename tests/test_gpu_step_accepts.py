"""Steps of one sequence at the sizes of which tests/test_step_split_host.py says what is chosen: smaller clusters than the largest, the
largest, the persistent form.  Each accepts nodes and moves cache rows.  The step equals the single calls: the attention within two bf16
results of one fp32 value (each within 2^-8 of the row's largest, by its own rounding and that of P), scores and log-sum-exp within
two 32-bit sums that are each within 1e-5 of the exact one, everything else exactly, the moved cache rows included."""
import math

import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H, Hkv, B, ctx, V, harvest", [
    (32, 8, 60, 1000, 128256, True), (32, 8, 60, 3001, 128256, True), (32, 8, 60, 1000, 128256, False), (16, 2, 128, 3001, 128256, True),
    (16, 16, 60, 829, 33000, True), (32, 32, 64, 2118, 33000, True), (32, 32, 128, 340, 32000, True),                        # smaller
    (32, 8, 60, 6000, 128256, True), (32, 8, 60, 3001, 128256, False), (32, 8, 80, 3001, 32000, True), (16, 2, 80, 766, 50000, False),
    (32, 32, 80, 2048, 32000, True), (32, 8, 60, 2859, 65536, False),                                                       # the largest
    (32, 32, 128, 1000, 128256, True), (40, 40, 80, 4096, 32000, False), (32, 8, 128, 2730, 32000, True),                    # persistent
    (32, 32, 128, 2048, 32000, False), (16, 2, 100, 500, 65536, True), (16, 2, 100, 500, 65536, False), (8, 8, 32, 300, 200000, False),
    (8, 8, 33, 1207, 65536, False)])                                                                                        # one item
def test_step_that_accepts_nodes_equals_the_single_calls(H, Hkv, B, ctx, V, harvest):
    from paper_2604_02047_b200 import binding
    g = binding.Goose(max_S=1, max_B=128, max_H=64)
    gen = torch.Generator(device="cuda").manual_seed(B)
    rs = np.random.default_rng(B)
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    q, kc, vc, logits = normal(1, B, H, 128), normal(ctx + B, Hkv, 128), normal(ctx + B, Hkv, 128), normal(B, V)
    parent = synth.spine_tree(rs, B, 8, 3)[0][None]
    tok = synth.distinct_sibling_tokens(rs, parent[0], V)[None]
    path = []                                                 # nodes that the walk accepts: the youngest child of the one before, three times
    for _ in range(3):
        path.append(int(np.nonzero(parent[0] == (path[-1] if path else 0))[0][-1]))
        if not (parent[0] == path[-1]).any():
            break
    for node in path:
        logits[int(parent[0, node]), int(tok[0, node])] = 30.0
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()
    parent, tok, ctx_len, row_off = i32(parent), i32(tok), i32([ctx]), torch.zeros(1, dtype=torch.int64, device="cuda")
    k, scale = 8, 1 / math.sqrt(128)

    out = g.tree_attn_gqa(q, kc, vc, row_off, ctx_len, parent, scale)[0]
    argmax, ids, vals = g.node_topk(logits, k)
    table = lambda: (torch.full((V, k), -1, dtype=torch.int32, device="cuda"), torch.zeros(V, k, device="cuda"))
    want_table = table()
    want_lse = g.harvest(logits, k, tok.view(-1), *want_table)[3]
    want_path, accepted, bonus = g.accept(tok, parent, argmax.view(1, B))
    want_k, want_v = kc.clone(), vc.clone()
    new_ctx = g.kv_compact(want_k, want_v, row_off, ctx_len, want_path, accepted)
    torch.cuda.synchronize()
    assert accepted.tolist() == [len(path)] and want_path[0, 1:len(path) + 1].tolist() == path
    assert not torch.equal(want_k, kc)                        # rows do move
    for _ in range(2):
        kc2, vc2, got_table = kc.clone(), vc.clone(), table()
        if harvest:
            o = g.verify_step_harvest(q, kc2, vc2, row_off, ctx_len, parent, tok, logits, k, scale, *got_table)
        else:
            o = g.verify_step_gqa(q, kc2, vc2, row_off, ctx_len, parent, tok, logits, k, scale)
        torch.cuda.synchronize()
        assert not g.last_status(1).any()
        diff = (o["out"].float() - out.float()).abs().amax(-1)
        assert (diff <= 2 * 2.0 ** -8 * out.float().abs().amax(-1)).all()
        assert torch.equal(o["argmax"], argmax) and torch.equal(o["topk_ids"], ids) and torch.equal(o["topk_vals"], vals)
        assert torch.equal(torch.sort(logits.float(), dim=1, descending=True, stable=True)[1][:, :k].int(), ids)
        assert torch.equal(o["path"], want_path) and torch.equal(o["accept_len"], accepted) and torch.equal(o["bonus"], bonus)
        assert torch.equal(o["new_ctx_len"], new_ctx) and torch.equal(kc2, want_k) and torch.equal(vc2, want_v)
        if harvest:
            assert torch.equal(got_table[0], want_table[0]) and torch.allclose(got_table[1], want_table[1], rtol=2e-5, atol=0)
            assert torch.allclose(o["row_lse"], want_lse, rtol=0, atol=2e-5)
    g.close()
