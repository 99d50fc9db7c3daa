"""Steps of one sequence whose top-k is long: the cluster's size is weighed against the SMs that the top-k gets, and a CTA of the top-k gets
whole rows where one item more allows it.  At sizes that fall on either side of both choices the step equals the single calls: the
attention within two bf16 results of one fp32 value (each within 2^-8 of the row's largest, by its own rounding and that of P), scores
within two 32-bit sums that are each within 1e-5 of the exact one, everything else exactly."""
import math

import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("harvest", [True, False])
@pytest.mark.parametrize("H, Hkv, B, ctx, V", [(32, 8, 60, 1000, 128256), (32, 8, 60, 3001, 128256), (32, 8, 60, 6000, 128256),
                                               (32, 8, 80, 3001, 32000), (16, 2, 128, 2500, 128256), (32, 32, 128, 2048, 32000),
                                               (16, 2, 100, 500, 65536), (8, 8, 32, 300, 200000)])
def test_step_equals_the_single_calls(H, Hkv, B, ctx, V, harvest):
    from paper_2604_02047_b200 import binding
    g = binding.Goose(max_S=1, max_B=128, max_H=64)
    gen = torch.Generator(device="cuda").manual_seed(B)
    rs = np.random.default_rng(B)
    normal = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    q, kc, vc, logits = normal(1, B, H, 128), normal(ctx + B, Hkv, 128), normal(ctx + B, Hkv, 128), normal(B, V)
    parent = synth.spine_tree(rs, B, 8, 3)[0][None]
    tok = synth.distinct_sibling_tokens(rs, parent[0], V)[None]
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()
    parent, tok, ctx_len, row_off = i32(parent), i32(tok), i32([ctx]), torch.zeros(1, dtype=torch.int64, device="cuda")
    k, scale = 8, 1 / math.sqrt(128)

    out = g.tree_attn_gqa(q, kc, vc, row_off, ctx_len, parent, scale)[0]
    argmax, ids, vals = g.node_topk(logits, k)
    table = lambda: (torch.full((V, k), -1, dtype=torch.int32, device="cuda"), torch.zeros(V, k, device="cuda"))
    want_table = table()
    g.harvest(logits, k, tok.view(-1), *want_table)
    path, accepted, bonus = g.accept(tok, parent, argmax.view(1, B))
    torch.cuda.synchronize()
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
        assert torch.equal(o["path"], path) and torch.equal(o["accept_len"], accepted) and torch.equal(o["bonus"], bonus)
        if harvest:
            assert torch.equal(got_table[0], want_table[0]) and torch.allclose(got_table[1], want_table[1], rtol=2e-5, atol=0)
    g.close()
