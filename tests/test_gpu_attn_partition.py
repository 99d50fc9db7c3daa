"""GPU parity of the persistent attention form's work partition: lists with idle items in front of every head (from two tiles
a CTA on) and without, one sequence and more than a warp has lanes, sequences that have left, heads that end on and next to
the edges of CTAs; every row against the oracle."""
import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth
from test_gpu_parity import ATTN_TOL, LSE_TOL, attn_row_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goose():
    from paper_2604_02047_b200 import binding, build
    build.build()
    g = binding.Goose(max_S=48, max_B=128, max_H=64)
    yield g
    g.close()


@pytest.mark.parametrize("H,Hkv,B,ctxs,counts", [
    (16, 16, 4, [30] * 40, None), (16, 16, 4, [30] * 40, [4, 0, 1, 4] * 10), (16, 4, 8, list(range(0, 480, 10)), None),
    (52, 52, 3, [900], None), (52, 52, 3, [700], None), (37, 37, 5, [1019, 1020], None), (37, 37, 5, [3, 2000, 0], [5, 5, 0]),
    (8, 8, 20, [4700], None), (64, 16, 40, [600, 200], None)])
def test_partition(goose, oracle, H, Hkv, B, ctxs, counts):
    from paper_2604_02047_b200 import binding
    S = len(ctxs)
    rng = np.random.default_rng([H, Hkv, B, S])
    x = synth.make_inputs(S, H, B, ctxs, [synth.random_tree(rng, B) for _ in ctxs], Hkv=Hkv, seed=7 * H + S, V=8, with_logits=False)
    ref, ref_lse = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)
    d = binding.to_device(x)
    nn = None if counts is None else torch.tensor(counts, dtype=torch.int32, device="cuda")
    out, lse = torch.full_like(d["q"], 7.0), torch.full(d["q"].shape[:3], 7.0, device="cuda")
    goose.tree_attn_gqa(d["q"], d["k_cache"], d["v_cache"], d["row_off"], d["ctx_len"], d["parent"], x.scale, out=out, lse=lse, n_nodes=nn)
    torch.cuda.synchronize()
    assert not goose.last_status(S).any()
    out, lse = out.float().cpu().numpy().astype(np.float64), lse.cpu().numpy()
    for s, n in enumerate(counts or [B] * S):
        assert np.all(out[s, n:] == 7.0) and np.all(lse[s, n:] == 7.0)
        if n:
            assert attn_row_err(out[s, :n], ref[s, :n]).max() <= ATTN_TOL and np.abs(lse[s, :n] - ref_lse[s, :n]).max() <= LSE_TOL


@pytest.mark.parametrize("H,Hkv,B,ctx", [(8, 8, 20, 4700), (8, 8, 20, 4716), (16, 2, 16, 4096), (40, 40, 16, 1000), (32, 32, 33, 300), (4, 4, 1, 0)])
def test_one_sequence_in_a_large_cache(goose, oracle, H, Hkv, B, ctx):
    """One sequence whose cache has 60000 spare rows: the persistent form, which the exact caches of these sizes do not meet.  The
    first two lists have CTAs with idle items alone (8 heads of 37 tiles: 2.1 items a CTA, two idle ones first)."""
    from paper_2604_02047_b200 import binding
    rng = np.random.default_rng([H, Hkv, B, ctx])
    x = synth.make_inputs(1, H, B, [ctx], [synth.random_tree(rng, B)], Hkv=Hkv, seed=H + ctx, V=8, with_logits=False)
    ref, ref_lse = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)
    d = binding.to_device(x)
    roomy = [torch.cat([d[n], torch.full((60000, Hkv, 128), float("nan"), dtype=torch.bfloat16, device="cuda")]) for n in ("k_cache", "v_cache")]
    before = goose.launch_count()
    out, lse = goose.tree_attn_gqa(d["q"], *roomy, d["row_off"], d["ctx_len"], d["parent"], x.scale, want_lse=True)
    torch.cuda.synchronize()
    assert goose.launch_count() == before + 2, "main kernel and merge"
    assert not goose.last_status(1).any()
    assert attn_row_err(out.float().cpu().numpy().astype(np.float64), ref).max() <= ATTN_TOL
    assert np.abs(lse.cpu().numpy() - ref_lse).max() <= LSE_TOL
