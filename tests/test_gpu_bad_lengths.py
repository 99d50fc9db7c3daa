"""Lengths and row offsets on the device that put a sequence outside the cache, up to the largest that their types hold: the sequence gets its status bit, zeros
and an untouched cache, the others in the batch their usual results, and nothing is written around the outputs."""
import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth
from test_gpu_parity import ATTN_TOL, LSE_TOL, attn_row_err

pytestmark = pytest.mark.gpu
BIG = 2 ** 31 - 1


@pytest.fixture(scope="module")
def goose():
    from paper_2604_02047_b200 import binding, build
    build.build()
    g = binding.Goose(max_S=4, max_B=128, max_H=64)
    yield g
    g.close()


def _framed(shape, dtype):
    """A tensor in the middle of a larger one that is filled with sevens; the second result says whether the frame still is."""
    n, guard = int(np.prod(shape)), 1 << 16
    whole = torch.full((n + 2 * guard,), 7.0, dtype=dtype, device="cuda")
    return whole[guard:guard + n].view(shape), lambda: bool((whole[:guard] == 7).all() and (whole[guard + n:] == 7).all())


@pytest.mark.parametrize("length", ["rows + 1", "rows - nodes + 1", 123456, BIG - 300, BIG - 150, BIG - 128, BIG])
@pytest.mark.parametrize("H,Hkv,B,ctxs,counts", [
    (32, 32, 16, [500], False), (32, 32, 16, [500], True), (16, 2, 60, [300], False), (52, 52, 80, [700], False),
    (8, 8, 16, [500, 130, 0], False), (16, 4, 33, [90, 600, 257], True)])
@pytest.mark.parametrize("step", [False, True])
def test_length_outside_the_cache(goose, oracle, H, Hkv, B, ctxs, counts, length, step):
    from paper_2604_02047_b200 import binding
    S, V, bad = len(ctxs), 512, len(ctxs) // 2
    rng = np.random.default_rng([H, Hkv, B, S])
    x = synth.make_inputs(S, H, B, ctxs, [synth.random_tree(rng, B) for _ in ctxs], Hkv=Hkv, seed=H + B, V=V, k=4)
    rows = x.k_cache.shape[0]
    ctx = x.ctx_len.copy()
    ctx[bad] = {"rows + 1": rows + 1, "rows - nodes + 1": rows - B + 1}.get(length, length)
    d = binding.to_device(x)
    d["ctx_len"] = torch.from_numpy(ctx).cuda()
    nn = torch.full((S,), B, dtype=torch.int32, device="cuda") if counts else None
    before = [d[n].clone() for n in ("k_cache", "v_cache")]
    out, out_frame = _framed((S, B, H, 128), torch.bfloat16)
    lse, lse_frame = _framed((S, B, H), torch.float32)
    if step:
        outs = goose.alloc_step_outputs(S, B, H, 128, 4)
        outs["out"], outs["lse"] = out, lse
        goose.verify_step_gqa(d["q"], d["k_cache"], d["v_cache"], d["row_off"], d["ctx_len"], d["parent"], d["draft_tok"], d["logits"],
                              4, x.scale, outs=outs, n_nodes=nn)
    else:
        goose.tree_attn_gqa(d["q"], d["k_cache"], d["v_cache"], d["row_off"], d["ctx_len"], d["parent"], x.scale, out=out, lse=lse, n_nodes=nn)
    torch.cuda.synchronize()
    assert goose.last_status(S).tolist() == [8 if s == bad else 0 for s in range(S)]
    assert out_frame() and lse_frame()
    assert (out[bad] == 0).all() and (lse[bad] == 0).all()
    ref, ref_lse = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)
    good = [s for s in range(S) if s != bad]
    if good:
        got = out[good].float().cpu().numpy().astype(np.float64)
        assert attn_row_err(got, ref[good]).max() <= ATTN_TOL and np.abs(lse[good].cpu().numpy() - ref_lse[good]).max() <= LSE_TOL
    r0, r1 = int(x.row_off[bad]), int(x.row_off[bad]) + ctxs[bad] + B
    for name, was in zip(("k_cache", "v_cache"), before):
        assert torch.equal(d[name][r0:r1], was[r0:r1])


@pytest.mark.parametrize("row", [2 ** 63 - 1, 2 ** 63 - 130, 2 ** 62, -2 ** 63])
def test_row_offset_outside_the_cache(goose, oracle, row):
    from paper_2604_02047_b200 import binding
    S, H, B, V = 2, 8, 16, 512
    x = synth.make_inputs(S, H, B, [130, 140], [synth.chain_tree(B)] * S, seed=3, V=V, k=4)
    d = binding.to_device(x)
    off = x.row_off.copy()
    off[1] = row
    d_off = torch.from_numpy(off).cuda()
    ref, _ = oracle.tree_attn(x.q, x.k_cache, x.v_cache, x.row_off, x.ctx_len, x.parent, x.scale)

    def check(out):
        torch.cuda.synchronize()
        assert goose.last_status(S).tolist() == [0, 8]
        assert (out[1] == 0).all() and attn_row_err(out[:1].float().cpu().numpy().astype(np.float64), ref[:1]).max() <= ATTN_TOL

    for impl in (binding.ATTN_MMA, binding.ATTN_UMMA):
        goose.set_attn_impl(impl)
        try:
            check(goose.tree_attn(d["q"], d["k_cache"], d["v_cache"], d_off, d["ctx_len"], d["parent"], x.scale)[0])
        finally:
            goose.set_attn_impl(binding.ATTN_AUTO)
    check(goose.verify_step(d["q"], d["k_cache"], d["v_cache"], d_off, d["ctx_len"], d["parent"], d["draft_tok"], d["logits"], 4, x.scale)["out"])
    before = [d[n].clone() for n in ("k_cache", "v_cache")]
    path = torch.tensor([[0, 2, 3] + [-1] * (B - 3)] * S, dtype=torch.int32).cuda()
    goose.kv_compact(d["k_cache"], d["v_cache"], d_off, d["ctx_len"], path, torch.tensor([2, 2], dtype=torch.int32).cuda())
    assert goose.last_status(S).tolist() == [0, 8]
    for name, was in zip(("k_cache", "v_cache"), before):
        assert torch.equal(d[name][146:], was[146:])
    if row > 0:                                               # on host buffers: refused before anything is enqueued
        h = {n: t.cpu().pin_memory() for n, t in d.items() if isinstance(t, torch.Tensor)}
        new = torch.zeros((S, B, H, 128), dtype=torch.bfloat16).pin_memory()
        outs = goose.alloc_step_outputs(S, B, H, 128, 4, device="cpu")
        with pytest.raises(binding.GooseError, match="invalid argument"):
            goose.verify_step_host(d["k_cache"], d["v_cache"], h["q"], new, new, torch.from_numpy(off), h["ctx_len"], h["parent"],
                                   h["draft_tok"], h["logits"], 4, x.scale, outs)
