"""The attention kernel looks at lengths and rows while the kernel in front of it may still be writing them (to bring its first
tile into L2): whatever it sees there, the results are those of the values that stand when its turn comes."""
import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goose():
    from paper_2604_02047_b200 import binding, build
    build.build()
    g = binding.Goose(max_S=48, max_B=128, max_H=64)
    yield g
    g.close()


@pytest.mark.parametrize("H,Hkv,B,ctxs,counts", [
    (32, 32, 16, [1000], None), (16, 4, 60, [700], None), (8, 8, 5, [300, 0, 2000], None), (16, 2, 17, [900, 64], [17, 0]),
    (16, 16, 4, [30] * 40, None)])
@pytest.mark.parametrize("junk", [0x7FFFFFFF, -5, 123456, 0])
def test_lengths_written_just_before(goose, H, Hkv, B, ctxs, counts, junk):
    from paper_2604_02047_b200 import binding
    S = len(ctxs)
    rng = np.random.default_rng([H, B, S])
    x = synth.make_inputs(S, H, B, ctxs, [synth.random_tree(rng, B) for _ in ctxs], Hkv=Hkv, seed=H + S, V=8, with_logits=False)
    d = binding.to_device(x)
    nn = None if counts is None else torch.tensor(counts, dtype=torch.int32, device="cuda")

    def call(row_off, ctx_len, n_nodes):
        out = torch.full_like(d["q"], 7.0)
        goose.tree_attn_gqa(d["q"], d["k_cache"], d["v_cache"], row_off, ctx_len, d["parent"], x.scale, out=out, n_nodes=n_nodes)
        return out

    want = call(d["row_off"], d["ctx_len"], nn)
    late = [None if t is None else torch.full_like(t, junk) for t in (d["row_off"], d["ctx_len"], nn)]
    busy = torch.zeros(1 << 26, device="cuda")
    torch.cuda.synchronize()
    busy.add_(1)                                              # the copies and the call are enqueued while this runs
    for t, v in zip(late, (d["row_off"], d["ctx_len"], nn)):
        if t is not None:
            t.copy_(v)
    got = [call(*late) for _ in range(2)]
    torch.cuda.synchronize()
    assert not goose.last_status(S).any()
    assert torch.equal(got[0], want) and torch.equal(got[1], want)
