"""The harvest's table is written by the top-k kernel itself: fewer rows than SMs, ranges of more items than a CTA has slots, rows whose
chunks are spread over CTAs and within one, tokens that many rows share or that are no row of the table.  Against the oracle: ids of the
table exact, untouched rows included, scores within the 1e-5 of a 32-bit sum."""
import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows, V, k, tokens", [(1, 8, 1, 8), (149, 64, 16, 64), (900, 4096, 8, 40), (2000, 512, 10, 512),
                                                (37, 32769, 8, 5), (75, 100001, 10, 30)])
def test_table_matches_the_oracle(oracle, rows, V, k, tokens):
    from paper_2604_02047_b200 import binding
    goose = binding.Goose(max_S=16, max_B=128, max_H=8)
    rng = np.random.default_rng(rows)
    ldl = (V + 7) & ~7
    bits = synth.f32_to_bf16_bits((2 * rng.standard_normal((rows, ldl))).astype(np.float32))
    tok = rng.integers(-1, tokens, rows).astype(np.int32)
    tok[rows // 2] = V                                        # outside the table
    ids0 = np.full((V, k), -7, np.int32)
    scores0 = np.full((V, k), -1.0, np.float32)
    logits = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    want_ids, want_scores, want_lse = oracle.harvest(bits, k, tok, ids0, scores0.astype(np.float64), V=V)
    for _ in range(2):                                        # a second call finds the counters as the first did
        ids, scores = torch.from_numpy(ids0).cuda(), torch.from_numpy(scores0).cuda()
        lse = goose.harvest(logits, k, torch.from_numpy(tok).cuda(), ids, scores, V=V)[3]
        torch.cuda.synchronize()
        assert np.array_equal(ids.cpu().numpy(), want_ids)
        got = scores.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - want_scores) <= 1e-5 * np.abs(want_scores) + 1e-12)
        assert np.abs(lse.cpu().numpy() - want_lse).max() <= 2e-5
    assert not goose.last_status(1).any()
    goose.close()
