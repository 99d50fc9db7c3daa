"""The harvest's table is written by the top-k kernel itself, and for many rows by a kernel behind it: fewer rows than SMs, ranges of
more items than a CTA has slots, rows whose chunks are spread over CTAs and within one, tokens that many rows share or that are no row of
the table, both sides of the line between the two.  Against the oracle: ids of the table exact, untouched rows included, scores within the
1e-5 of a 32-bit sum."""
import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows, V, k, tokens", [(1, 8, 1, 8), (149, 64, 16, 64), (900, 4096, 8, 40), (2000, 512, 10, 512),
                                                (37, 32769, 8, 5), (75, 100001, 10, 30),
                                                (1536, 1000, 8, 1000), (1537, 1000, 8, 1000), (1536, 640, 10, 3)])
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


@pytest.mark.parametrize("rows, V, k, tokens", [(60, 128256, 10, 20), (149, 128256, 8, 149)])
def test_table_of_rows_that_are_merged_over_ctas(oracle, rows, V, k, tokens):
    chunks, sms = -(-V // 32768), torch.cuda.get_device_properties(0).multi_processor_count
    share = -(-rows * chunks // sms)                          # items of a CTA: ranges of them start inside rows
    assert share > 1 and share % chunks and (share + 1) % chunks
    test_table_matches_the_oracle(oracle, rows, V, k, tokens)


@pytest.mark.parametrize("rows, V", [(8192, 4096), (5000, 32000)])
def test_many_rows_cost_what_their_logits_cost(rows, V):
    """The look for a later row with a row's token grows with the rows; the call may not.  The log-sum-exp and the table take 1.3 to 1.55
    times the top-k alone where nothing waits for that look, 1.9 to 6 times where the top-k's CTAs do."""
    from paper_2604_02047_b200 import binding
    goose = binding.Goose(max_S=64, max_B=128, max_H=8)
    logits = torch.randn(rows, V, generator=torch.Generator(device="cuda").manual_seed(0), device="cuda", dtype=torch.bfloat16)
    tok = torch.arange(rows, dtype=torch.int32, device="cuda")           # distinct: no look ends early
    ids, scores = torch.zeros((rows, 8), dtype=torch.int32, device="cuda"), torch.zeros((rows, 8), device="cuda")

    def fastest(call):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        times = []
        for _ in range(7):
            call()
            ev[0].record()
            for _ in range(5):
                call()
            ev[1].record()
            torch.cuda.synchronize()
            times.append(ev[0].elapsed_time(ev[1]) / 5 * 1e3)
        return min(times)

    alone, harvest = fastest(lambda: goose.node_topk(logits, 8)), fastest(lambda: goose.harvest(logits, 8, tok, ids, scores))
    print("%d x %d: top-k %.1f us, harvest %.1f" % (rows, V, alone, harvest))
    goose.close()
    assert harvest <= 1.75 * alone
