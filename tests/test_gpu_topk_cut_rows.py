"""Rows of the top-k that are merged over CTAs: sizes whose share of a CTA is no multiple of a row's chunks, so that some CTA starts inside a
row, through each form of the kernel.  And harvests on both sides of the number of rows above which a kernel behind the top-k writes the
table."""
import numpy as np
import pytest
import torch

import test_gpu_harvest as harvest
import test_gpu_harvest_table as table
import test_gpu_parity as parity
from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def goose():
    from paper_2604_02047_b200 import binding
    g = binding.Goose(max_S=16, max_B=128, max_H=8)
    yield g
    g.close()


def share(rows, V):
    """Items of a CTA as long as whole rows are not within one more of it; a range of them starts inside a row then."""
    chunks, sms = -(-V // 32768), torch.cuda.get_device_properties(0).multi_processor_count
    q = -(-rows * chunks // sms)
    assert q % chunks and (q + 1) % chunks
    return q


@pytest.mark.parametrize("rows, V, k", [(60, 100000, 8), (30, 128256, 16)])
def test_topk(goose, oracle, rows, V, k):
    share(rows, V)
    parity.test_topk_more_items_than_sms(goose, oracle, rows, V, k)


def test_harvest(goose, oracle):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    V, k = 70000, 8
    rows = next(rows for rows in range(sms, 2 * sms) if -(-3 * rows // sms) % 3 == 1)
    assert share(rows, V) == 4
    rng = np.random.default_rng(31)
    bits = synth.f32_to_bf16_bits((rng.standard_normal((rows, V)) * 3).astype(np.float32))
    harvest._check(goose, oracle, bits, k, rng.permutation(V)[:rows].astype(np.int32), V, V=V)


@pytest.mark.parametrize("rows, V, k, tokens", [(60, 128256, 10, 20), (149, 128256, 8, 149)])
def test_table(oracle, rows, V, k, tokens):
    assert share(rows, V) > 1
    table.test_table_matches_the_oracle(oracle, rows, V, k, tokens)


@pytest.mark.parametrize("rows, V, k, tokens", [(1536, 1000, 8, 1000), (1537, 1000, 8, 1000), (1536, 640, 10, 3)])
def test_table_at_the_line(oracle, rows, V, k, tokens):
    table.test_table_matches_the_oracle(oracle, rows, V, k, tokens)


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
