"""GPU parity of the top-k's candidate selection where it can go wrong: rows with many elements at or above the
threshold, chunk lengths at the edges of a thread's, a sweep's and a chunk's share, masked rows, and row log-sum-exps whose
largest value comes late, far above the first sweep's, or not at all.  Identifiers and values bit-exact against the oracle;
the log-sum-exp against numpy in 64 bits: fp32 sums of at most 2^18 terms in chains of at most 64, then trees, hence
|error| <= (64 + 20) 2^-24 + 2 ulp of ex2.approx (2^-22) + the rounding of two arguments below 16 (2^-20 ln 2) = 6e-6, plus
half an ulp of the largest |lse| here (2^-17)."""
import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu

NEG_INF, LOWEST = 0xFF80, 0xFF7F


@pytest.fixture(scope="module")
def goose():
    from paper_2604_02047_b200 import binding, build
    build.build()
    g = binding.Goose(max_S=2, max_B=128, max_H=4)
    yield g
    g.close()


def _rows(V, rng):
    """bf16 bit patterns, one row per kind."""
    bf = synth.f32_to_bf16_bits
    noise = lambda: bf(rng.standard_normal(V).astype(np.float32))  # noqa: E731
    rows = [noise(), np.full(V, bf(np.float32([2.5]))[0], np.uint16)]
    rows += [bf(np.sort(rng.standard_normal(V)).astype(np.float32)), bf(-np.sort(rng.standard_normal(V)).astype(np.float32))]
    rows.append(bf(rng.integers(0, 2, V).astype(np.float32)))                       # half the row ties at the top
    for lo, n in ((V // 2, 1200), (0, 900), (max(0, V - 1500), 1500), (V // 3, 5000)):   # a band far above the rest
        r = noise()
        band = r[lo:lo + n]
        band[:] = bf((50 + 4 * rng.standard_normal(len(band))).astype(np.float32))
        rows.append(r)
    for mask in (NEG_INF, LOWEST):
        r = np.full(V, mask, np.uint16)                                             # all but a few masked; the last one too
        keep = rng.choice(V, min(V, 5), replace=False)
        r[keep] = bf(rng.standard_normal(len(keep)).astype(np.float32))
        rows.append(r)
        r = noise()
        r[:V // 2] = mask
        rows.append(r)
    r = noise()
    r[V - 1] = bf(np.float32([90.0]))[0]                                           # the largest comes last, far above
    rows.append(r)
    rows.append(bf((rng.standard_normal(V) * 1e4).astype(np.float32)))
    return np.stack(rows)


@pytest.mark.parametrize("k", [1, 8, 16])
@pytest.mark.parametrize("V", [16, 248, 4096, 4104, 32000, 32768, 32776, 70008, 128256, 262144])
def test_candidates_of_odd_rows(goose, oracle, V, k):
    rng = np.random.default_rng([V, k])
    bits = _rows(V, rng)
    rows = len(bits)
    x = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    ref_am, ref_ids, ref_vals = oracle.node_topk(bits, k)
    am, ids, vals = goose.node_topk(x, k)
    adj_ids = torch.zeros((rows, k), dtype=torch.int32, device="cuda")
    adj_sc = torch.zeros((rows, k), dtype=torch.float32, device="cuda")
    am2, ids2, vals2, lse = goose.harvest(x, k, torch.arange(rows, dtype=torch.int32, device="cuda"), adj_ids, adj_sc)
    torch.cuda.synchronize()
    for a, i, v in ((am, ids, vals), (am2, ids2, vals2)):
        assert np.array_equal(i.cpu().numpy(), ref_ids) and np.array_equal(a.cpu().numpy(), ref_am)
        assert np.array_equal(v.cpu().numpy().astype(np.float64), ref_vals)
    wide = x.double().cpu().numpy()
    top = wide.max(axis=1)
    ref = top + np.log(np.exp(wide - top[:, None]).sum(axis=1))
    got = lse.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 6e-6 + np.abs(ref) * 2.0 ** -23), (got - ref)
    assert goose.last_status(2).tolist() == [0, 0]


@pytest.fixture(scope="module")
def goose_many():
    from paper_2604_02047_b200 import binding, build
    build.build()
    g = binding.Goose(max_S=8, max_B=128, max_H=4)
    yield g
    g.close()


@pytest.mark.parametrize("k", [8, 16])
@pytest.mark.parametrize("V,repeats", [(4104, 62), (32768, 62), (70008, 21), (128256, 16), (262144, 8)])
def test_odd_rows_many_a_cta(goose_many, oracle, V, repeats, k):
    """The same rows repeated and shuffled: six items and more for every CTA, so that stages and slots come back into use
    behind odd rows, and several chunks of a masked row meet in one CTA or in two."""
    rng = np.random.default_rng([V, k])
    kinds = _rows(V, rng)
    n, sms = len(kinds), torch.cuda.get_device_properties(0).multi_processor_count
    assert n * repeats * -(-V // 32768) > 6 * sms
    which = rng.permutation(np.repeat(np.arange(n), repeats))
    x = torch.from_numpy(kinds.view(np.int16)).view(torch.bfloat16).cuda()[torch.from_numpy(which).cuda()].contiguous()
    ref_am, ref_ids, ref_vals = (a[which] for a in oracle.node_topk(kinds, k))
    rows = len(which)
    wide = torch.from_numpy(kinds.view(np.int16)).view(torch.bfloat16).double().numpy()
    top = wide.max(axis=1)
    ref = (top + np.log(np.exp(wide - top[:, None]).sum(axis=1)))[which]
    for _ in range(3):
        am, ids, vals = goose_many.node_topk(x, k)
        adj_ids = torch.zeros((rows, k), dtype=torch.int32, device="cuda")
        adj_sc = torch.zeros((rows, k), dtype=torch.float32, device="cuda")
        am2, ids2, vals2, lse = goose_many.harvest(x, k, torch.arange(rows, dtype=torch.int32, device="cuda"), adj_ids, adj_sc)
        torch.cuda.synchronize()
        for a, i, v in ((am, ids, vals), (am2, ids2, vals2)):
            assert np.array_equal(i.cpu().numpy(), ref_ids) and np.array_equal(a.cpu().numpy(), ref_am)
            assert np.array_equal(v.cpu().numpy().astype(np.float64), ref_vals)
        got = lse.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - ref) <= 6e-6 + np.abs(ref) * 2.0 ** -23), (got - ref)
    assert goose_many.last_status(8).tolist() == [0] * 8


@pytest.mark.parametrize("V", [32000, 128256])
@pytest.mark.parametrize("below", [0, 8, 12, 24, 43])
def test_log_sum_exp_of_late_values(goose_many, V, below):
    """Rows of which the first eighth of every chunk (what the warps see first) lies `below` the rest.  28000 and more terms of
    one size: their own roundings average out, what is left is half an ulp of a result in [8, 16) (2^-21), the two arguments'
    roundings while they are below 16 (2^-21 ln 2 each) and an ulp of the logarithm (2^-22 of at most 3): 1.9e-6 at worst,
    and 1.2e-6 without the logarithm's, which is rarely a whole one.  With arguments up to 64 it was 1.6e-6."""
    g = torch.Generator(device="cuda").manual_seed(below)
    x = torch.randn((300, V), generator=g, device="cuda")
    x[:, torch.arange(V, device="cuda") % (V // -(-V // 32768)) < 4096] -= below
    x = x.bfloat16()
    adj_ids = torch.zeros((300, 8), dtype=torch.int32, device="cuda")
    adj_sc = torch.zeros((300, 8), dtype=torch.float32, device="cuda")
    lse = goose_many.harvest(x, 8, torch.arange(300, dtype=torch.int32, device="cuda"), adj_ids, adj_sc)[3]
    assert (lse.double() - torch.logsumexp(x.double(), 1)).abs().max().item() <= 1.2e-6


@pytest.mark.parametrize("V,k", [(70008, 8), (128256, 10), (262144, 16)])
def test_long_rows_with_node_counts(goose_many, oracle, V, k):
    """Rows of several chunks, most of them left out by node counts: fewer items than CTAs, and a row's parts are counted over
    the CTAs that have one.  (Counted over empty CTAs between them too, such a row waits for arrivals that never come: nothing
    is written, and the counter in memory, which calls share, spoils the calls behind.)  Outputs hold a mark before each call."""
    S, B = 4, 15
    bits = _rows(V, np.random.default_rng([V, k]))[:B]
    ref_am, ref_ids, ref_vals = oracle.node_topk(bits, k)
    x = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda().repeat(S, 1).contiguous()
    for counts in ([15, 0, 7, 1], None, [1, 1, 1, 15], [0, 15, 15, 3], None):
        nn = None if counts is None else torch.tensor(counts, dtype=torch.int32, device="cuda")
        outs = (torch.full((S * B,), -7, dtype=torch.int32, device="cuda"), torch.full((S * B, k), -7, dtype=torch.int32, device="cuda"),
                torch.full((S * B, k), -7.0, device="cuda"))
        goose_many.node_topk(x, k, n_nodes=nn, B=B, outs=outs)
        torch.cuda.synchronize()
        am, ids, vals = (o.cpu().numpy().reshape(S, B, -1) for o in outs)
        for s, n in enumerate(counts or [B] * S):
            assert np.array_equal(ids[s, :n], ref_ids[:n]) and np.array_equal(am[s, :n, 0], ref_am[:n]), (counts, s)
            assert np.array_equal(vals[s, :n].astype(np.float64), ref_vals[:n])
            assert np.all(am[s, n:] == -7) and np.all(ids[s, n:] == -7) and np.all(vals[s, n:] == -7.0)
