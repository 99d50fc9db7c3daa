"""Which form of the attention a step of one sequence takes and how many SMs its top-k gets, asked of the library itself with the figures of
one device: the choice is host arithmetic."""
import ctypes
import subprocess

import pytest

from paper_2604_02047_b200 import build

SOURCE = r"""
#include "goose_internal.cuh"
#include "topk_deal.cuh"
extern "C" void split(const int* max_clusters, int sms, int S, int B, int H, int Hkv, long long kv_rows, int V, int k, int harvest, int counts, int* out) {
    goose_ctx c = {};
    c.num_sms = sms;
    for (int n = 2; n <= 8; ++n) c.max_clusters[n] = max_clusters[n];
    const goose::StepSplit s = goose::step_split(&c, S, B, H, Hkv, kv_rows, V, k, harvest, counts);
    const bool long_topk = harvest || goose::topk_items(S * B, V) > sms;
    out[0] = s.cluster; out[1] = s.topk_ctas;
    out[2] = goose::attn_cluster(&c, S, B, H, Hkv, kv_rows, long_topk ? 2 : 1); out[3] = goose::attn_heads(B, H, Hkv);
    out[4] = s.cluster > 1 ? goose::attn_cluster_fits(&c, s.cluster, S, B, H, Hkv, kv_rows, long_topk ? 2 : 1) : 1;
    out[5] = goose::topk_items(S * B, V);
}
"""
MAX_CLUSTERS = [0, 0, 74, 45, 33, 26, 22, 15, 15]     # of 2 to 8 CTAs, on a device of 148 SMs
SMS = 148


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    src, so = str(d / "split.cu"), str(d / "split.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    r = subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", src, build.build(), "-o", so, "-Xlinker", "-rpath=" + build.HERE],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(so)
    most = (ctypes.c_int * 9)(*MAX_CLUSTERS)

    def call(S, B, H, Hkv, kv_rows, V, harvest, counts=False, k=8):
        out = (ctypes.c_int * 6)()
        lib.split(most, SMS, S, B, H, Hkv, ctypes.c_longlong(kv_rows), V, k, int(harvest), int(counts), out)
        return list(out)

    return call


CHOICES = [  # heads, rows, keys, spare rows of the cache, vocabulary, with the harvest -> CTAs a head
    # smaller clusters than the largest, or clusters where the largest leave the top-k too few SMs
    (32, 8, 60, 1000, 0, 128256, True, 5), (32, 8, 60, 3001, 0, 128256, True, 5), (32, 8, 60, 1000, 0, 128256, False, 5),
    (16, 2, 128, 3001, 0, 128256, True, 4), (16, 16, 60, 829, 0, 33000, True, 5), (32, 32, 64, 2118, 0, 33000, True, 3),
    (32, 32, 128, 340, 0, 32000, True, 2),
    # the largest: nothing, or too little, is gained by fewer
    (32, 8, 60, 6000, 0, 128256, True, 6), (32, 8, 60, 3001, 0, 128256, False, 6), (32, 8, 80, 3001, 0, 32000, True, 5),
    (32, 8, 16, 630, 0, 200000, True, 8), (16, 2, 80, 766, 0, 50000, False, 8), (32, 32, 80, 2048, 0, 32000, True, 4),
    # a top-k of one item an SM: not weighed
    (32, 32, 16, 512, 0, 32000, False, 4), (32, 8, 60, 2859, 0, 65536, False, 6),
    # the persistent form: too many items for the SMs that clusters leave, too long a prefix, more to lose than to gain
    (32, 32, 128, 1000, 0, 128256, True, 1), (40, 40, 80, 4096, 0, 32000, False, 1), (32, 8, 128, 2730, 0, 32000, True, 1),
    # spare rows: the cache's length decides, and a gain has to stand with a quarter of it
    (32, 8, 60, 3001, 13000, 128256, True, 1), (32, 8, 100, 662, 2648, 33000, True, 1), (32, 8, 60, 3001, 3100, 128256, True, 6),
]


@pytest.mark.parametrize("H, Hkv, B, ctx, spare, V, harvest, cluster", CHOICES)
def test_choice(split, H, Hkv, B, ctx, spare, V, harvest, cluster):
    got, ctas, largest, heads, fits, items = split(1, B, H, Hkv, ctx + B + spare, V, harvest)
    assert got == cluster
    assert ctas == (SMS - heads * got - 4 if got > 1 else 0)


# a row that is cut over so many CTAs that their lists have more than 32 candidates is dear to merge
MERGES = [  # heads, rows, keys, vocabulary, k -> CTAs a head
    (32, 8, 21, 586, 128256, 8, 7), (32, 8, 21, 586, 128256, 10, 8), (40, 8, 16, 488, 200000, 8, 8), (16, 16, 31, 1535, 152064, 16, 6),
    (40, 40, 16, 479, 152064, 16, 3), (32, 8, 60, 3001, 128256, 10, 5),
]


@pytest.mark.parametrize("H, Hkv, B, ctx, V, k, cluster", MERGES)
def test_choice_knows_what_a_merge_costs(split, H, Hkv, B, ctx, V, k, cluster):
    assert split(1, B, H, Hkv, ctx + B, V, True, k=k)[0] == cluster


def test_every_choice_is_one_that_the_device_holds(split):
    changed = 0
    for H, Hkv in ((32, 32), (40, 40), (52, 52), (32, 8), (16, 2), (32, 4), (8, 8), (4, 4)):
        for B in (1, 16, 33, 60, 100, 128):
            for kv_rows in (1, 129, 700, 1500, 3100, 8000, 16512, 2 ** 31 - 1):
                for V in (1000, 32000, 65536, 128256, 262144):
                    for harvest in (False, True):
                        for counts in (False, True):
                            got, ctas, largest, heads, fits, items = split(1, B, H, Hkv, kv_rows, V, harvest, counts)
                            assert fits and 1 <= got <= 8
                            if got == 1:
                                assert ctas == 0
                            else:
                                assert MAX_CLUSTERS[got] >= heads and ctas == SMS - heads * got - 4 > 0 and items <= 7 * ctas
                            if not harvest and items <= SMS:
                                assert got in (largest, 1)
                            changed += got not in (largest, 1)
    assert changed > 50
    for S in (2, 16):
        assert split(S, 60, 32, 8, 6000, 128256, True)[:2] == [1, 0]
