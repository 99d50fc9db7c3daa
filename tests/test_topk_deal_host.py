"""How the top-k's items are dealt to its CTAs, compiled for the host from the library's own header: every item once and in order, no CTA
above the share, no row cut where the share is whole rows, and with node counts as many CTAs as the items of all rows need."""
import ctypes
import subprocess

import pytest

from paper_2604_02047_b200 import build

SOURCE = r"""
#include <cstdint>
#include "topk_deal.cuh"
using namespace goose;
// 0, or what is wrong; *cut: CTAs that start inside a row
extern "C" int walk(int rows, int V, int ctas, int no_second, int counts, int* cut, int* share, int* grid) {
    const int chunks = topk_chunks(V), items = topk_items(rows, V);
    const TopkDeal d = topk_deal(rows, chunks, ctas, no_second, counts);
    *share = topk_share(items, chunks, ctas, no_second); *grid = d.grid; *cut = 0;
    if (d.grid < 1 || d.grid > ctas || d.start(0) != 0 || d.start(d.grid) != items) return 1;
    for (int c = 0; c < d.grid; ++c) {
        const int n = d.start(c + 1) - d.start(c);
        if (n < 1 || n > *share) return 2;
        *cut += d.start(c) % chunks != 0;
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("deal")
    src, so = str(d / "walk.cu"), str(d / "walk.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    r = subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", src, "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(so)

    def call(rows, V, ctas, no_second, counts=False):
        out = [ctypes.c_int() for _ in range(3)]
        rc = lib.walk(rows, V, ctas, int(no_second), int(counts), *map(ctypes.byref, out))
        assert rc == 0, (rc, rows, V, ctas, no_second, counts)
        return [x.value for x in out]                         # CTAs that start inside a row, share, CTAs

    return call


@pytest.mark.parametrize("V", [1, 32000, 32768, 32769, 65536, 98304, 128256, 200000, 262144])
def test_items_are_dealt_once_and_no_row_is_cut_where_the_share_is_whole_rows(walk, V):
    chunks = -(-V // 32768)
    for ctas in (148, 132, 64, 33, 1):
        for rows in list(range(1, 300)) + [500, 511, 900, 1001, 1500, 2000, 2045, 16384]:
            for no_second in (False, True):
                cut, share, grid = walk(rows, V, ctas, no_second)
                least = -(-rows * chunks // ctas)             # of any dealing
                assert least <= share <= least + (chunks > 1)
                if share % chunks == 0:
                    assert cut == 0, (rows, ctas, no_second)
                # node counts: the CTAs that the items as they are need, over which the kernel deals the rows that exist
                assert walk(rows, V, ctas, no_second, True)[2] == -(-rows * chunks // least)


@pytest.mark.parametrize("rows, V, ctas, no_second, share", [(100, 128256, 148, False, 4), (250, 128256, 148, True, 8), (60, 65536, 148, False, 2),
                                                             (60, 65536, 148, True, 1), (33, 65536, 80, True, 1),
                                                             (64, 33000, 48, True, 4), (900, 65536, 148, True, 14), (122, 200000, 148, False, 7),
                                                             (60, 128256, 64, True, 4), (60, 128256, 148, False, 2), (1500, 32000, 148, True, 11)])
def test_the_share(walk, rows, V, ctas, no_second, share):
    assert walk(rows, V, ctas, no_second)[1] == share
