"""The attention's work partition, compiled for the host from the kernels' own header and walked as the roles walk it: every tile of
every head dealt exactly once, in order, within the arrays -- for lengths that no kernel should meet as well (they are device data),
where a sequence counts as one of the whole cache.  The merge's idea of which CTAs have a part of a head agrees.  And the check that
every kernel makes of a sequence's rows."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2604_02047_b200 import build

SOURCE = r"""
#include "tree_attn_combine.cuh"
using namespace goose;
static uint32_t magic(int n) { return (uint32_t)((0x100000000ull + n - 1) / n); }
// 0, or what is wrong.  idle: CTAs whose range is idle items alone.  first / last [S][Hw]: the CTAs that have a part of the head; dealt [S][Hw]: its tiles so far
extern "C" int walk(int S, int B, int Hw, int G, int cluster, int kv_rows, const int32_t* ctx_len, const int32_t* n_nodes,
                    int32_t* first, int32_t* last, int32_t* dealt, int32_t* idle) {
    const int grid = cluster > 1 ? Hw * cluster : G;
    Work wk;
    wk.ctx_len = ctx_len; wk.n_nodes = n_nodes; wk.S = S; wk.H = Hw; wk.B = B; wk.G = grid; wk.kv_rows = kv_rows;
    wk.G_magic = magic(cluster > 1 ? cluster : grid);
    wk.init();
    for (int cta = 0; cta < grid; ++cta) {
        Cursor cu;
        long long w_begin, w_end;
        if (cluster > 1) {
            const int head = (int)mul_hi(cta, wk.G_magic), rank = cta - head * cluster, T = wk.tiles(0);
            w_begin = (long long)head * T + cluster_start(T, rank, cluster, wk.G_magic);
            w_end = (long long)head * T + cluster_start(T, rank + 1, cluster, wk.G_magic);
            cu.w = w_begin; cu.s = 0; cu.h = head; cu.t = cluster_start(T, rank, cluster, wk.G_magic); cu.T = T;
        } else {
            w_begin = wk.cta_start(cta); w_end = wk.cta_start(cta + 1);
            if (w_begin < w_end) cu.seek(wk, w_begin);
        }
        if (w_begin > w_end) return 1;
        if (w_begin == w_end) continue;
        if (!cu.any(w_end)) { ++*idle; continue; }
        while (cu.w < w_end) {
            if (cu.s < 0 || cu.s >= S || cu.h < 0 || cu.h >= Hw) return 2;
            const int at = cu.s * Hw + cu.h, n = cu.run(w_end);
            if (cu.T != wk.tiles(cu.s) || cu.t != dealt[at]) return 3;
            if (n < 1 || cu.t + n > cu.T) return 4;
            if (first[at] < 0) first[at] = cta;
            last[at] = cta; dealt[at] += n;
            cu.skip(wk, n);
        }
    }
    if (cluster > 1) return 0;
    long long off = 0;                                      // the merge's side
    for (int s = 0; s < S; ++s) {
        const int T = wk.tiles(s);
        for (int h = 0; h < Hw && T > 0; ++h) {
            const long long w = off + (long long)h * wk.width(T) + wk.pad;
            if (wk.cta_of(w) != first[s * Hw + h] || wk.cta_of(w + T - 1) != last[s * Hw + h]) return 5;
        }
        off += (long long)Hw * wk.width(T);
    }
    return 0;
}
extern "C" int outside(int64_t row, int ctx, int nn, int64_t kv_rows) { return rows_outside(row, ctx, nn, kv_rows); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("partition")
    src, lib = str(d / "walk.cu"), str(d / "walk.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    r = subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", src, "-o", lib], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(lib)


@pytest.fixture(scope="module")
def walk(lib):
    def call(B, Hw, G, cluster, kv_rows, ctx, counts):
        S = len(ctx)
        c = np.asarray(ctx, np.int32)
        nn = None if counts is None else np.asarray(counts, np.int32)
        first, last, dealt = (np.full((S, Hw), v, np.int32) for v in (-1, -1, 0))
        call.idle = ctypes.c_int32(0)
        p = lambda a: None if a is None else a.ctypes.data_as(ctypes.c_void_p)
        return lib.walk(S, B, Hw, G, cluster, kv_rows, p(c), p(nn), p(first), p(last), p(dealt), ctypes.byref(call.idle)), dealt

    return call


BIG = 2 ** 31 - 1
LENGTHS = [0, 1, 111, 112, 113, 127, 128, 895, 896, 900, 901, 1028, 123456, BIG - 300, BIG - 144, BIG - 143, BIG - 128, BIG - 16, BIG,
           -1, -5, -2 ** 31]


@pytest.mark.parametrize("counts", [False, True])
@pytest.mark.parametrize("form", ["cluster", "persistent"])
@pytest.mark.parametrize("B", [1, 16, 128])
def test_every_tile_is_dealt_once(walk, form, B, counts):
    kv_rows = 900
    rng = np.random.default_rng([B, counts, len(form)])
    shapes = [(n, 148 // n, 1) for n in range(2, 9)] + [(n, 1, 1) for n in (2, 8)] if form == "cluster" else \
             [(1, Hw, S) for Hw, S in ((1, 1), (4, 1), (37, 1), (52, 1), (8, 3), (32, 5), (7, 40))]
    for cluster, Hw, S in shapes:
        for length in LENGTHS:
            # the length in question among good ones, and (S > 1) by itself everywhere
            lists = [[length]] if S == 1 else [[int(rng.integers(0, kv_rows - B + 1)) for _ in range(S - 1)] + [length], [length] * S]
            for ctx in lists:
                nn = [int(rng.choice([0, 1, B, B, -3, B + 1])) for _ in ctx] if counts else None
                rc, dealt = walk(B, Hw, 148, cluster, kv_rows, ctx, nn)
                assert rc == 0, (rc, cluster, Hw, ctx, nn)
                for s, c in enumerate(ctx):
                    n = B if nn is None else nn[s] if 0 <= nn[s] <= B else 0
                    assert (dealt[s] == (0 if n == 0 else -(-(min(max(c, 0), kv_rows) + n) // 128))).all()


@pytest.mark.parametrize("Hw,B,ctx,idle", [(8, 20, 4700, True), (8, 20, 4716, True), (32, 16, 9000, False)])
def test_ranges_of_idle_items_alone(walk, Hw, B, ctx, idle):
    """Two idle items stand in front of a head: with about two items a CTA some CTAs have nothing else, and count as without work."""
    rc, dealt = walk(B, Hw, 148, 1, ctx + B, [ctx], None)
    assert rc == 0 and (dealt == -(-(ctx + B) // 128)).all() and (walk.idle.value > 0) == idle


@pytest.mark.parametrize("kv_rows", [1, 900, BIG, 2 ** 40])
def test_rows_outside_the_cache(lib, kv_rows):
    """Row offsets up to the ends of 64 bits, against integers without an end."""
    ends = [0, 1, 5, kv_rows - 17, kv_rows - 16, kv_rows, kv_rows + 1, 2 ** 62, 2 ** 63 - 2 ** 31 - 200, 2 ** 63 - 300, 2 ** 63 - 16, 2 ** 63 - 1, -1, -2 ** 63]
    for row in ends:
        for ctx in (0, 1, 16, 883, 899, 900, BIG - 200, BIG, -1, -2 ** 31):
            for n in (1, 16, 128):
                want = ctx < 0 or row < 0 or row + ctx + n > kv_rows
                assert lib.outside(ctypes.c_int64(row), ctx, n, ctypes.c_int64(kv_rows)) == want, (row, ctx, n)
