"""The attention kernel looks at lengths, node counts and rows while the kernel in front of it may still be writing them (to bring its
first tile into L2, and to know its place): whatever it sees there, the results are those of the values that stand when its turn comes.
The kernel in front is one of the test's own: it releases its dependents at once and writes the words half a millisecond later, so that the
look falls on the stale ones (a copy or an element-wise kernel of torch would end before the attention starts)."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2604_02047_b200 import synth

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
__global__ void late_words(int* dst, const int* src, int n) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t0 = clock64();
    for (int i = 0; i < 1000000 && clock64() - t0 < 1000000; ++i) {}
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}
extern "C" int write_late(void* dst, const void* src, int n, void* stream) {
    late_words<<<1, 128, 0, (cudaStream_t)stream>>>((int*)dst, (const int*)src, n);
    return cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def goose():
    from paper_2604_02047_b200 import binding, build
    build.build()
    g = binding.Goose(max_S=48, max_B=128, max_H=64)
    yield g
    g.close()


@pytest.fixture(scope="module")
def write_late(tmp_path_factory):
    from paper_2604_02047_b200 import build
    d = tmp_path_factory.mktemp("late")
    src, lib = str(d / "late.cu"), str(d / "late.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    r = subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", src, "-o", lib], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    fn = ctypes.CDLL(lib).write_late

    def call(dst, src):
        rc = fn(ctypes.c_void_p(dst.data_ptr()), ctypes.c_void_p(src.data_ptr()), dst.numel(),
                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
    return call


# what stands in the arrays before: lengths, node counts, row offsets (None: the right ones)
STALE = {"short": (lambda c, rows: c // 3, lambda n: n, None), "long": (lambda c, rows: min(c + 129, rows), lambda n: n, None),
         "zero": (lambda c, rows: 0 * c, lambda n: 0 * n, 0), "negative": (lambda c, rows: -5, lambda n: -3, -7),
         "beyond": (lambda c, rows: rows + 1, lambda n: n + 200, 1 << 20), "largest": (lambda c, rows: 0x7FFFFFFF, lambda n: 0x7FFFFFFF, (1 << 63) - 1),
         "one node": (lambda c, rows: c, lambda n: 1, None), "rows alone": (lambda c, rows: c, lambda n: n, 3)}


@pytest.mark.parametrize("H,Hkv,B,ctxs,counts", [
    (32, 32, 16, [1000], None), (32, 32, 60, [380], [51]), (16, 4, 60, [700], None), (16, 4, 20, [700], [13]),   # a cluster a head
    (8, 8, 5, [300, 0, 2000], None), (8, 8, 33, [300, 7, 2000], [33, 0, 18]), (40, 40, 8, [900, 1500], None),    # persistent
    (16, 2, 17, [900, 64], [17, 0]), (16, 2, 60, [900, 64, 1300], None),
    (16, 16, 4, [30] * 40, None)])                                                                               # no look: more than 32
@pytest.mark.parametrize("stale", STALE)
@pytest.mark.parametrize("step", [False, True])
def test_lengths_written_just_before(goose, write_late, H, Hkv, B, ctxs, counts, stale, step):
    from paper_2604_02047_b200 import binding
    S = len(ctxs)
    rng = np.random.default_rng([H, B, S])
    x = synth.make_inputs(S, H, B, ctxs, [synth.random_tree(rng, B) for _ in ctxs], Hkv=Hkv, seed=H + S, V=512, k=4)
    rows = x.k_cache.shape[0]
    old_ctx, old_nn, old_row = STALE[stale]
    nn = [B] * S if counts is None else counts

    def words(ctx, n, row):
        return torch.from_numpy(np.concatenate([np.asarray(row, np.int64).view(np.int32), np.asarray(ctx, np.int32), np.asarray(n, np.int32)])).cuda()

    right = words(x.ctx_len, nn, x.row_off)
    wrong = words([old_ctx(int(c), rows) for c in x.ctx_len], [old_nn(n) for n in nn], x.row_off if old_row is None else [old_row] * S)

    def call(buf, front):
        d = binding.to_device(x)
        row_off, ctx_len, n_nodes = buf[:2 * S].view(torch.int64), buf[2 * S:3 * S], buf[3 * S:] if counts else None
        outs = goose.alloc_step_outputs(S, B, H, 128, 4)
        for t in outs.values():
            t.fill_(7)
        torch.cuda.synchronize()
        if front:
            write_late(buf, right)
        if step:
            goose.verify_step_gqa(d["q"], d["k_cache"], d["v_cache"], row_off, ctx_len, d["parent"], d["draft_tok"], d["logits"], 4, x.scale,
                                  outs=outs, n_nodes=n_nodes)
        else:
            goose.tree_attn_gqa(d["q"], d["k_cache"], d["v_cache"], row_off, ctx_len, d["parent"], x.scale, out=outs["out"], n_nodes=n_nodes)
        torch.cuda.synchronize()
        assert not goose.last_status(S).any()
        return list(outs.values()) + [d["k_cache"], d["v_cache"]]

    want, got = call(right.clone(), False), call(wrong, True)
    assert all(torch.equal(a, b) for a, b in zip(want, got))
