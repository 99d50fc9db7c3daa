"""The attention kernel keeps a row of scores in 128 registers a thread, with one warp a scheduler and so nothing to hide a spill
behind: every instantiation has to fit its registers."""
import os
import re
import subprocess

from paper_2604_02047_b200 import build


def test_attention_kernel_does_not_spill(tmp_path):
    cmd = [build._nvcc()] + build.NVCC_FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, "tree_attn_umma.cu"),
                                                "-o", str(tmp_path / "x.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    found = re.findall(r"Compiling entry function '(\w*tree_attn_umma_kernel\w*)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
                       r.stdout + r.stderr, re.S)
    assert len(found) == 8, "grouped x counts x cluster"
    assert [(s, l) for _, s, l in found] == [("0", "0")] * 8
