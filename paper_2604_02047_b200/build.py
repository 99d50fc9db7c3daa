"""Build libgoose.so (the CUDA library behind the C ABI, nvcc for sm_100a) and, where torch is installed, the extension module
_marshal (its argument marshalling for Python) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libgoose.so")
# named for the interpreter whose ABI it has: another one does not import it
MARSHAL = os.path.join(HERE, "_marshal" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
MARSHAL_SOURCE = "marshal.cpp"
SOURCES = ["api.cu", "node_topk.cu", "harvest.cu", "accept.cu", "kv_compact.cu", "tree_attn_mma.cu",
           "tree_attn_umma.cu", "spine_tree.cpp"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
              "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


HASH_FILE = LIB + ".srchash"
MARSHAL_HASH_FILE = MARSHAL + ".srchash"


def _hash(files, *words) -> str:
    """Hash of what is built from (contents, not time stamps: a copied tree keeps no mtimes)."""
    import hashlib
    h = hashlib.sha256()
    for f in files:
        h.update(os.path.basename(f).encode())
        h.update(open(f, "rb").read())
    h.update(" ".join(words).encode())
    return h.hexdigest()


def _source_hash() -> str:
    files = sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != MARSHAL_SOURCE)
    return _hash(files + [os.path.join(INCLUDE, "goose.h")], *NVCC_FLAGS, *SOURCES)


def _up_to_date(built: str, hash_file: str, want: str) -> bool:
    return os.path.exists(built) and os.path.exists(hash_file) and open(hash_file).read().strip() == want


def _marshal_flags(torch) -> list:
    return ["-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi()), '-DGOOSE_BUILT_FOR="%s"' % torch.__version__]


def _build_marshal(force: bool) -> None:
    """Host code only; the torch headers and libraries are those of the running interpreter's torch, whose version and the
    interpreter's ABI are part of the hash."""
    try:
        import torch
    except ImportError:                                       # callers of the C ABI need no Python module
        return
    flags = _marshal_flags(torch)
    want = _hash([os.path.join(CSRC, MARSHAL_SOURCE), os.path.join(INCLUDE, "goose.h")], *flags, sysconfig.get_config_var("SOABI") or "")
    if not force and _up_to_date(MARSHAL, MARSHAL_HASH_FILE, want):
        return
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = MARSHAL + ".tmp%d" % os.getpid()
    cmd = ["g++"] + flags
    for d in (INCLUDE, os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
              os.path.join(cuda, "include"), sysconfig.get_path("include")):
        cmd += ["-I", d]
    cmd += [os.path.join(CSRC, MARSHAL_SOURCE), "-o", tmp, "-L", HERE, "-l:libgoose.so", "-L", os.path.join(root, "lib"),
            "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("building the extension module _marshal failed")
    os.replace(tmp, MARSHAL)
    with open(MARSHAL_HASH_FILE, "w") as f:
        f.write(want + "\n")


def build(force: bool = False, verbose: bool = False) -> str:
    """Build what does not match its sources; returns the path of libgoose.so."""
    _build_library(force, verbose)
    _build_marshal(force)
    return LIB


def _build_library(force: bool, verbose: bool) -> None:
    """Compile every source for sm_100a and link libgoose.so; no-op when the library matches the sources."""
    src_hash = _source_hash()
    if not force and _up_to_date(LIB, HASH_FILE, src_hash):
        return
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    nvcc = _nvcc()
    extra = ["-Xptxas", "-v"] if verbose else []

    def compile_one(src: str) -> str:
        obj = os.path.join(objdir, os.path.splitext(src)[0] + ".o")
        cmd = [nvcc] + NVCC_FLAGS + extra + ["-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed for %s" % src)
        return obj

    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + ".tmp%d" % os.getpid()
    r = subprocess.run([nvcc, "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"],
                       capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("link failed")
    os.replace(tmp, LIB)
    with open(HASH_FILE, "w") as f:
        f.write(src_hash + "\n")


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
