"""What build() makes again, and what it needs."""
import os
import sys
import types

import pytest
import torch

from paper_2604_02047_b200 import binding, build


@pytest.fixture
def commands(monkeypatch, tmp_path):
    """build() as it stands, in a folder of its own, with every command noted instead of run."""
    build.build()
    for name in ("LIB", "HASH_FILE", "MARSHAL", "MARSHAL_HASH_FILE"):
        at = tmp_path / os.path.basename(getattr(build, name))
        at.write_bytes(b"" if name in ("LIB", "MARSHAL") else open(getattr(build, name), "rb").read())
        monkeypatch.setattr(build, name, str(at))
    ran = []

    def run(cmd, **kw):
        ran.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(build, "HERE", str(tmp_path))
    monkeypatch.setattr(build.subprocess, "run", run)
    return ran


def test_nothing_changed(commands):
    build.build()
    assert commands == []


def test_another_torch(commands, monkeypatch):
    """The module reads tensors by the layout of the torch that it was compiled for; the CUDA library knows nothing of torch."""
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    build.build()
    assert len(commands) == 1 and commands[0][0] == "g++"
    del commands[:]
    build.build()
    assert commands == []


def test_another_interpreter(commands, monkeypatch):
    var = build.sysconfig.get_config_var
    assert build.MARSHAL.endswith(var("EXT_SUFFIX"))
    monkeypatch.setattr(build.sysconfig, "get_config_var", lambda name: "cpython-999" if name == "SOABI" else var(name))
    build.build()
    assert len(commands) == 1 and commands[0][0] == "g++"


def test_without_torch(commands, monkeypatch):
    """The C ABI alone: nvcc for every source and the link, no module."""
    monkeypatch.setitem(sys.modules, "torch", None)              # import torch raises ImportError
    os.remove(build.MARSHAL)
    build.build(force=True)
    assert len(commands) == len(build.SOURCES) + 1 and all("nvcc" in c[0] for c in commands)
    assert not os.path.exists(build.MARSHAL)


def test_a_module_of_another_torch_is_not_used(monkeypatch):
    build.build()
    binding.load_marshal()
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    with pytest.raises(binding.GooseError, match="built for torch"):
        binding.load_marshal()
