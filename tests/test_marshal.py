"""The argument marshalling of the stream-ordered calls, as far as it goes without a GPU: what it does with tensors happens
before the first CUDA call."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2604_02047_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def marshal():
    build.build()
    return binding.load_marshal()


def test_a_tensor_that_raises_is_an_exception():
    """A subclass that answers is_contiguous() in Python and raises there (in a process of its own: as a C++ exception that
    leaves the entry it ends the interpreter)."""
    code = '''
import torch
from paper_2604_02047_b200 import binding

class Raises(torch.Tensor):
    @staticmethod
    def __new__(cls):
        return torch.Tensor._make_wrapper_subclass(cls, (4,), dtype=torch.float32, device="cuda", dispatch_sizes_strides_policy="strides")
    @classmethod
    def __torch_dispatch__(cls, func, types, args=(), kwargs=None):
        raise KeyError("not here")

try:
    binding.load_marshal().check("f", Raises())
except KeyError as e:
    print("raised", e)
'''
    build.build()
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0 and "raised 'not here'" in r.stdout, (r.returncode, r.stdout, r.stderr[-500:])


def test_what_is_written_is_not_shared(marshal):
    """A copy-on-write clone among the outputs gets memory of its own; one among the inputs need not."""
    def accept(tok, path):
        x = torch.zeros(4, dtype=torch.int32)
        try:
            marshal.accept(None, tok, x, None, x, 1, 4, path, x, x)   # no context: an error code where there is a GPU
        except RuntimeError:
            pass                                                      # no current stream without one

    base = torch.zeros(4, dtype=torch.int32)
    read, written = torch._lazy_clone(base), torch._lazy_clone(base)
    accept(read, written)
    assert torch._C._is_cow_tensor(read) and not torch._C._is_cow_tensor(written)
    assert written.data_ptr() != torch._C._data_address(base) and written.tolist() == [0, 0, 0, 0]


@pytest.mark.parametrize("number", [0, 1, 4096, True])
def test_a_number_is_not_an_address(marshal, number):
    x = torch.zeros(4, dtype=torch.int32)
    for at in (1, 2, 4, 7, 9):                                        # each tensor of the call, read or written
        args = [None, x, x, None, x, 1, 4, x, x, x]
        args[at] = number
        with pytest.raises(AttributeError):
            marshal.accept(*args)
