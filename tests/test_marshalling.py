"""The native marshalling module's C entries: what throws inside comes out as a Python exception (no GPU)."""
import subprocess
import sys
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SIZES_IN_PYTHON = """
import torch
from paper_2605_11196_b200 import binding as b

class Sized(torch.Tensor):      # claims to be on a GPU and answers for its sizes in Python
    @staticmethod
    def __new__(cls):
        return torch.Tensor._make_wrapper_subclass(cls, (2, 3, 40, 32), dtype=torch.float32, device="cuda", dispatch_sizes_strides_policy="sizes")
    @classmethod
    def __torch_dispatch__(cls, func, types, args=(), kwargs=None):
        raise LookupError("no sizes today")

x, n = Sized(), None
try:
    %s
except LookupError as e:
    print("raised", e)
"""


@pytest.mark.parametrize("call", ["b.native().forward(x, x, x, 1.0, n, n, n, n, 0, 1e-4, n, n, n, n, n, True, 0, n, 0)",
                                  "b.native().scan(x, x, x, 1.0, n, n, n, n, 0, 1e-4, torch.zeros((), dtype=torch.int32))"])
def test_an_exception_in_a_tensor_argument_comes_out_as_itself(call):
    """In a process of its own: an exception that leaves a C entry ends the process."""
    r = subprocess.run([sys.executable, "-c", _SIZES_IN_PYTHON % call], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "raised no sizes today" in r.stdout, (r.returncode, r.stderr[-500:])
