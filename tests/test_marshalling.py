"""The native marshalling module's C entries: what throws inside comes out as a Python exception (no GPU), and a
launch that has to wait does not stop the other Python threads (-m gpu)."""
import os
import subprocess
import sys
import threading
import time

import pytest
import torch

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


@pytest.mark.gpu
@pytest.mark.parametrize("train", [False, True])
def test_other_threads_go_on_while_the_launch_queue_is_full(train):
    """Behind a second of GPU work more calls are made than the launch queue holds: the caller waits in the driver for
    most of that second, and this thread must not."""
    import paper_2605_11196_b200 as vla
    x = torch.randn((1, 1, 1, 32), device="cuda")
    call = (lambda: vla.vla_scan(x, x, x, 1.0)) if train else (lambda: vla.vla_forward(x, x, x, 1.0))
    call()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    torch.cuda._sleep(2_000_000_000)     # cycles: about a second
    b.record()
    t = threading.Thread(target=lambda: [call() for _ in range(6000)])
    t.start()
    longest, last = 0.0, time.perf_counter()
    while t.is_alive():
        time.sleep(1e-3)
        now = time.perf_counter()
        longest, last = max(longest, now - last), now
    t.join()
    torch.cuda.synchronize()
    assert longest < 0.25 * a.elapsed_time(b) * 1e-3, (longest, a.elapsed_time(b))


@pytest.mark.gpu
def test_want_status_takes_any_truth_value():
    import paper_2605_11196_b200 as vla
    x = torch.randn((1, 1, 1, 32), device="cuda")
    for yes in (True, 1, "yes"):
        assert vla.vla_forward(x, x, x, 1.0, want_status=yes).status is not None
    for no in (False, 0, None):
        assert vla.vla_forward(x, x, x, 1.0, want_status=no).status is None
