"""Buffers that a call can do without, on a device that is short of memory: a
child process holds most of it, so that the larger buffer is refused and the
least one fits."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
COMMON = """
import sys
sys.path.insert(0, {root!r})
import torch
import paper_1801_04723_gb300 as spin
from paper_1801_04723_gb300 import inputs

MB = 1 << 20
def hold(left):
    "Allocate all but `left` bytes of the device's free memory."
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - left, dtype=torch.uint8, device="cuda:0")

A = inputs.spd_gram_device(4161, 5, "cuda:0", alpha=0.3)
B = A[:4096, :4096].contiguous()
X, Y = torch.empty_like(A), torch.empty_like(B)
small = inputs.spd_gram_device(256, 5, "cuda:0", alpha=0.3)
side = torch.cuda.Stream()
with torch.cuda.stream(side):  # kernels and contexts in place before memory is short
    spin.invert(small)
    spin.invert(small, precision="bf16x3")
torch.cuda._sleep(1000)
torch.cuda.synchronize()
torch.cuda.empty_cache()
"""


def child(body):
    r = subprocess.run([sys.executable, "-c", COMMON.format(root=ROOT) + body], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("which,precision", [("A", "fp64"), ("B", "bf16x3")])
def test_a_refused_buffer_is_not_asked_for_again(which, precision):
    """After the first call, calls neither free nor allocate: they return while another stream's work runs."""
    child(f"""
M, R = {which}, {'X' if which == 'A' else 'Y'}
n = M.shape[0]
kept = hold(spin.workspace_bytes(n, precision={precision!r}) + 300 * MB)
s, busy = torch.cuda.Stream(), torch.cuda.Stream()
with torch.cuda.stream(s):
    for i in range(2):
        spin.invert(M, out=R, precision={precision!r})
torch.cuda.synchronize()
with torch.cuda.stream(busy):
    torch.cuda._sleep(1 << 30)  # about half a second
    done = busy.record_event()
with torch.cuda.stream(s):
    for tol in (1e-10, 1e-9, 1e-8):  # other arguments: launches, then captures
        spin.invert(M, out=R, precision={precision!r}, tol=tol, blocking=False)
assert not done.query(), "a call waited for the device"
torch.cuda.synchronize()
with torch.cuda.stream(s):
    info = spin.sync()
assert info["status"] == 0
del kept
torch.cuda.empty_cache()
assert (M @ R - torch.eye(n, dtype=M.dtype, device="cuda:0")).norm() <= 1e-8 * M.norm() * R.norm()
""")


def test_an_idle_arena_makes_way():
    """The arena of large FP64 products on one stream is given back when another call's workspace does not fit."""
    child("""
s, t = torch.cuda.Stream(), torch.cuda.Stream()
with torch.cuda.stream(s):
    spin.invert(A, out=X)
    first, diff = X.clone(), X.clone()
torch.cuda.synchronize()
torch.cuda.empty_cache()
kept = hold(spin.workspace_bytes(4096, precision="bf16x3") // 2)
with torch.cuda.stream(t):
    _, info = spin.invert(B, out=Y, precision="bf16x3")
assert info["status"] == 0 and info["rel_residual"] <= 1e-10
with torch.cuda.stream(s):
    for i in range(3):  # launches, capture, replay; with an arena or without
        X.zero_()
        _, info = spin.invert(A, out=X)
        assert info["status"] == 0
        assert torch.sub(X, first, out=diff).norm() <= 1e-12 * first.norm()
""")
