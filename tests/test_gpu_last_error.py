"""A call that fails reports it in its status and leaves the last error of the library's
CUDA runtime clear: the launch check of the next call, on a good stream, does not find
it.  The failure is a launch into a stream whose capture was invalidated on the host (a
synchronisation inside it)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys, numpy as np, torch
sys.path.insert(0, sys.argv[1])
from paper_2204_07137_gb300 import inputs as I, _lib
from paper_2204_07137_gb300.shac import td_lambda
from paper_2204_07137_gb300.sim import Simulator
m, N = I.cartpole(), int(sys.argv[2])
sim = Simulator([(m, N)], form="batched", h_max=1)
q, qd = (torch.from_numpy(np.ascontiguousarray(x).reshape(-1)).cuda() for x in I.initial_state(m, N, 0))
act = torch.zeros(N, device="cuda")
out = sim.step(q, qd, act)
x = torch.zeros(1000, device="cuda")
reward, value = torch.zeros(4, 8, device="cuda"), torch.zeros(5, 8, device="cuda")
s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
torch.cuda.synchronize()
with torch.cuda.stream(s):
    graph.capture_begin(capture_error_mode="thread_local")
    try:
        s.synchronize()
        print("synchronised")
    except RuntimeError:
        pass
    try:
        sim.step(q, qd, act, out=out, stream=s)
        print("launched")
    except _lib.ShacError as e:
        print("status", e.status)
with torch.cuda.stream(torch.cuda.default_stream()):
    x.add_(1.0)
    td_lambda(reward, value, None, 0.9, 0.9)
    print("next launch ok")
with torch.cuda.stream(s):
    try:
        graph.capture_end()
    except RuntimeError:
        pass
"""


@pytest.mark.parametrize("n", [8, 200000])   # a warp for every item, and items on a counter (its memset fails first)
def test_failed_launch_leaves_no_last_error(n):
    out = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(n)], capture_output=True, text=True, timeout=300)
    lines = out.stdout.split("\n")
    assert lines[:2] == ["status 3", "next launch ok"], out.stdout[-1000:] + out.stderr[-2000:]
