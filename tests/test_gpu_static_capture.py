"""The allocation-free step captured after one ordinary call of the same model
and smoothing, as its contract asks, with another obstacle set: few obstacles
first and many in the capture, or the other way round.  In a process of its
own, whose first step this is."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import ctypes as C, sys
import numpy as np, torch
from paper_2504_06437_gb300 import binding, workloads as W
lib = binding.load()
first, then, window = (int(v) for v in sys.argv[1:])
f64 = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
def caller(J):
    w = W.quad2d(2, K=16384, T=40)
    w.params.update(sgf_window=window, sgf_order=2 if window else 0)
    ob = W.obstacle_field(W.rng(3), J, (0, 0), (5.0 + J, 10), 0.2, 0.6, keep_clear=(w.x_start, w.goal))
    x = w.x_start
    return binding.make_params(w.params), J, [f64(ob), f64(x), f64(w.reference(x)), f64(np.zeros((40, 2))),
                                              f64([w.params["mu_coarse"], 0, 1, 0, 0]), f64(np.zeros(2))]
def call(c, stream):
    p, J, t = c
    q = [C.c_void_p(a.data_ptr()) for a in t]
    rc = lib.mppi_step_static(C.byref(p), q[0], C.c_int32(J), *q[1:], None, C.c_void_p(stream.cuda_stream))
    assert rc == 0, lib.mppi_last_error().decode()
a, b, c = caller(first), caller(then), caller(then)
s = torch.cuda.Stream()
torch.cuda.synchronize()
call(a, s)
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, stream=s):
    call(b, s)
graph.replay()
torch.cuda.synchronize()
call(c, s)
torch.cuda.synchronize()
assert all(torch.equal(u, v) for u, v in zip(b[2][3:], c[2][3:]))
"""


@pytest.mark.parametrize("first,then", [(4, 200), (200, 4)])
@pytest.mark.parametrize("window", [0, 5])
def test_one_call_prepares_a_capture(first, then, window):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", PROGRAM, str(first), str(then), str(window)], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
