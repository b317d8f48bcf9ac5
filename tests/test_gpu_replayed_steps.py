"""Steps launched by a graph the library does not see: what is read back after
them, and after ordinary steps that follow, is the last step's."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("replays", [1, 2, 3, 4])
def test_control_after_replayed_device_steps(replays):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = W.quad2d(1, K=2048, T=60)
    x, xref = w.x_start, w.reference(w.x_start)
    dx, dr = (torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (x, xref))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with binding.Controller(w.params) as g:
        g.set_obstacles(w.obstacles)
        g.step(x, xref, s)
        g.get_control(want_U=True)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            g.step_device(dx.data_ptr(), dr.data_ptr(), s)
        with torch.cuda.stream(s):
            for _ in range(replays):
                graph.replay()
        for _ in range(6):
            g.step(x, xref, s)
            u0, U = g.get_control(want_U=True)
            assert np.array_equal(U, g.get_state()["U"]) and np.array_equal(u0, g.get_debug()["Ustar"][0])
            g.step(x, xref, s)
            assert np.array_equal(g.get_control(), g.get_debug()["Ustar"][0])


def test_control_after_replays_of_a_captured_host_step():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = W.quad2d(1, K=2048, T=60)
    x, xref = w.x_start, w.reference(w.x_start)
    s = torch.cuda.Stream()
    with binding.Controller(w.params) as g:
        g.set_obstacles(w.obstacles)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            g.step(x, xref, s)
        for _ in range(5):
            with torch.cuda.stream(s):
                graph.replay()
            u0, U = g.get_control(want_U=True)
            assert np.array_equal(U, g.get_state()["U"]) and np.array_equal(u0, g.get_debug()["Ustar"][0])
