"""Steps of one controller on changing streams.  mppi_get_control returns when
the step's outputs are on the host, which can be before the step has written
all of the state that the next one reads; whichever stream the next step runs
on, and captured or not, the results are those of one stream bit for bit."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("want_U", [True, False])
@pytest.mark.parametrize("make", [W.unicycle_small, lambda s: W.quad2d(s, K=300, T=250)])
def test_streams_in_turn_give_the_bits_of_one_stream(make, want_U):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = make(3)
    x, xref = w.x_start, w.reference(w.x_start)
    dx, dr = (torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (x, xref))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), None, torch.cuda.Stream(), torch.cuda.default_stream()]
    with binding.Controller(w.params) as one, binding.Controller(w.params) as g:
        for c in (one, g):
            c.set_obstacles(w.obstacles)
        for i in range(40):
            if i % 5 == 4:        # device inputs in between
                one.step_device(dx.data_ptr(), dr.data_ptr())
                g.step_device(dx.data_ptr(), dr.data_ptr(), streams[i % 4])
            else:
                one.step(x, xref)
                g.step(x, xref, streams[i % 4])
            a, b = one.get_control(want_U), g.get_control(want_U)
            assert np.array_equal(np.concatenate([np.ravel(v) for v in (a if want_U else [a])]),
                                  np.concatenate([np.ravel(v) for v in (b if want_U else [b])])), i
        s1, s2 = one.get_state(), g.get_state()
        assert np.array_equal(s1["U"], s2["U"]) and s1["S_e"] == s2["S_e"] and s1["iter"] == s2["iter"] == 40


def test_a_step_captured_after_get_control_waits_for_the_step_before():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = W.quad2d(5, K=512, T=200)
    x, xref = w.x_start, w.reference(w.x_start)
    dx, dr = (torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (x, xref))
    torch.cuda.synchronize()
    with binding.Controller(w.params) as one, binding.Controller(w.params) as g:
        for c in (one, g):
            c.set_obstacles(w.obstacles)
            c.step(x, xref)
            c.get_control(want_U=True)
        for _ in range(3):
            one.step_device(dx.data_ptr(), dr.data_ptr())
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=side):
            g.step_device(dx.data_ptr(), dr.data_ptr(), side)
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        a, b = one.get_state(), g.get_state()
        assert np.array_equal(a["U"], b["U"]) and a["S_e"] == b["S_e"] and a["iter"] == b["iter"] == 4
