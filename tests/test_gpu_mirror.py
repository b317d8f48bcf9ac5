"""The sequence read back after a step (mppi_get_control with U) against the
controller's device state, wherever it may come from: the mirror that the
step wrote, or the device after a state set from the host or a device step."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [W.unicycle_small, lambda s: W.quad2d(s, K=300, T=1), lambda s: W.ackermann(s, K=1, T=256)])
def test_sequence_read_back_is_the_device_state(make):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = make(1)
    x, T = w.x_start, int(w.params["T"])
    xref = w.reference(x)
    y = x + 0.05
    with binding.Controller(w.params) as g, binding.Controller(w.params) as other:
        for c in (g, other):
            c.set_obstacles(w.obstacles)
        for _ in range(3):
            g.step(x, xref)
            u0, U = g.get_control(want_U=True)
            st = g.get_state()
            assert np.array_equal(U, st["U"])
            assert np.array_equal(u0, g.get_debug()["Ustar"][0])
        # a state set from the host is what is read back before the next step
        V = np.full((T, 2), 0.01)
        g.set_state(V, st["S_e"], st["beta"], False, 2)
        assert np.array_equal(g.get_control(want_U=True)[1], V)
        # and the step after it, whose number the mirror has shown before,
        # gives its own outputs
        other.set_state(V, st["S_e"], st["beta"], False, 2)
        for c in (g, other):
            c.step(y, xref)
        (ua, Ua), (ub, Ub) = g.get_control(want_U=True), other.get_control(want_U=True)
        assert np.array_equal(ua, ub) and np.array_equal(Ua, Ub) and np.array_equal(Ua, g.get_state()["U"])
        d = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (x, xref)]
        g.step_device(d[0].data_ptr(), d[1].data_ptr())
        assert np.array_equal(g.get_control(want_U=True)[1], g.get_state()["U"])
