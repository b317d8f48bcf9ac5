"""A step with far-field cells is not slower than the same step without them:
however many samples carry weight (with no bound on the second look, these took
2.5 to 13 times as long with cells), and where the cells' shared memory would
leave one CTA on an SM instead of two (1.33 and 1.38 times)."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cases():
    few = W.quad2d(1, K=74, T=172)
    few.obstacles = W.obstacle_field(W.rng(2), 771, (0, 0), (385, 10), 0.2, 0.6, keep_clear=(few.x_start, few.goal))
    field = lambda J, box, r, w: W.obstacle_field(W.rng(7), J, (0, 0), box, *r, keep_clear=(w.x_start, w.goal))  # noqa: E731
    quad, uni = W.quad2d(1, K=41425, T=133), W.unicycle_stress(1, K=16259, T=137)
    quad.obstacles, uni.obstacles = field(36, (20, 10), (0.2, 0.6), quad), field(50, (22, 22), (0.3, 0.8), uni)
    return dict(quad_one_cta=(quad, 1.0e9), unicycle_one_cta=(uni, 1.0e9), vehicle_small=(W.ackermann(3, K=221, T=132, J=378), 252.0),
                vehicle=(W.ackermann(5, K=1076, T=156, J=577), 213.0),
                quad5=(W.quad5(2, K=1589, T=121, J=197), 19.0),
                flat=(few, 1.0e9),
                long=(W.ackermann(4, K=800, T=200, J=120), 1.0e3))


@pytest.mark.parametrize("case", ["vehicle_small", "vehicle", "quad5", "flat", "long", "quad_one_cta",
                                  "unicycle_one_cta"])
def test_cells_do_not_cost_time(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w, lam = _cases()[case]
    w.params["lambda"] = lam
    x, xref = (torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (w.x_start, w.reference(w.x_start)))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def ms(cells):
        with binding.Controller(w.params) as g:
            g.set_obstacles(w.obstacles)
            g.debug_set_form(cells=cells)
            best = np.inf
            for _ in range(6):
                g.set_state(np.zeros((g.T, 2)), w.params["mu_coarse"], 0.0, True, 0)   # the same steps again
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(s)
                for _ in range(8):
                    g.step_device(x.data_ptr(), xref.data_ptr(), s)
                b.record(s)
                b.synchronize()
                best = min(best, a.elapsed_time(b))
            return best

    assert ms(True) <= 1.2 * ms(False)
