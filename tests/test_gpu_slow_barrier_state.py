"""Barrier states that hardly decay (gamma_bas next to 1): the sums of the
unrolled recursion against the oracle, which steps it.  The goal lies beside
an obstacle, so the sum of the barrier state's reference term (T (T + 1) / 2
of them at gamma 1) is most of the cost."""
import numpy as np
import pytest

from cost_checks import cost_errors
from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("one_minus", [1e-2, 1e-5, 1e-8, 1e-12, 2.0 ** -53])
@pytest.mark.parametrize("T", [1, 37, 256])
def test_costs_with_a_barrier_state_that_hardly_decays(one_minus, T, orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = W.unicycle_small(0)
    p = dict(w.params, K=200, T=T, gamma_bas=1.0 - one_minus)
    obs = np.concatenate([w.obstacles, [[w.goal[0] + 1.0, w.goal[1], 0.95]]])
    x = w.x_start
    xref = W.line_reference(p, w.x_start, w.goal, x, w.v_ref)
    ro = orc.step(p, obs, x, xref, orc.new_controller(p))
    with binding.Controller(p) as g:
        g.set_obstacles(obs)
        g.step(x, xref)
        S = g.get_debug()["costs"]
    assert cost_errors(ro, S)[2] <= 1.0
