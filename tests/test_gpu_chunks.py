"""Tiles taken several in a row by one CTA: the results are those of the same
tiles taken one by one, bit for bit.  The one-controller step, the batch and
the device queue choose their own number of tiles in a row (1, 2, 4 or 8), and
all must agree; the last chunk of a grid and of a merge group is ragged."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [257 * 3, 4097, 40003, 131071])
def test_rows_of_tiles_do_not_change_the_results(K, orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = W.unicycle_small(4)
    p = dict(w.params, K=K, T=9)
    tiling = dict(samples_per_cta=3, threads=256, positions_per_thread=8)
    x = w.x_start
    xref = W.line_reference(p, w.x_start, w.goal, x, w.v_ref)
    ro = orc.step(p, w.obstacles, x, xref, orc.new_controller(p))
    with binding.Controller(p, tiling=tiling) as g, binding.Batch(1, 256 << 20) as b, \
            binding.Server(1, 256 << 20) as s:
        g.set_obstacles(w.obstacles)
        g.step(x, xref)
        u0, U = g.get_control(want_U=True)
        costs = g.get_debug()["costs"]
        slot = b.add(p, w.obstacles, tiling=tiling)
        b.step([slot], [x], [xref])
        assert np.array_equal(b.controls()[0], u0)
        st = b.state(slot)
        assert np.array_equal(st["U"], U) and np.array_equal(st["costs"], costs)
        assert np.max(np.abs(costs - ro["costs"]) / np.maximum(np.abs(ro["costs"]), 1.0)) < 1e-4
        # the queue's robots have tiles of 32: against a controller of that shape
        s.set_policy(small_ops_max=0.0, device_queue=True)
        r = s.join(p, w.obstacles)
        s.submit(r, x, xref)
        done = []
        while not done:
            done = s.poll()
    with binding.Controller(p, tiling=dict(tiling, samples_per_cta=32)) as g:
        g.set_obstacles(w.obstacles)
        g.step(x, xref)
        assert done[0][4] == 0 and np.array_equal(done[0][1], g.get_control())
