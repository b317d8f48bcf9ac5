"""Tiles taken one, two, four or eight in a row by a CTA give the same bits:
every output of a step, for problems whose last row and last merge group are
ragged, with and without far-field cells, in the plain, smoothing and grid
forms.  And the step with rows agrees with the oracle."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cases():
    uni = lambda K, T, J, **p: _field(W.unicycle_stress(3, K=K, T=T), J, **p)  # noqa: E731
    grid = W.ackermann_grid(2, K=4099, T=24)
    grid.obstacles = W.ackermann(2, J=90).obstacles
    return dict(plain=(uni(9001, 9, 10), 3), groups=(uni(40003, 12, 10), 3), cells=(uni(20011, 40, 200), 13),
                cells_groups=(uni(33001, 30, 200), 11), smoothed=(uni(16001, 30, 200, sgf_window=7, sgf_order=2), 7),
                quad=(_field(W.quad2d(3, K=8201, T=30), 130), 9), grid=(grid, 5))


def _field(w, J, **p):
    side = 10.0 * np.sqrt(max(J, 10) / 10.0)
    w.params.update(p)
    w.obstacles = W.obstacle_field(W.rng(4), J, (0, 0), (side, side), 0.2, 0.6, keep_clear=(w.x_start, w.goal))
    return w


@pytest.mark.parametrize("case", ["plain", "groups", "cells", "cells_groups", "smoothed", "quad", "grid"])
def test_rows_of_tiles_give_the_bits_of_single_tiles(case, orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w, S = _cases()[case]
    p, x = w.params, w.x_start
    xref = w.reference(x)
    got = {}
    for rows in (1, 2, 4, 8):
        with binding.Controller(p, tiling=dict(samples_per_cta=S, threads=256, positions_per_thread=0)) as g:
            g.set_obstacles(w.obstacles)
            if p.get("grid") is not None:
                g.set_grid(p["grid"], p["grid_ox"], p["grid_oy"], p["grid_res"])
            g.debug_set_form(tiles_per_cta=rows)
            out = []
            for _ in range(2):
                g.step(x, xref)
                d = g.get_debug()
                out.append([*g.get_control(want_U=True), *(d[k] for k in ("costs", "coll", "weights", "Ustar", "Z", "rho"))])
            got[rows] = out
    for rows in (2, 4, 8):
        for a, b in zip(got[1], got[rows]):
            assert all(np.array_equal(u, v) for u, v in zip(a, b)), rows
    ro = orc.step(p, w.obstacles, x, xref, orc.new_controller(p))
    S_, coll, weights, Us = got[8][0][2:6]
    assert np.max(np.abs(S_ - ro["costs"]) / np.maximum(np.abs(ro["costs"]), 1.0)) < 1e-4
    # U* within what the weights' differences explain: |dU*| <= sum_k |dw_k| |du_k|
    du = 2.0 * np.maximum(np.abs(np.asarray(p["u_min"])), np.abs(np.asarray(p["u_max"]))).max()
    assert np.abs(Us - ro["Ustar"]).max() <= 1e-5 + np.abs(weights - ro["weights"]).sum() * du
