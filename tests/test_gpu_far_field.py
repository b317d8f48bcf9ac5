"""Far-field cells of the barrier against the oracle: every sample's cost, the
collided set, the weights and U*, at sizes where cells are used and at the
edges of the rule that sorts obstacles into near and far.

Cost tolerance, from the arithmetic: a point's sum over J obstacles carries at
most J / 2 FP32 roundings (u = 2^-24) whichever way it is formed, the
polynomial's remainder is at most 2 u, and the draws are within 2e-6 of the
oracle's; at J <= 2000 that is below 8e-5 of the cost, and for J <= 512 below
2e-5.  What a rollout's FP32 positions may add is cost_checks' second term."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W
from cost_checks import POS_ETA
from weight_checks import check_weights

pytestmark = pytest.mark.gpu


def _uni(K, T, J, side, seed=0, r=(0.3, 0.8), **more):
    g = W.rng(seed)
    p = W.base_params(W.UNICYCLE, K=K, T=T, dt=0.05, seed=seed)
    start, goal = np.array([1.0, 1.0, 0.7]), np.array([side - 1.0, side - 1.0, 0.7])
    p.update(x_goal=goal, **more)
    return W.World(p, W.obstacle_field(g, J, (0, 0), (side, side), *r, keep_clear=(start, goal)), start, goal, 1.0)


def _quad(K, T, J, length, seed=0, **more):
    w = W.quad2d(seed, K=K, T=T)
    w.params.update(more)
    return W.World(w.params, W.obstacle_field(W.rng(seed + 1), J, (0, 0), (length, 10), 0.2, 0.6,
                                              keep_clear=(w.x_start, w.goal)), w.x_start, w.goal, 1.0)


def _cases():
    tri = np.array([[0.2, 0.0], [-0.1, 0.15], [-0.1, -0.15]])
    inside = _uni(16001, 50, 150, 40.0, seed=5)
    inside.obstacles[17] = (1.0, 1.5, 3.0)            # the start lies in it
    away = _uni(9999, 50, 200, 45.0, seed=6)
    off = np.array([2.0e5, -3.0e5])
    away.obstacles[:, :2] += off
    for a in (away.x_start, away.goal):
        a[:2] += off
    away.params["x_goal"] = away.goal
    car = W.ackermann(3, K=5003, T=41, J=117)
    grid = W.ackermann_grid(2, K=4096, T=30)
    grid.obstacles = W.ackermann(2, J=80).obstacles
    return dict(
        plain=(_uni(16001, 50, 200, 45.0), None),
        quad=(_quad(8191, 40, 60, 30.0), None),
        quad_points_8=(_quad(4096, 40, 130, 65.0), dict(samples_per_cta=20, threads=512, positions_per_thread=8)),
        car=(car, None),
        car_grid=(grid, None),
        three_points=(_uni(8192, 50, 120, 35.0, shape=tri), None),
        all_near=(_quad(8192, 60, 64, 3.0), None),     # every obstacle within a few metres
        list_full=(_uni(2048, 30, 2000, 6.0, r=(0.005, 0.01)), None),  # over 512 near obstacles
        inside_circle=(inside, None),
        far_origin=(away, None),
        high_floor=(_uni(16384, 40, 200, 45.0, h_eps=4.0), None),
        smoothed=(_uni(16384, 40, 200, 45.0, sgf_window=9, sgf_order=3), None),
        long=(_uni(4096, 256, 100, 32.0), None),
        small_tiles=(_uni(16384, 50, 200, 45.0, **{"lambda": 40.0}),  # many weights, several passes of 3
                     dict(samples_per_cta=3, threads=128, positions_per_thread=8)),
        flat=(_uni(16384, 50, 200, 45.0, **{"lambda": 1.0e5}), None),
        few_warps=(_uni(16384, 50, 200, 45.0), dict(samples_per_cta=32, threads=64, positions_per_thread=14)),
        crowd=(_quad(2048, 100, 500, 250.0), None),
    )


@pytest.mark.parametrize("case", ["plain", "quad", "quad_points_8", "car", "car_grid", "three_points", "all_near",
                                  "list_full", "inside_circle", "far_origin", "high_floor", "smoothed", "long",
                                  "small_tiles", "flat", "few_warps", "crowd"])
def test_far_field_costs_match_the_oracle(case, orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w, tiling = _cases()[case]
    p = w.params
    x = w.x_start
    ctl = orc.new_controller(p)
    ro = orc.step(p, w.obstacles, x, w.reference(x), ctl)
    with binding.Controller(p, tiling=tiling) as g:
        g.set_obstacles(w.obstacles)
        if p.get("grid") is not None:
            g.set_grid(p["grid"], p["grid_ox"], p["grid_oy"], p["grid_res"])
        g.step(x, w.reference(x))
        dbg = g.get_debug()
        g.set_state(np.zeros((int(p["T"]), 2)), p["mu_coarse"], 0.0, True, 0)
        g.step(x, w.reference(x))
        again = g.get_debug()
    S = np.asarray(ro["costs"])
    tol = (2e-5 if len(w.obstacles) <= 512 else 8e-5) * np.maximum(np.abs(S), 1.0)
    tol += POS_ETA * (np.asarray(ro["reach"]) + 1.0) * np.asarray(ro["sens"])
    ratio = np.abs(dbg["costs"] - S) / tol
    assert ratio.max() <= 1.0, f"cost error {ratio.max():.3f} of its tolerance at sample {ratio.argmax()}"
    sure = np.abs(ro["minh"]) > 1e-4
    assert np.array_equal(ro["coll"][sure], dbg["coll"][sure])
    check_weights(ro, dbg, float(p["lambda"]), case)
    # U* within what the weights' errors explain: |dU*| <= sum_k |dw_k| |du_k|
    du = np.maximum(np.abs(np.asarray(p["u_min"])), np.abs(np.asarray(p["u_max"]))) * 2.0
    bound = 1e-5 + np.abs(dbg["weights"] - ro["weights"]).sum() * du.max()
    assert np.abs(dbg["Ustar"] - ro["Ustar"]).max() <= bound
    for k in ("costs", "coll", "Ustar"):               # the same bits again
        assert np.array_equal(dbg[k], again[k])


@pytest.mark.parametrize("T", [200, 240])
def test_served_tiles_near_the_shared_memory_limit(T, orc):
    """Tiles of 32 samples of a long horizon fill the serving kernel's shared
    memory; with no room for cells beside them the request still runs, and
    gives the bits of the same shape alone."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    w = _uni(2048, T, 400, 63.0, seed=8)
    x, xref = w.x_start, w.reference(w.x_start)
    with binding.Server(1, 256 << 20) as s:
        s.set_policy(small_ops_max=0.0, device_queue=True)
        r = s.join(w.params, w.obstacles)
        s.submit(r, x, xref)
        done = []
        while not done:
            done = s.poll()
    assert done[0][4] == 0
    with binding.Controller(w.params, tiling=dict(samples_per_cta=32, threads=256, positions_per_thread=0)) as g:
        g.set_obstacles(w.obstacles)
        g.step(x, xref)
        assert np.array_equal(done[0][1], g.get_control())
