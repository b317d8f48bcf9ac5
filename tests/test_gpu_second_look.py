"""The second look at the samples that carry the weights (far-field cells).

Two properties.  The update is the softmax of the costs that are reported,
also where costs move by more than the temperature when they are summed again
(a start inside a circle, a small floor h_eps, small temperatures).  And the
samples looked at end with the costs of the direct evaluation but for one
common amount: the differences between the two forms of the step are the same
for all of them."""
import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W
from weight_checks import SELF_RTOL

pytestmark = pytest.mark.gpu


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    return binding


def _unicycle(K, T, J, side, seed=0, **more):
    p = W.base_params(W.UNICYCLE, K=K, T=T, dt=0.05, seed=seed)
    x, goal = np.array([1.0, 1.0, 0.7]), np.array([side - 1.0, side - 1.0, 0.7])
    p.update(x_goal=goal, **more)
    return W.World(p, W.obstacle_field(W.rng(seed), J, (0, 0), (side, side), 0.3, 0.8, keep_clear=(x, goal)), x, goal, 1.0)


def _quad(K, T, J, length, seed=0):
    w = W.quad2d(seed, K=K, T=T)
    return W.World(w.params, W.obstacle_field(W.rng(seed + 1), J, (0, 0), (length, 10), 0.2, 0.6,
                                              keep_clear=(w.x_start, w.goal)), w.x_start, w.goal, 1.0)


def _step(binding, w, tiling=None, cells=True):
    p = w.params
    with binding.Controller(p, tiling=tiling) as g:
        g.set_obstacles(w.obstacles)
        if p.get("grid") is not None:
            g.set_grid(p["grid"], p["grid_ox"], p["grid_oy"], p["grid_res"])
        g.debug_set_form(cells=cells)
        g.step(w.x_start, w.reference(w.x_start))
        return g.get_debug()


def _softmax(costs, lam):
    e = np.exp(-(costs - costs.min()) / lam)
    return e / e.sum()


INSIDE = [(m, h, lam) for m in ("unicycle", "quad2d") for h in (1e-3, 1e-5, 1e-6, 1e-7) for lam in (1.0, 30.0)
          if (m, h) != ("quad2d", 1e-7)]  # (there a cost's last bit is 512 lambda)


def _start_inside(model, h_eps, lam, seed):
    w = _unicycle(20000, 50, 150, 38.0, seed) if model == "unicycle" else _quad(8192, 40, 60, 30.0, seed)
    x = w.x_start
    w.obstacles[len(w.obstacles) // 2] = (x[0], x[1] + 0.5, 3.0)      # the start lies in it
    w.params.update({"h_eps": h_eps, "lambda": lam})
    return w


@pytest.mark.parametrize("seed", range(8))
@pytest.mark.parametrize("model,h_eps,lam", INSIDE + [("unicycle", 1e-3, 0.05), ("quad2d", 1e-3, 0.05)])
def test_update_is_the_softmax_of_the_costs(model, h_eps, lam, seed):
    binding = _gpu()
    w = _start_inside(model, h_eps, lam, seed)
    p = w.params
    d = _step(binding, w)
    # Z is taken relative to the high part of the smallest cost's float pair,
    # which is within half a last place of it
    rel = d["costs"].min() - d["rho"]
    assert np.isfinite(d["Z"]) and d["Z"] >= 0.999 * np.exp(-(abs(rel) + 2.0 ** -24 * abs(d["rho"])) / lam)
    ww = _softmax(d["costs"], lam)
    big = ww > 1e-8
    assert np.abs(d["weights"][big] / ww[big] - 1.0).max() <= SELF_RTOL
    lo, hi = np.asarray(p["u_min"]), np.asarray(p["u_max"])
    draws = binding.debug_draws(p, d["S_e_used"], 0, int(p["K"]), int(p["T"]))[1]
    du = np.clip(draws.astype(np.float64), lo.astype(np.float32), hi.astype(np.float32))
    assert np.abs(d["Ustar"] - np.clip(np.einsum("k,ktd->td", ww, du), lo, hi)).max() <= 1e-5


def _cases():
    tri = np.array([[0.2, 0.0], [-0.1, 0.15], [-0.1, -0.15]])
    car, grid = W.ackermann(3, K=9973, T=41, J=117), W.ackermann_grid(2, K=8192, T=30)
    grid.obstacles = W.ackermann(2, J=90).obstacles
    smooth = _unicycle(16384, 40, 200, 45.0)
    smooth.params.update(sgf_window=9, sgf_order=3)
    return dict(plain=(_unicycle(16001, 50, 200, 45.0), None), three_points=(_unicycle(16384, 50, 120, 35.0, shape=tri), None),
                quad=(_quad(16383, 40, 80, 40.0), None),
                quad_points_8=(_quad(8192, 40, 130, 65.0), dict(samples_per_cta=20, threads=512, positions_per_thread=8)),
                car=(car, None), car_grid=(grid, None), smoothed=(smooth, None),
                two_levels=(_unicycle(65536, 40, 200, 45.0), None),
                several_passes=(_unicycle(32768, 50, 200, 45.0), dict(samples_per_cta=3, threads=128, positions_per_thread=8)))


@pytest.mark.parametrize("case", ["plain", "three_points", "quad", "quad_points_8", "car", "car_grid", "smoothed",
                                  "two_levels", "several_passes"])
def test_samples_looked_at_have_the_direct_costs_but_for_one_amount(case):
    binding = _gpu()
    w, tiling = _cases()[case]
    # a temperature at which five samples weigh over a hundredth (a first
    # step's costs do not depend on it)
    S = _step(binding, w, tiling, cells=False)["costs"]
    lam = next(v for v in np.geomspace(1e-2, 1e3, 400) if (_softmax(S, v) >= 0.01).sum() >= 5)
    w.params["lambda"] = float(lam)
    direct, cells = _step(binding, w, tiling, cells=False), _step(binding, w, tiling)
    listed = _softmax(S, lam) >= 0.01
    shift = cells["costs"] - direct["costs"]
    assert np.abs(shift[~listed]).max() > 0.0          # cells were used
    # the change of a cost is a float, its common part too: two roundings each
    tol = 4.0 * 2.0 ** -24 * np.abs(shift).max() + 2.0 ** -50 * np.abs(S).max()
    assert np.ptp(shift[listed]) <= tol
    assert np.abs(cells["weights"][listed] / cells["weights"][listed].sum()
                  - direct["weights"][listed] / direct["weights"][listed].sum()).max() <= 3e-6


@pytest.mark.parametrize("seed", [0, 1])
@pytest.mark.parametrize("model,h_eps", [("unicycle", 1e-5), ("unicycle", 1e-7), ("quad2d", 1e-5), ("quad2d", 1e-6)])
def test_samples_looked_at_do_not_move_against_the_others(model, h_eps, seed):
    """Terms of 1 / h_eps round differently in the two forms, by much the same
    for every sample; the step's relative costs must not show by how much."""
    binding = _gpu()
    w = _start_inside(model, h_eps, 1.0, seed)
    S = _step(binding, w, cells=False)["costs"]
    lam = next(v for v in np.geomspace(1e-2, 1e3, 400) if (_softmax(S, v) >= 0.01).sum() >= 5)
    w.params["lambda"] = float(lam)
    direct, cells = _step(binding, w, cells=False), _step(binding, w)
    listed = _softmax(S, lam) >= 0.01
    shift = cells["costs"] - direct["costs"]
    rest = shift[~listed]
    assert np.abs(shift[listed] - np.median(rest)).max() <= 5.0 * rest.std()
