"""Obstacle values that only the allocation-free step can meet (it reads them
from device memory and cannot check them), in problems where far obstacles
enter through cells: what they mean is what the direct sum makes of them."""
import ctypes as C

import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _static(w, obstacles, shift=0):
    import torch
    from paper_2504_06437_gb300 import binding
    lib = binding.load()
    p, T, x = w.params, int(w.params["T"]), w.x_start
    f64 = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    # the set starts `shift` bytes off a boundary
    d_o = torch.zeros(24 * len(obstacles) + 16, dtype=torch.uint8, device="cuda")
    d_o[shift:shift + 24 * len(obstacles)] = f64(obstacles).view(torch.uint8).flatten()
    d_x, d_r, d_U = f64(x), f64(w.reference(x)), f64(np.zeros((T, 2)))
    d_ctl, d_u0 = f64([p["mu_coarse"], 0.0, 1.0, 0.0, 0.0]), f64(np.zeros(2))
    d_c, params = f64(np.zeros(int(p["K"]))), binding.make_params(p)
    ptr = lambda a: C.c_void_p(a.data_ptr())  # noqa: E731
    rc = lib.mppi_step_static(C.byref(params), C.c_void_p(d_o.data_ptr() + shift), C.c_int32(len(obstacles)), ptr(d_x), ptr(d_r), ptr(d_U),
                              ptr(d_ctl), ptr(d_u0), ptr(d_c), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.mppi_last_error().decode()
    torch.cuda.synchronize()
    return [a.cpu().numpy() for a in (d_c, d_U, d_u0, d_ctl)]


def _world(model, J):
    if model == "unicycle":
        p = W.base_params(W.UNICYCLE, K=16001, T=50, dt=0.05, seed=2)
        x, goal = np.array([1.0, 1.0, 0.7]), np.array([40.0, 40.0, 0.7])
        p["x_goal"] = goal
        return W.World(p, W.obstacle_field(W.rng(2), J, (0, 0), (45, 45), 0.3, 0.8, keep_clear=(x, goal)), x, goal, 1.0)
    w = W.quad2d(2, K=8192, T=40)
    return W.World(w.params, W.obstacle_field(W.rng(3), J, (0, 0), (30, 10), 0.2, 0.6, keep_clear=(w.x_start, w.goal)),
                   w.x_start, w.goal, 1.0)


@pytest.mark.parametrize("model,J", [("unicycle", 200), ("quad2d", 61)])
def test_a_radius_counts_by_its_square(model, J):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = _world(model, J)
    minus = w.obstacles * np.array([1.0, 1.0, -1.0])
    for a, b in zip(_static(w, w.obstacles), _static(w, minus)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("where", [np.inf, -np.inf, 1e25, 1e300])
def test_an_obstacle_out_of_sight_adds_nothing(where):
    """A set padded to a fixed size with obstacles far beyond anything, at 14
    points per lane (one reciprocal per obstacle, which any distance suits)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = _world("quad2d", 61)
    pad = np.concatenate([w.obstacles, np.tile([[where, 0.0, 0.0]], (3, 1))])
    a, b = _static(w, w.obstacles), _static(w, pad)
    assert np.isfinite(b[0]).all()
    assert (np.abs(a[0] - b[0]) <= 2e-5 * np.maximum(np.abs(a[0]), 1.0)).all()


@pytest.mark.parametrize("J", [1, 60, 61])
@pytest.mark.parametrize("shift", [1, 4, 8])
def test_a_set_off_every_boundary_is_copied(J, shift):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = _world("quad2d", J)
    for a, b in zip(_static(w, w.obstacles), _static(w, w.obstacles, shift)):
        assert np.array_equal(a, b)
