"""Obstacles of the allocation-free step: read where the caller keeps them when
a bulk copy can (an even number from a 16-byte boundary), copied first when
not; either way the bits of the context API, and the caller's state and
control written by the step itself."""
import ctypes as C

import numpy as np
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J", [1, 2, 7, 8, 40])
@pytest.mark.parametrize("offset", [0, 1])
def test_static_step_obstacles_in_place_or_copied(J, offset):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    lib = binding.load()
    w = W.quad2d(2, K=333, T=31)
    obs = w.obstacles[:J]
    p, T, x = w.params, 31, w.x_start
    xref = w.reference(x)
    with binding.Controller(p) as g:
        g.set_obstacles(obs)
        for _ in range(2):
            g.step(x, xref)
        u0, U = g.get_control(want_U=True)
        st = g.get_state()
    f64 = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
    block = f64(np.concatenate([np.full(offset, np.nan), obs.ravel()]))  # the set starts 8 bytes off a boundary
    d_x, d_r, d_U = f64(x), f64(xref), f64(np.zeros((T, 2)))
    d_ctl, d_u0 = f64([p["mu_coarse"], 0.0, 1.0, 0.0, 0.0]), f64(np.zeros(2))
    params, ptr = binding.make_params(p), lambda a: C.c_void_p(a.data_ptr())
    for _ in range(2):
        rc = lib.mppi_step_static(C.byref(params), C.c_void_p(block.data_ptr() + 8 * offset), C.c_int32(J), ptr(d_x),
                                  ptr(d_r), ptr(d_U), ptr(d_ctl), ptr(d_u0), None,
                                  C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0, lib.mppi_last_error().decode()
    torch.cuda.synchronize()
    ctl = d_ctl.cpu().numpy()
    assert np.array_equal(d_u0.cpu().numpy(), u0) and np.array_equal(d_U.cpu().numpy(), U)
    assert ctl[0] == st["S_e"] and ctl[1] == st["beta"] and ctl[2] == 0 and ctl[3] == 2 and ctl[4] == 0
