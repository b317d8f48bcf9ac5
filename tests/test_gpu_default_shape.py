"""The launch shape that the library takes when the caller leaves it open:
problems of up to 96 samples per SM run in one wave, also at the sizes where
the tile is rounded or has to leave room for obstacles, and a small problem
with long chains of points gets tiles of its own."""
import pytest

from paper_2504_06437_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _shape(p):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_06437_gb300 import binding
    with binding.Controller(p) as g:
        t = g.tiling()
    return t, torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("per_sm", [7, 12, 16, 20, 28, 31, 32, 33, 48, 56, 62, 63, 64, 65, 84, 93, 95, 96])
@pytest.mark.parametrize("more", [-1, 0])
def test_one_wave(per_sm, more):
    _, sms = _shape(W.unicycle_small(0).params)
    K = per_sm * sms + more
    t, sms = _shape(dict(W.unicycle_small(0).params, K=K, T=20))
    ctas = 1 if t["threads"] == 512 else 2 if K <= 64 * sms else 3
    assert t["n_ctas"] <= ctas * sms


@pytest.mark.parametrize("K", [1200, 3300, 4000, 4864])
def test_long_horizons_keep_one_wave_beside_the_largest_set(K):
    t, sms = _shape(dict(W.unicycle_small(0).params, K=K, T=256))
    assert t["n_ctas"] <= (1 if t["threads"] == 512 else 2) * sms


@pytest.mark.parametrize("K", [1, 3, 115, 700])
def test_small_problems(K):
    short, sms = _shape(W.quad2d(0, K=K, T=20).params)
    long_, _ = _shape(W.quad2d(0, K=K, T=200).params)
    assert (short["samples_per_cta"], short["threads"]) == (min(K, 5), 256)
    assert (long_["samples_per_cta"], long_["threads"]) == (-(-K // sms), 512)
