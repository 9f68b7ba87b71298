"""The per-view geometry and its tangents are worked on by several views (or tangent directions) of a
warp side by side: whatever the number of views, and with a degenerate view among them, a view's own
results are bit for bit the same."""
import pytest

from tests import test_gpu_calibration as cal
from tests import test_gpu_grad as grad

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [2, 3, 4, 5, 8, 9, 19])
@pytest.mark.parametrize("broken", [False, True])
def test_a_view_does_not_depend_on_its_neighbours(n, broken):
    cfg, sc, S = grad._case()

    def run(n, broken):
        P, S32, th = sc["P"][-n:].copy(), S[-n:].astype("float32"), sc["motion"][-n:]
        if broken:
            P[0] = float("nan")
        pairs = [(n - 2, n - 1), (n - 1, n - 2)]
        total, g, per_pair = grad._gpu_grad(P, S32, cfg.W, cfg.H, cfg.K, 0.0, th, pairs)
        total_P, gP = cal._gpu_grad_P(P, S32, cfg.W, cfg.H, cfg.K, 0.0, th, pairs)
        assert total == total_P
        assert not g[:-2].any() and not gP[:-2].any()
        return total, per_pair.tolist(), g[-2:].tolist(), gP[-2:].tolist()

    assert run(n, broken and n > 2) == run(20, False)
