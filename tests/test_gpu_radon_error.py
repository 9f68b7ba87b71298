"""The many-view dRadon/ds precompute is no further from 64 bits than the view-by-view one: both forms
on the same views (a call with a few views is computed view by view), against the FP64 oracle.  White
noise, where every tap counts and the sums do not cancel, and smooth projections; the grids of the
short scan and of the large detector, two thousand steps along a line, and lines less than half a cell
apart."""
import numpy as np
import pytest

from oracle import oracle as orc
from tests import helpers as H
from tests import test_gpu_radon_views as views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _smooth(n, W, Hh, rng):
    x, y = np.arange(W)[None, :] / W, np.arange(Hh)[:, None] / Hh
    out = np.zeros((n, Hh, W), dtype=np.float32)
    for _ in range(6):
        cx, cy = rng.uniform(0.3, 0.7, (2, n, 1, 1))
        rx, ry = rng.uniform(0.05, 0.4, (2, n, 1, 1))
        out += rng.uniform(0.5, 2.0) * np.sqrt(np.maximum(1 - ((x - cx) / rx) ** 2 - ((y - cy) / ry) ** 2, 0))
    return out


@pytest.mark.parametrize("noise", [True, False])
@pytest.mark.parametrize("W,Hh,n_alpha,n_s", [
    (620, 480, 768, 768),
    (976, 976, 1024, 1382),
    (2000, 64, 512, 1700),
    (900, 64, 512, 2000),
])
def test_no_further_from_64_bits_than_view_by_view(W, Hh, n_alpha, n_s, noise):
    import paper_1806_02637_gb300 as ecc
    n, few = 64, 3
    P, images = views._scan(n, W, Hh, 31 * W + Hh)
    if not noise:
        images = _smooth(n, W, Hh, np.random.default_rng(W))
    many = views._precompute(P, images, n_alpha, n_s)[0][:few].cpu().numpy()
    with ecc.Context(0) as ctx:
        ecc.ecc_profile_enable(ctx)
        by_view = ecc.ecc_precompute_radon_derivative(ctx, torch.from_numpy(P[:few]).cuda(),
                                                      torch.from_numpy(images[:few]).cuda(), n_alpha, n_s)[0]
        assert "joseph_kernel" in ecc.ecc_profile_read(ctx)
    ref = orc.radon_derivative(P[:few], images[:few], n_alpha, n_s)
    most = np.abs(ref).max(axis=(1, 2))

    def errors(S):
        e = np.abs(S - ref) / most[:, None, None]
        return e.max(), np.sqrt((e * e).mean())

    m, v = errors(many), errors(by_view.cpu().numpy())
    print(f"{W}x{Hh} {n_alpha}x{n_s} {'noise' if noise else 'smooth'}: max {m[0]:.2e} rms {m[1]:.2e}, "
          f"view by view {v[0]:.2e} {v[1]:.2e}")
    assert m[0] <= v[0] and m[1] <= v[1]
    assert m[0] <= H.TOL_F32
