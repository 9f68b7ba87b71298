"""Paths that meet the many-view dRadon/ds precompute with something else than ordinary images of a direct
call: NaN and infinite pixels, which must stay in their view and on the lines that cross them, a degenerate
projection among good ones, and served jobs, whose scratch holds one group of views."""
import time

import numpy as np
import pytest

import synth
from tests import test_gpu_radon_views as views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

W, HH, N_ALPHA, N_S = 300, 260, 512, 400


def _precompute(ctx, P, images, dtype=torch.float32):
    import paper_1806_02637_gb300 as ecc
    return ecc.ecc_precompute_radon_derivative(ctx, torch.from_numpy(P).cuda(), torch.from_numpy(images).cuda(),
                                               N_ALPHA, N_S, dtype=dtype)[0].cpu().numpy()


def _spread(mask):
    """Entries next to one of the mask along s: a line within rounding of a cell's edge may take either cell."""
    out = mask.copy()
    out[..., 1:] |= mask[..., :-1]
    out[..., :-1] |= mask[..., 1:]
    return out


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_pixels_stay_on_their_lines(value):
    import paper_1806_02637_gb300 as ecc
    P, images = views._scan(40, W, HH, 77)
    bad = images.copy()
    spots = {3: [(100, 150)], 17: [(0, 0), (HH - 1, W - 1)], 38: [(130, 40), (131, 41), (20, 299)]}
    for v, at in spots.items():
        for y, x in at:
            bad[v, y, x] = value
    with ecc.Context(0) as ctx:
        clean, S = _precompute(ctx, P, images), _precompute(ctx, P, bad)
        some = sorted(spots)
        by_view = _precompute(ctx, P[some], bad[some])
    others = [v for v in range(40) if v not in spots]
    assert np.array_equal(S[others], clean[others])
    for i, v in enumerate(some):
        many, one = ~np.isfinite(S[v]), ~np.isfinite(by_view[i])
        assert one.any() and not one.all()
        assert not (many & ~_spread(one)).any() and not (one & ~_spread(many)).any()
        assert np.array_equal(S[v][~many], clean[v][~many])


def test_degenerate_view_among_good_ones():
    import paper_1806_02637_gb300 as ecc
    P, images = views._scan(40, W, HH, 78)
    broken = P.copy()
    broken[5] = np.nan
    broken[33, 2] = 0.0
    with ecc.Context(0) as ctx:
        clean = _precompute(ctx, P, images)
        assert ecc.ecc_status(ctx) == 0
        S = _precompute(ctx, broken, images)
        assert ecc.ecc_status(ctx) == 1
        by_view = _precompute(ctx, broken[[5, 33]], images[[5, 33]])
    good = [v for v in range(40) if v not in (5, 33)]
    assert np.array_equal(S[good], clean[good])
    assert np.array_equal(np.isfinite(S[[5, 33]]), np.isfinite(by_view))


@pytest.mark.parametrize("dtype", ["float32", "float16", "bfloat16"])
@pytest.mark.parametrize("n", [26, 70])
def test_served_job_matches_the_direct_calls(n, dtype):
    """The served total against ecc_evaluate on the direct call's sinograms, to the rounding of separately
    compiled copies of the per-sample code (held to 1e-6)."""
    import paper_1806_02637_gb300 as ecc
    P, images = views._scan(n, W, HH, 5 * n)
    cfg = synth.ScanConfig("views", n_views=n, arc_deg=200.0, full_scan=False, W=W, H=HH, pixel_mm=1.0)
    P = synth.trajectory(cfg)
    with ecc.Context(0) as ctx:
        t = ecc.ecc_submit(ctx, P, images, W, HH, N_ALPHA, N_S, 65, n_iters=1, step=0.0, dtype=dtype)
        t0 = time.time()
        while (r := ecc.ecc_poll(ctx, t)) is None:
            assert time.time() - t0 < 60.0
            time.sleep(0.002)
        Pd = torch.from_numpy(P).cuda()
        S, scales = ecc.ecc_precompute_radon_derivative(ctx, Pd, torch.from_numpy(images).cuda(), N_ALPHA, N_S,
                                                        dtype=getattr(torch, dtype))
        total = float(ecc.ecc_evaluate(ctx, Pd, S, W, HH, 65, scales=scales)["total"].cpu()[0])
    assert r["status"] == 0 and r["flags"] == 0
    assert abs(r["total_last"] - total) <= 1e-6 * abs(total)
