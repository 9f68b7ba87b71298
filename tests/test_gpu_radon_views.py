"""The many-view dRadon/ds precompute against the FP64 oracle at the edges of its tiles: view counts
that leave groups of 32 partly filled, chunks of 16 lines and blocks of alpha rows with remainders,
lines closer together than a cell (both in one) and almost two cells apart (a cell in between),
detectors of either orientation.  The images are white noise, so every tap counts.  The sizes are
those from which the library takes this form (the more views, the smaller the grid)."""
import numpy as np
import pytest

import synth
from oracle import oracle as orc
from tests import helpers as H

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _scan(n, W, Hh, seed):
    cfg = synth.ScanConfig("views", n_views=n, arc_deg=200.0, full_scan=False, W=W, H=Hh, pixel_mm=300.0 / max(W, Hh))
    rng = np.random.default_rng(seed)
    P = synth.trajectory(cfg) * rng.uniform(-2.0, 2.0, (n, 1, 1))
    return P, rng.standard_normal((n, Hh, W)).astype(np.float32)


def _precompute(P, images, n_alpha, n_s, dtype=torch.float32, budget=0):
    import paper_1806_02637_gb300 as ecc
    with ecc.Context(0, hbm_budget_bytes=budget) as ctx:
        ecc.ecc_profile_enable(ctx)
        S, scales = ecc.ecc_precompute_radon_derivative(ctx, torch.from_numpy(P).cuda(),
                                                        torch.from_numpy(images).cuda(), n_alpha, n_s, dtype=dtype)
        assert "radon_views_kernel" in ecc.ecc_profile_read(ctx)
        assert ecc.ecc_status(ctx) == 0
        return S, scales


# the bar of the FP32 precompute (max|dS| <= 1e-5 max|S| per view)
@pytest.mark.parametrize("n,W,Hh,n_alpha,n_s", [
    (26, 300, 260, 512, 400),   # one group, partly filled
    (354, 97, 61, 90, 113),     # eleven groups and two views
    (460, 40, 100, 61, 200),    # line spacing 0.54 .. 0.77 cells: two lines in one cell
    (185, 101, 33, 256, 78),    # line spacing 1.38 .. 1.95 cells
    (351, 31, 30, 160, 44),     # image narrower than a chunk of lines
    (353, 48, 47, 96, 67),      # line spacing 1.00 .. 1.44 cells
    (168, 18, 126, 101, 276),   # eight alpha rows per block
])
def test_many_views_against_oracle(n, W, Hh, n_alpha, n_s):
    P, images = _scan(n, W, Hh, 1000 * n + W)
    S, _ = _precompute(P, images, n_alpha, n_s)
    ref = orc.radon_derivative(P, images, n_alpha, n_s)
    assert H.sino_rel_err(S.cpu().numpy(), ref).max() <= H.TOL_F32
    # a view's values do not depend on the views beside it
    S3, _ = _precompute(P[3:], images[3:], n_alpha, n_s)
    assert torch.equal(S3, S[3:])
    bf, _ = _precompute(P, images, n_alpha, n_s, torch.bfloat16)
    assert torch.equal(bf, S.bfloat16())
    h, scales = _precompute(P, images, n_alpha, n_s, torch.float16)
    want = S.abs().amax((1, 2)) / 16384.0
    assert torch.equal(scales, want)
    assert torch.equal(h, (S / want[:, None, None]).half())


def test_many_views_within_a_budget():
    """Scratch for all groups at once, for one group, and for one axis of one group at a time (in MiB:
    46, 23 and 12 on this grid, and 1 for the rest): the same values."""
    P, images = _scan(40, 300, 260, 5)
    S, _ = _precompute(P, images, 512, 400)
    for budget in (40, 20):
        assert torch.equal(_precompute(P, images, 512, 400, budget=budget << 20)[0], S)
