"""The call from pinned host buffers uploads its images pass by pass of the precompute, on a second stream,
behind one event each: with a short first pass and a ragged last one, in the many-view form and view by
view, the total is that of the pageable call, which uploads in one piece."""
import numpy as np
import pytest

from tests import test_gpu_radon_views as views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,W,Hh,n_alpha,n_s,kernel,passes", [
    (300, 300, 260, 512, 400, "weight_views_kernel", 3),   # 32, 128 and 140 views
    (100, 620, 480, 90, 300, "weight_kernel", 3),          # lines too far apart for the form: 38, 38 and 24
])
def test_uploads_in_passes(n, W, Hh, n_alpha, n_s, kernel, passes):
    import paper_1806_02637_gb300 as ecc
    P, images = views._scan(n, W, Hh, n)
    with ecc.Context(0) as ctx:
        want = ecc.ecc_scan_consistency_host(ctx, P, images, n_alpha, n_s, 65)
        pinned = torch.from_numpy(images).pin_memory()
        other = torch.from_numpy(np.random.default_rng(1).standard_normal(images.shape, dtype=np.float32)).pin_memory()
        for _ in range(3):
            ecc.ecc_scan_consistency_host(ctx, P, other, n_alpha, n_s, 65)   # not these images' sinograms
            ecc.ecc_profile_enable(ctx)
            ecc.ecc_profile_read(ctx)
            assert ecc.ecc_scan_consistency_host(ctx, P, pinned, n_alpha, n_s, 65) == want
            assert ecc.ecc_profile_read(ctx)[kernel][0] == passes
            ecc.ecc_profile_enable(ctx, False)
