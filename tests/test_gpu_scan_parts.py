"""The precompute of some views of a scan: told how many views the scan has, it gives the bits of one call
on all of them, whatever the parts; so the ranks of a sharded scan hold the sinograms that one GPU would."""
import pytest

from tests import test_gpu_radon_views as views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _scan(n, W, Hh):
    P, images = views._scan(n, W, Hh, 5 * n + W)
    return torch.from_numpy(P).cuda(), torch.from_numpy(images).cuda()


@pytest.mark.parametrize("n,W,Hh,n_alpha,n_s", [
    (28, 620, 480, 768, 768),    # many views at once from 16 views on
    (26, 300, 260, 512, 400),    # from 23
    (12, 620, 480, 768, 768),    # all view by view
])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
def test_parts_are_those_of_the_whole(n, W, Hh, n_alpha, n_s, dtype):
    import paper_1806_02637_gb300 as ecc
    from paper_1806_02637_gb300 import distributed as D
    P, images = _scan(n, W, Hh)
    with ecc.Context(0) as ctx:
        whole, scales = ecc.ecc_precompute_radon_derivative(ctx, P, images, n_alpha, n_s, dtype=dtype)
        for world in (2, 3, n):
            for b, e in D.view_slices(n, world):
                part, s = ecc.ecc_precompute_radon_derivative(ctx, P[b:e], images[b:e], n_alpha, n_s, dtype=dtype,
                                                              scan_views=n)
                assert torch.equal(part, whole[b:e])
                assert s is None or torch.equal(s, scales[b:e])
        with pytest.raises(ecc.EccError):
            ecc.ecc_precompute_radon_derivative(ctx, P, images, n_alpha, n_s, scan_views=n - 1)


def test_ranks_of_a_sharded_scan(monkeypatch):
    """Each rank's slice as sharded_consistency computes it, the collectives replaced: nothing waits."""
    import paper_1806_02637_gb300 as ecc
    from paper_1806_02637_gb300 import distributed as D
    n, W, Hh, n_alpha, n_s = 28, 620, 480, 768, 768
    P, images = _scan(n, W, Hh)
    with ecc.Context(0) as ctx:
        whole, _ = ecc.ecc_precompute_radon_derivative(ctx, P, images, n_alpha, n_s)
        seen = []

        def gather(local, n_views, world, group=None):
            seen.append(local)
            return whole

        monkeypatch.setattr(D, "all_gather_views", gather)
        monkeypatch.setattr(D, "all_reduce_sum_fp64", lambda total, grad=None, group=None: (total, grad))
        for rank in range(4):
            D.sharded_consistency(ctx, P, images, W, Hh, n_alpha, n_s, 65, rank, 4)
        assert torch.equal(torch.cat(seen), whole)
