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


@pytest.mark.parametrize("K", [31, 77, 256])
def test_pairs_set_up_by_one_thread_or_by_two(K):
    """Short pair lists are set up by two threads per pair: the results of a pair are those it has among
    all pairs, and an evaluation with the planes kept gives them again."""
    import paper_1806_02637_gb300 as ecc
    import synth
    n, n_alpha, n_s = 160, 64, 90   # 12720 pairs
    cfg = synth.ScanConfig("pairs", n_views=n, arc_deg=200.0, full_scan=False, W=61, H=48, pixel_mm=5.0)
    gen = torch.Generator(device="cuda").manual_seed(K)
    P = torch.from_numpy(synth.trajectory(cfg)).cuda()
    sino = torch.randn((n, n_alpha, n_s), generator=gen, device="cuda")
    motion = 0.01 * torch.randn((n, 6), generator=gen, device="cuda", dtype=torch.float64)
    with ecc.Context(0) as ctx:
        every = ecc.ecc_evaluate(ctx, P, sino, cfg.W, cfg.H, K, motion=motion)
        pairs = torch.triu_indices(n, n, 1, device="cuda").T.contiguous().int()
        order = torch.randperm(len(pairs), generator=gen, device="cuda")
        for count in (1, 15, 16, 17, 9000):
            some = order[:count]
            listed = pairs[some].contiguous()
            a = ecc.ecc_evaluate(ctx, P, sino, cfg.W, cfg.H, K, motion=motion, pairs=listed)
            b = ecc.ecc_evaluate_frozen(ctx, P, sino, cfg.W, cfg.H, K, motion=motion, pairs=listed)
            for r in (a, b):
                assert torch.equal(r["per_pair"], every["per_pair"][some])
                assert torch.equal(r["nkappa"], every["nkappa"][some])
