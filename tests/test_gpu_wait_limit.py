"""A bounded device wait of the many-view precompute that gives up: the kernel ends, the context's
status word says so, and the next call is whole again.  The limit is set to zero, at which a wait gives
up unless its first tries succeed; nothing else of the launch changes."""
import ctypes

import pytest

from tests import test_gpu_radon_views as views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TIMEOUT = 8


def _set_wait_ns(ctx, ns):
    import paper_1806_02637_gb300 as ecc
    f = ecc.load().ecc_internal_set_wait_ns
    f.argtypes = [ctypes.c_void_p, ctypes.c_ulonglong]
    assert f(ctx.handle, ns) == 0


@pytest.mark.parametrize("n,W,Hh,n_alpha,n_s", [
    (40, 300, 260, 512, 400),
    (460, 40, 100, 61, 200),     # lines closer than a cell
])
def test_a_wait_that_gives_up_is_reported_and_the_next_call_is_whole(n, W, Hh, n_alpha, n_s):
    import paper_1806_02637_gb300 as ecc
    P, images = views._scan(n, W, Hh, 17)
    P, images = torch.from_numpy(P).cuda(), torch.from_numpy(images).cuda()
    with ecc.Context(0) as ctx:
        S, _ = ecc.ecc_precompute_radon_derivative(ctx, P, images, n_alpha, n_s)
        assert ecc.ecc_status(ctx) == 0
        for _ in range(3):
            _set_wait_ns(ctx, 0)
            ecc.ecc_precompute_radon_derivative(ctx, P, images, n_alpha, n_s)
            assert ecc.ecc_status(ctx) == TIMEOUT
            _set_wait_ns(ctx, 10 ** 9)
            again, _ = ecc.ecc_precompute_radon_derivative(ctx, P, images, n_alpha, n_s)
            assert ecc.ecc_status(ctx) == 0
            assert torch.equal(again, S)


def test_the_call_from_host_buffers_reports_its_own_wait():
    """ecc_scan_consistency_host is synchronous: a wait that gave up in it is its error, and a bit left by an
    earlier call is not."""
    import paper_1806_02637_gb300 as ecc
    P, images = views._scan(40, 300, 260, 18)
    with ecc.Context(0) as ctx:
        total = ecc.ecc_scan_consistency_host(ctx, P, images, 512, 400, 65)
        _set_wait_ns(ctx, 0)
        with pytest.raises(ecc.EccError, match=r"\(-4\)"):
            ecc.ecc_scan_consistency_host(ctx, P, images, 512, 400, 65)
        _set_wait_ns(ctx, 10 ** 9)
        assert ecc.ecc_scan_consistency_host(ctx, P, images, 512, 400, 65) == total
        assert ecc.ecc_status(ctx) & TIMEOUT
        assert ecc.ecc_status(ctx) == 0
        P[0] = float("nan")   # other bits go on to ecc_status as before
        ecc.ecc_scan_consistency_host(ctx, P, images, 512, 400, 65)
        assert ecc.ecc_status(ctx) & 1
