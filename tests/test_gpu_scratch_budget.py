"""Scratch memory of the precompute: a context with a budget takes every sequence of calls that fits the
budget with the view-by-view form's buffers, a context without one the same on a device with that much
memory left, and the results do not depend on either.  Budgets are swept from the least one upwards, so
that each size of the many-view form's scratch is met with too little left behind it."""
import ctypes

import numpy as np
import pytest

from tests import test_gpu_radon_views as views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N, W, HH, N_ALPHA, N_S, K = 500, 300, 260, 512, 400, 65
MIB = 1 << 20


def _lib():
    import paper_1806_02637_gb300 as ecc
    lib = ecc.load()
    lib.ecc_internal_set_device_limit.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    lib.ecc_internal_held.argtypes = [ctypes.c_void_p]
    lib.ecc_internal_held.restype = ctypes.c_size_t
    return lib


def _by_view_bytes(dtype):
    """View records, line table and weights, weighted images (pairs along rows and along columns, up to
    256 MiB) and FP16 staging of the view-by-view form."""
    vb, pb = ctypes.c_int(), ctypes.c_int()
    _lib().ecc_internal_record_sizes(ctypes.byref(vb), ctypes.byref(pb))
    pad = int(np.ceil(31 * np.hypot(W, HH) / (N_S - 1) * np.sqrt(2) + 8))
    plane = 8 * (HH * (W + 2 * pad) + W * (HH + 2 * pad))
    batch = min(N, 256 * MIB // plane)
    stage = 4 * N_ALPHA * N_S * batch if dtype == torch.float16 else 0
    return N * vb.value + N * (40 * N_ALPHA + 16) + plane * batch + stage


@pytest.fixture(scope="module")
def scan():
    P, images = views._scan(N, W, HH, 11)
    return torch.from_numpy(P).cuda(), torch.from_numpy(images).cuda()


def _calls(ctx, scan, dtype):
    """A precompute and a gradient behind it, as a motion estimate issues them."""
    import paper_1806_02637_gb300 as ecc
    P, images = scan
    S, scales = ecc.ecc_precompute_radon_derivative(ctx, P, images, N_ALPHA, N_S, dtype=dtype)
    g = ecc.ecc_evaluate_grad(ctx, P, S, W, HH, K, scales=scales, want_per_pair=False)
    assert ecc.ecc_status(ctx) == 0
    return S, scales, g["total"], g["grad"]


def _same(a, b):
    return all((x is None and y is None) or torch.equal(x, y) for x, y in zip(a, b))


def _gradient_bytes(scan):
    import paper_1806_02637_gb300 as ecc
    P, images = scan
    S = torch.zeros((N, N_ALPHA, N_S), device="cuda")
    with ecc.Context(0) as ctx:
        ecc.ecc_evaluate_grad(ctx, P, S, W, HH, K, want_per_pair=False)
        torch.cuda.synchronize()
        return _lib().ecc_internal_held(ctx.handle)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("limited", ["budget", "device"])
def test_calls_that_fit_view_by_view_are_taken(scan, dtype, limited):
    import paper_1806_02637_gb300 as ecc
    with ecc.Context(0) as ctx:
        want = _calls(ctx, scan, dtype)
    least = _by_view_bytes(dtype) + _gradient_bytes(scan)
    for room in [least + i * 35 * MIB for i in range(0, 32)] + [least + 4096 * MIB]:
        with ecc.Context(0, hbm_budget_bytes=room if limited == "budget" else 0) as ctx:
            if limited == "device":
                assert _lib().ecc_internal_set_device_limit(ctx.handle, room) == 0
            assert _same(_calls(ctx, scan, dtype), want), room
            assert _lib().ecc_internal_held(ctx.handle) <= room


def test_host_call_that_fits_view_by_view_is_taken(scan):
    import paper_1806_02637_gb300 as ecc
    P, images = scan[0].cpu().numpy(), scan[1].cpu().pin_memory()
    run = lambda ctx: ecc.ecc_scan_consistency_host(ctx, P, images, N_ALPHA, N_S, K)
    with ecc.Context(0) as ctx:
        want = run(ctx)
    with ecc.Context(0) as ctx:   # the evaluation's own scratch
        ecc.ecc_evaluate(ctx, scan[0], torch.zeros((N, N_ALPHA, N_S), device="cuda"), W, HH, K, want_per_pair=False)
        torch.cuda.synchronize()
        evaluation = _lib().ecc_internal_held(ctx.handle)
    least = _by_view_bytes(torch.float32) + evaluation + N * (96 + 4 * W * HH + 4 * N_ALPHA * N_S) + 8
    for room in [least + i * 50 * MIB for i in range(0, 16)]:
        with ecc.Context(0, hbm_budget_bytes=room) as ctx:
            assert run(ctx) == want, room


def test_scratch_without_a_budget_is_bounded(scan):
    """FP16 staging counts towards the many-view form's scratch."""
    import paper_1806_02637_gb300 as ecc
    P, images = scan
    with ecc.Context(0) as ctx:
        for dtype in (torch.float16, torch.bfloat16, torch.float32):
            ecc.ecc_precompute_radon_derivative(ctx, P, images, N_ALPHA, N_S, dtype=dtype)
            torch.cuda.synchronize()
            assert _lib().ecc_internal_held(ctx.handle) <= (1152 + 16) * MIB


def test_many_small_and_many_large_calls_in_one_budget(scan):
    """Buffers only grow: whatever the order of storage types, the budget that holds the largest
    view-by-view buffers of all of them holds the calls."""
    import paper_1806_02637_gb300 as ecc
    P, images = scan
    room = _by_view_bytes(torch.float16)
    for order in ((torch.float32, torch.float16), (torch.float16, torch.float32, torch.float16)):
        with ecc.Context(0, hbm_budget_bytes=room) as ctx:
            for n in (3, 40, N):
                for dtype in order:
                    ecc.ecc_precompute_radon_derivative(ctx, P[:n], images[:n], N_ALPHA, N_S, dtype=dtype)
            assert ecc.ecc_status(ctx) == 0


def test_fp16_short_scan_in_every_budget_from_the_least():
    """The 496-view short scan in FP16: line sums and staging of one group take more than 256 MiB here."""
    import paper_1806_02637_gb300 as ecc
    import synth
    c = synth.CONFIGS["c2"]
    images = torch.randn((c.n_views, c.H, c.W), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    P = torch.from_numpy(synth.trajectory(c)).cuda()
    out = torch.empty((c.n_views, c.n_alpha, c.n_s), dtype=torch.float16, device="cuda")
    with ecc.Context(0) as ctx:
        want, scales = ecc.ecc_precompute_radon_derivative(ctx, P, images, c.n_alpha, c.n_s, dtype=out.dtype)
    for room in range(390 * MIB, 1200 * MIB, 35 * MIB):   # 376 MiB view by view
        with ecc.Context(0, hbm_budget_bytes=room) as ctx:
            S, s = ecc.ecc_precompute_radon_derivative(ctx, P, images, c.n_alpha, c.n_s, dtype=out.dtype, out=out)
            assert torch.equal(S, want) and torch.equal(s, scales), room
