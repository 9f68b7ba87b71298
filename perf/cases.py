"""Performance cases of the epipolar-consistency library: the calls that its users make, through the
public entry points, over the range of scans that the library is for.

Two kinds of work: the dRadon/ds precompute of a scan's projections ("precompute"), and the consistency of
view pairs on resident sinograms, forward ("evaluate", "noalloc") and with gradients ("grad", "autograd",
"grad_projection").  Projections are analytic cone-beam images of seeded ellipsoids; sinograms are those of
seeded Gaussian blobs in closed form (the derivative of the plane integral) with 1 % noise, so that pairs
are nearly consistent, as on a real scan.  `exact` restates every result in 64 bits in plain torch.
"""
import math

import numpy as np
import torch

import paper_1806_02637_gb300 as ecc

DEV = "cuda:0"
SID, SDD = 750.0, 1200.0
TORCH_TYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def _scan(name, kind, views, arc, W, H, pixel, n_alpha, n_s, dtype="f32", K=0, cauchy=0.0, motion=False, n_list=0):
    return {"name": name, "kind": kind, "views": views, "arc": arc, "W": W, "H": H, "pixel": pixel,
            "n_alpha": n_alpha, "n_s": n_s, "dtype": dtype, "K": K, "cauchy": cauchy, "motion": motion,
            "n_list": n_list}


def listed():
    return [
        # the smallest scan: two views 90 degrees apart on a 256 x 256 detector, as a two-view check sends it
        _scan("precompute_two_views", "precompute", 2, 90.0, 256, 256, 1.0, 256, 363),
        # a mid-size motion-compensation job: the smallest served detector, FP16 sinograms, a ragged view count
        _scan("precompute_job_f16", "precompute", 173, 200.0, 256, 256, 1.4, 256, 363, "f16"),
        # the 200-degree short scan of the paper, every view, FP32: the set-up of every motion estimate
        _scan("precompute_short_scan", "precompute", 496, 200.0, 620, 480, 0.6, 768, 768),
        # a quarter of a 1240-view full scan on the 976 x 976 detector, BF16 sinograms
        _scan("precompute_976_bf16", "precompute", 310, 90.0, 976, 976, 0.3, 1024, 1382, "bf16"),
        # one pair of views: the latency of a single evaluation
        _scan("evaluate_pair", "evaluate", 2, 90.0, 256, 256, 1.0, 256, 363, K=256),
        # all pairs of the short scan: one step of a derivative-free motion estimate
        _scan("evaluate_short_scan", "evaluate", 496, 200.0, 620, 480, 0.6, 768, 768, K=512, motion=True),
        # a full scan on the large detector with FP16 sinograms, 1024 planes and the Cauchy norm
        _scan("evaluate_976_f16", "evaluate", 320, 360.0, 976, 976, 0.3, 1024, 1382, "f16", K=1024, cauchy=0.5),
        # a list of pairs with BF16 sinograms in the allocation-free form, a ragged number of planes
        _scan("noalloc_list_bf16", "noalloc", 61, 200.0, 620, 480, 0.6, 512, 600, "bf16", K=333, n_list=900),
        # the motion gradient of the 248-view scan: one step of a gradient-based estimate
        _scan("grad_248_views", "grad", 248, 200.0, 620, 480, 0.6, 768, 768, K=512, motion=True),
        # the same through torch.autograd on a small FP16 job with a ragged number of planes and the Cauchy norm
        _scan("autograd_job_f16", "autograd", 97, 200.0, 256, 256, 1.4, 256, 363, "f16", K=333, cauchy=0.5,
              motion=True),
        # geometric calibration: the gradient with respect to the projection matrices
        _scan("grad_projection_120", "grad_projection", 120, 200.0, 620, 480, 0.6, 768, 768, K=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["precompute", "precompute", "evaluate", "grad", "autograd", "grad_projection", "noalloc"])
    W, H = _log_int(rng, 160, 976), _log_int(rng, 160, 976)
    n_alpha = _log_int(rng, 180, 1024)
    n_s = int(round(math.hypot(W, H) * rng.uniform(0.8, 1.05)))
    dtype = rng.choice(["f32", "f32", "f16", "bf16"])
    pixel = 350.0 / max(W, H)
    c = _scan("", kind, 2, rng.choice([200.0, 360.0]), W, H, pixel, n_alpha, n_s, dtype)
    del c["name"]
    if kind == "precompute":  # up to the taps of the largest listed scan
        taps = 310 * 1024 * 1382 * 976
        c["views"] = min(_log_int(rng, 2, 500), max(2, int(taps / (n_alpha * n_s * max(W, H)))))
        return c
    c["K"] = _log_int(rng, 65, 1024)
    c["cauchy"] = rng.choice([0.0, 0.5])
    c["motion"] = rng.choice([True, False])
    if kind == "noalloc":
        c["views"] = _log_int(rng, 3, 120)
        c["n_list"] = _log_int(rng, 2, min(3000, 131072 // ((c["K"] + 31) // 32)))
    else:  # up to the samples of the largest listed evaluation, or of the largest gradient
        c["views"] = _log_int(rng, 2, 400 if kind == "evaluate" else 240)
    return c


# ---------------------------------------------------------------- inputs
def _trajectory(c):
    n, W, H = c["views"], c["W"], c["H"]
    i = np.arange(n, dtype=np.float64)
    th = np.deg2rad(i * 360.0 / n) if c["arc"] == 360.0 else np.deg2rad(i * c["arc"] / max(n - 1, 1))
    f = SDD / c["pixel"]
    Kc = np.array([[f, 0, 0.5 * (W - 1)], [0, f, 0.5 * (H - 1)], [0, 0, 1.0]])
    P = np.empty((n, 3, 4))
    for k, t in enumerate(th):
        co, si = math.cos(t), math.sin(t)
        R = np.array([[-si, co, 0.0], [0.0, 0.0, -1.0], [-co, -si, 0.0]])
        P[k] = Kc @ np.hstack([R, -(R @ (SID * np.array([co, si, 0.0])))[:, None]])
    return P


def _field_of_view(c):
    half_w, half_h = 0.5 * c["W"] * c["pixel"], 0.5 * c["H"] * c["pixel"]
    r = SID * math.sin(math.atan(half_w / SDD))
    return 0.9 * r, 0.9 * half_h * (SID - r) / SDD


def _images(c, P, rng):
    """Line integrals of 12 seeded ellipsoids through every pixel centre, FP32 [n, H, W]."""
    n, W, H = c["views"], c["W"], c["H"]
    r, z = _field_of_view(c)
    out = torch.zeros((n, H, W), dtype=torch.float32, device=DEV)
    back = np.linalg.inv(P[:, :, :3])            # pixel -> ray direction
    src = -(back @ P[:, :, 3:])[:, :, 0]
    x = torch.arange(W, dtype=torch.float32, device=DEV)
    y = torch.arange(H, dtype=torch.float32, device=DEV)[:, None]
    step = max(1, (1 << 25) // (W * H))
    for _ in range(12):
        q, _r = np.linalg.qr(rng.standard_normal((3, 3)))
        axes = rng.uniform(0.08, 0.45, 3) * min(r, 2 * z)
        ph, rad = rng.uniform(0, 2 * math.pi), 0.5 * r * math.sqrt(rng.uniform())
        centre = np.array([rad * math.cos(ph), rad * math.sin(ph), rng.uniform(-0.5, 0.5) * z])
        Q = np.diag(1.0 / axes) @ q
        density = rng.uniform(0.1, 1.0) / 25.0
        y0 = (src - centre) @ Q.T                  # source in the unit-sphere frame
        D = Q @ back                               # direction = D (x, y, 1)
        y0t = torch.from_numpy(y0).float().to(DEV)[:, :, None, None]
        Dt = torch.from_numpy(D).float().to(DEV)
        bt = torch.from_numpy(back).float().to(DEV)
        for v in range(0, n, step):
            def ray(m, k):
                return m[v:v + step, k, 0, None, None] * x + m[v:v + step, k, 1, None, None] * y \
                    + m[v:v + step, k, 2, None, None]
            yy = yb = ll = 0.0
            for k in range(3):
                a = ray(Dt, k)
                yy = yy + a * a
                yb = yb + a * y0t[v:v + step, k]
                ll = ll + ray(bt, k) ** 2
            cc = (y0t[v:v + step, :, 0, 0] ** 2).sum(1)[:, None, None] - 1.0
            out[v:v + step] += (2.0 * density) * torch.sqrt(torch.clamp(yb * yb - yy * cc, min=0.0) * ll) / yy
    return out


def _sinograms(c, P, rng, seed):
    """Derivative of the plane integrals of 8 Gaussian blobs on the (alpha, s) grid, 1 % noise, FP32."""
    n, W, H, na, ns = c["views"], c["W"], c["H"], c["n_alpha"], c["n_s"]
    r, z = _field_of_view(c)
    al = np.arange(na) * math.pi / na
    ca, sa = np.cos(al), np.sin(al)
    ds = math.hypot(W, H) / (ns - 1)
    s = torch.from_numpy((np.arange(ns) - 0.5 * (ns - 1)) * ds).float().to(DEV)
    l0 = np.stack([ca, sa, -(0.5 * (W - 1) * ca + 0.5 * (H - 1) * sa)], 1)    # the line at s = 0
    plane = torch.from_numpy(np.einsum("mi,vij->vmj", l0, P)).float().to(DEV)  # [n, na, 4]
    slope = torch.from_numpy(-P[:, 2, :]).float().to(DEV)                     # d plane / d s
    out = torch.zeros((n, na, ns), dtype=torch.float32, device=DEV)
    blobs = []
    for _ in range(8):
        ph, rad = rng.uniform(0, 2 * math.pi), 0.7 * r * math.sqrt(rng.uniform())
        blobs.append((rad * math.cos(ph), rad * math.sin(ph), rng.uniform(-0.7, 0.7) * z, rng.uniform(8.0, 25.0),
                      rng.uniform(0.5, 1.0)))
    step = max(1, (1 << 24) // (na * ns))
    for v in range(0, n, step):
        def at(j):
            return plane[v:v + step, :, j, None] + slope[v:v + step, None, j, None] * s
        nx, ny, nz, off = at(0), at(1), at(2), at(3)
        inv = torch.rsqrt(nx * nx + ny * ny + nz * nz)
        for bx, by, bz, sig, amp in blobs:
            d = (nx * bx + ny * by + nz * bz + off) * inv * (1.0 / sig)
            out[v:v + step] -= amp * d * torch.exp(-0.5 * d * d)
    gen = torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)
    for v in range(0, n, step):
        part = out[v:v + step]
        part += 0.002 * torch.randn(part.shape, generator=gen, device=DEV)
    return out


def _stored(S, dtype):
    """FP32 sinograms as the library stores them, with the per-view scales of FP16 storage."""
    if dtype == "f32":
        return S, None
    if dtype == "bf16":
        return S.bfloat16(), None
    scales = S.abs().amax((1, 2)) / 16384.0
    return (S / scales[:, None, None]).half(), scales


def _inputs(c, seed):
    """The inputs of a case, as a dict of tensors on the GPU."""
    rng = np.random.default_rng([int(seed), c["views"], c["W"]])
    P = _trajectory(c)
    P = P * rng.uniform(0.5, 2.0, (len(P), 1, 1))      # the scale of a projection matrix is arbitrary
    s = {"P": torch.from_numpy(P).to(DEV)}
    if c["kind"] == "precompute":
        s["images"] = _images(c, P, rng)
        return s
    s["motion"] = None
    if c["motion"]:
        th = rng.standard_normal((len(P), 6)) * np.array([0.002] * 3 + [0.5] * 3)
        s["motion"] = torch.from_numpy(th).to(DEV)
    s["pairs"] = None
    if c["n_list"]:
        n, m = c["views"], c["n_list"]
        a = rng.integers(0, n, m)
        b = (a + rng.integers(1, n, m)) % n
        s["pairs"] = torch.from_numpy(np.stack([a, b], 1).astype(np.int32)).to(DEV)
    s["sino"], s["scales"] = _stored(_sinograms(c, P, rng, seed), c["dtype"])
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if case["kind"] != "noalloc":
        s["ctx"] = ecc.Context(0)
    else:
        s["total"] = torch.empty(1, dtype=torch.float64, device=DEV)
        s["per_pair"] = torch.empty((case["n_list"], 2), dtype=torch.float64, device=DEV)
        s["nkappa"] = torch.empty(case["n_list"], dtype=torch.int32, device=DEV)
    return s


def run(s):
    c = s["case"]
    kind, W, H, K = c["kind"], c["W"], c["H"], c["K"]
    if kind == "precompute":
        sino, scales = ecc.ecc_precompute_radon_derivative(s["ctx"], s["P"], s["images"], c["n_alpha"], c["n_s"],
                                                           dtype=TORCH_TYPE[c["dtype"]])
        return {"sino": sino, "scales": scales}
    if kind == "noalloc":
        return ecc.ecc_evaluate_noalloc(s["P"], s["sino"], W, H, K, s["total"], cauchy_c=c["cauchy"],
                                        motion=s["motion"], pairs=s["pairs"], scales=s["scales"],
                                        per_pair=s["per_pair"], nkappa=s["nkappa"])
    if kind == "autograd":
        th = s["motion"] if s["motion"] is not None else torch.zeros((c["views"], 6), dtype=torch.float64, device=DEV)
        th = th.detach().requires_grad_(True)
        total = ecc.consistency(s["ctx"], th, s["P"], s["sino"], W, H, K, cauchy_c=c["cauchy"], scales=s["scales"])
        total.backward()
        return {"total": total.detach(), "grad": th.grad}
    call = {"evaluate": ecc.ecc_evaluate, "grad": ecc.ecc_evaluate_grad,
            "grad_projection": ecc.ecc_evaluate_grad_projection}[kind]
    return call(s["ctx"], s["P"], s["sino"], W, H, K, cauchy_c=c["cauchy"], motion=s["motion"], scales=s["scales"])


def work(c):
    """Each input read once and each output written once; the operations of the definition: per tap of a
    detector line two multiply-adds, per line-pair sample two lines, two bilinear look-ups and the
    square (40), with gradients the slopes and their products with the plane's direction too (100)."""
    n, W, H = c["views"], c["W"], c["H"]
    size = 4 if c["dtype"] == "f32" else 2
    grid = n * c["n_alpha"] * c["n_s"] * size
    if c["kind"] == "precompute":
        # the lines of one direction together cross the detector's area once, at unit steps along one axis
        # and ds / |cos| along the other: about W H / (ds 1.12) taps per view and direction
        ds = math.hypot(W, H) / (c["n_s"] - 1)
        taps = n * c["n_alpha"] * W * H / (1.12 * ds)
        return {"bytes": n * W * H * 4 + grid + n * 96, "flops": 4.0 * taps}
    pairs = c["n_list"] or n * (n - 1) // 2
    samples = float(pairs) * c["K"]
    per = 40.0 if c["kind"] in ("evaluate", "noalloc") else 100.0
    # the sinogram cells that the samples touch, at most the whole sinograms
    touched = min(grid, samples * 2 * 4 * size)
    return {"bytes": touched + n * 144 + pairs * 20, "flops": per * samples}


# ---------------------------------------------------------------- the results in 64 bits
def _views64(P, motion):
    """Moved and normalised projections: M, its cofactor rows, source and up axis."""
    if motion is not None:
        cx, cy, cz = torch.cos(motion[:, 0]), torch.cos(motion[:, 1]), torch.cos(motion[:, 2])
        sx, sy, sz = torch.sin(motion[:, 0]), torch.sin(motion[:, 1]), torch.sin(motion[:, 2])
        R = torch.stack([cz * cy, cz * sy * sx - sz * cx, cz * sy * cx + sz * sx,
                         sz * cy, sz * sy * sx + cz * cx, sz * sy * cx - cz * sx,
                         -sy, cy * sx, cy * cx], 1).reshape(-1, 3, 3)
        P = torch.cat([P[:, :, :3] @ R, P[:, :, :3] @ motion[:, 3:, None] + P[:, :, 3:]], 2)
    M = P[:, :, :3]
    det = torch.linalg.det(M.detach())
    P = P * (torch.sign(det) / torch.linalg.norm(M[:, 2], dim=1).clone())[:, None, None]
    M = P[:, :, :3]
    m1, m2, m3 = M[:, 0], M[:, 1], M[:, 2]
    cof = torch.stack([torch.cross(m2, m3, dim=1), torch.cross(m3, m1, dim=1), torch.cross(m1, m2, dim=1)], 1)
    C = -torch.einsum("vji,vj->vi", cof, P[:, :, 3]) / (m1 * cof[:, 0]).sum(1, keepdim=True)
    up = torch.cross(m3, m1, dim=1)
    return P, cof, C, up / torch.linalg.norm(up, dim=1, keepdim=True)


def _radon64(c, s):
    n, W, H, na, ns = c["views"], c["W"], c["H"], c["n_alpha"], c["n_s"]
    P, _, _, _ = _views64(s["P"], None)
    m1, m2, m3 = P[:, 0, :3], P[:, 1, :3], P[:, 2, :3]
    u0, v0 = (m1 * m3).sum(1), (m2 * m3).sum(1)
    D = torch.sqrt((m1 * m1).sum(1) - u0 * u0)
    ds, cx, cy = math.hypot(W, H) / (ns - 1), 0.5 * (W - 1), 0.5 * (H - 1)
    x = torch.arange(W, dtype=torch.float64, device=DEV)
    y = torch.arange(H, dtype=torch.float64, device=DEV)
    sig = (torch.arange(ns + 1, dtype=torch.float64, device=DEV) - 0.5 * ns) * ds
    sn = (torch.arange(ns, dtype=torch.float64, device=DEV) - 0.5 * (ns - 1)) * ds
    out = torch.empty((n, na, ns), dtype=torch.float32 if n * na * ns > 1 << 28 else torch.float64, device=DEV)
    step = max(1, min(n, (1 << 27) // ((ns + 1) * max(W, H))))
    for v in range(0, n, step):
        u, w, d = u0[v:v + step, None], v0[v:v + step, None], D[v:v + step, None]
        g = s["images"][v:v + step].double()
        g *= d[:, :, None] / torch.sqrt((d * d)[:, :, None] + ((x - u) ** 2)[:, None, :] + ((y - w) ** 2)[:, :, None])
        planes = (torch.nn.functional.pad(g, (1, 2)).flatten(1),
                  torch.nn.functional.pad(g.transpose(1, 2), (1, 2)).flatten(1))
        for m in range(na):
            rows = 4 * m <= na or 4 * m >= 3 * na
            ca, sa = math.cos(m * math.pi / na), math.sin(m * math.pi / na)
            if rows:
                at, top, line = cx + (sig[:, None] - (y - cy) * sa) / ca, W, y
            else:
                at, top, line = cy + (sig[:, None] - (x - cx) * ca) / sa, H, x
            at = at.clamp(-1.0, float(top))     # zero outside the detector
            i = torch.floor(at)
            f = at - i
            k = (line * (top + 3) + 1 + i).long().flatten()
            p = planes[0 if rows else 1]
            t0, t1 = p[:, k], p[:, k + 1]
            t0 += f.flatten() * (t1 - t0)
            rho = t0.reshape(-1, *f.shape).sum(2) / abs(ca if rows else sa)
            spp = sn - (u - cx) * ca - (w - cy) * sa
            out[v:v + step, m] = ((rho[:, 1:] - rho[:, :-1]) / ds * (d * d + spp * spp) / (d * d)).to(out.dtype)
    if c["dtype"] != "f16":
        return {"sino": out, "scales": None}
    scales = out.abs().amax((1, 2)).double() / 16384.0
    return {"sino": out / scales[:, None, None], "scales": scales}


def _arc64(A, X, W, H):
    """Valid arc (lo, len) of each pair in one view; A [p, 3, 2], X corners [4, 3]."""
    q = torch.einsum("ci,pij->pcj", X, A)
    kap = torch.atan2(-q[..., 0], q[..., 1])
    kap = kap - math.pi * torch.floor(kap / math.pi + 0.5)
    kap = torch.sort(kap, dim=1).values
    end = torch.cat([kap[:, 1:], kap[:, :1] + math.pi], 1)
    mid = 0.5 * (kap + end)
    l = torch.einsum("pij,pgj->pgi", A, torch.stack([torch.cos(mid), torch.sin(mid)], 2))
    off = l[..., 0] * 0.5 * (W - 1) + l[..., 1] * 0.5 * (H - 1) + l[..., 2]
    miss = off.abs() > 0.5 * W * l[..., 0].abs() + 0.5 * H * l[..., 1].abs()
    gap = torch.where(miss, end - kap, torch.full_like(kap, -1.0))
    best, g = gap.max(1)
    lo = end.gather(1, g[:, None])[:, 0]
    lo = lo - math.pi * torch.floor(lo / math.pi + 0.5)
    full = best < 0
    return (torch.where(full, torch.full_like(lo, -0.5 * math.pi), lo),
            torch.where(full, torch.full_like(lo, math.pi), math.pi - best))


def _look_up64(flat, view, na, ns, W, H, l):
    """S at the lines l [3][p, K] of the views view [p] (any orientation), and whether they meet the detector."""
    h = torch.sqrt(l[0] * l[0] + l[1] * l[1])
    s = -(l[0] * 0.5 * (W - 1) + l[1] * 0.5 * (H - 1) + l[2]) / h
    hit = s.abs() <= 0.5 * W * (l[0] / h).abs() + 0.5 * H * (l[1] / h).abs()
    al = torch.atan2(l[1], l[0])
    sg = torch.where(al < 0, -1.0, 1.0).double()
    al, s = torch.where(al < 0, al + math.pi, al), s * sg
    over = al >= math.pi
    al, sg, s = torch.where(over, al - math.pi, al), torch.where(over, -sg, sg), torch.where(over, -s, s)
    ia, isn = al * (na / math.pi), s * ((ns - 1) / math.hypot(W, H)) + 0.5 * (ns - 1)
    m, n0 = torch.floor(ia.detach()), torch.floor(isn.detach()).clamp(0, ns - 2)
    fa, fs = ia - m, isn - n0
    m, n0 = m.long().clamp(0, na - 1), n0.long()
    base = view[:, None] * (na * ns)
    i0 = base + m * ns + n0
    wrap = m + 1 >= na
    i1 = torch.where(wrap, base + (ns - 1 - n0), i0 + ns)
    back = torch.where(wrap, -1, 1)
    t0 = flat[i0].double() * (1 - fs) + flat[i0 + 1].double() * fs
    t1 = (flat[i1].double() * (1 - fs) + flat[i1 + back].double() * fs) * back
    return sg * ((1 - fa) * t0 + fa * t1), hit


def _pairs64(c, s, leaf):
    """d, e and (for a gradient) the total's backward pass over chunks of pairs; leaf: motion, P or None."""
    n, W, H, na, ns, K = c["views"], c["W"], c["H"], c["n_alpha"], c["n_s"], c["K"]
    P0, th = s["P"].double(), s["motion"]
    if c["kind"] == "autograd" and th is None:
        th = torch.zeros((n, 6), dtype=torch.float64, device=DEV)
    wrt = None
    if leaf == "motion":
        wrt = th = (th if th is not None else torch.zeros((n, 6), dtype=torch.float64, device=DEV)).requires_grad_(True)
    elif leaf == "P":
        wrt = P0 = P0.clone().requires_grad_(True)
    pairs = s["pairs"].long() if s["pairs"] is not None else torch.triu_indices(n, n, 1, device=DEV).T
    flat = s["sino"].reshape(-1)
    cxy = torch.tensor([[i * W / 2 + 0.5 * (W - 1), j * H / 2 + 0.5 * (H - 1), 1.0] for i in (-1, 1) for j in (-1, 1)],
                       dtype=torch.float64, device=DEV)
    sc = s["scales"].double() if s["scales"] is not None else torch.ones(n, dtype=torch.float64, device=DEV)
    ds_, es_, grad = [], [], None
    step = max(1, (1 << (21 if leaf else 23)) // K)
    ks = (torch.arange(K, dtype=torch.float64, device=DEV) + 0.5) / K
    with torch.set_grad_enabled(leaf is not None):
        for p in range(0, len(pairs), step):
            a, b = pairs[p:p + step, 0], pairs[p:p + step, 1]
            _, cof, C, up = _views64(P0, th)
            base = C[b] - C[a]
            u = base / torch.linalg.norm(base, dim=1, keepdim=True)
            r = up[a] + up[b]
            w = r - (r * u).sum(1, keepdim=True) * u
            w = w / torch.linalg.norm(w, dim=1, keepdim=True)
            F = torch.stack([w, torch.cross(w, u, dim=1)], 2)
            A, B = cof[a] @ F, cof[b] @ F
            with torch.no_grad():
                lo_a, len_a = _arc64(A, cxy, W, H)
                lo_b, len_b = _arc64(B, cxy, W, H)
                first = len_a <= len_b + 1e-9 * torch.maximum(len_a, len_b)
                kap = torch.where(first, lo_a, lo_b)[:, None] + ks * torch.where(first, len_a, len_b)[:, None]
                ck, sk = torch.cos(kap), torch.sin(kap)
            lines = [[L[:, i, 0, None] * ck + L[:, i, 1, None] * sk for i in range(3)] for L in (A, B)]
            Sa, hit_a = _look_up64(flat, a, na, ns, W, H, lines[0])
            Sb, hit_b = _look_up64(flat, b, na, ns, W, H, lines[1])
            ok = hit_a & hit_b
            diff = torch.where(ok, sc[a][:, None] * Sa - sc[b][:, None] * Sb, torch.zeros_like(Sa))
            d = (diff * diff).sum(1) / ok.sum(1).clamp(min=1)
            e = d / (1 + d / c["cauchy"]) if c["cauchy"] > 0 else d
            ds_.append(d.detach())
            es_.append(e.detach())
            if leaf:
                g, = torch.autograd.grad(e.sum(), wrt)
                grad = g if grad is None else grad + g
    d, e = torch.cat(ds_), torch.cat(es_)
    return torch.stack([d, e], 1), e.sum().reshape(1), grad


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "precompute":
        return _radon64(case, s)
    per_pair, total, grad = _pairs64(case, s, {"grad": "motion", "autograd": "motion", "grad_projection": "P"}.get(kind))
    if kind == "autograd":
        return {"total": total[0], "grad": grad}
    out = {"total": total, "per_pair": per_pair, "nkappa": None}
    if kind == "grad":
        out["grad"] = grad
    if kind == "grad_projection":
        out["grad_P"] = grad.reshape(-1, 12)
    return out
