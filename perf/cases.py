"""The work a user of the IRT-PS library has it do, as measurable cases.

Kinds (every one goes through the Python binding of the C ABI):
  trace    one reverted Monte-Carlo trace over a surface estimate (`Context.trace`), per light or
           light-shared, with many samples or the single-sample variant with hole filling
  normals  subtract + photometric stereo of K images given the indirect light (`Context.solve_normals`)
  integrate  normals -> surface (`Context.integrate`)
  classic  iteration 0 from device-resident images (`Context.set_images`): classic photometric stereo
           and its surface, by least squares or by the robust (Huber) integration
  loop     iteration 0 and a few IRT iterations of one object (`set_images` + `iterate`)
  batch    the same for a batch of objects of different sizes (`Batch`)

Scenes are random bumps, dents and bowls with Voronoi albedo, a cosine environment and a jittered ring of
lights, drawn from the seed on the GPU.
"""
import math

import numpy as np
import torch

from paper_1811_02357_gb300 import irtps

DEV = "cuda"


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest job: a 64 x 64 one-channel bowl, 8 lights, three iterations; launches and latency count
        dict(name="loop_bowl_64", kind="loop", H=64, W=64, K=8, C=1, spp=64, bounces=1, iters=3, f16=False),
        # the middle configuration's trace: 512 x 512 RGB, 12 lights, 256 samples, two bounces
        dict(name="trace_512", kind="trace", H=512, W=512, K=12, C=3, spp=256, bounces=2, shared=False, fill=False),
        # the large configuration's trace at a part of its samples and lights
        dict(name="trace_2048", kind="trace", H=2048, W=2048, K=16, C=3, spp=16, bounces=2, shared=False, fill=False),
        # one path per sample for all the lights, with a shadow ray per light at each hit
        dict(name="trace_shared_512", kind="trace", H=512, W=512, K=12, C=3, spp=64, bounces=2, shared=True,
             fill=False),
        # the single-sample variant on a ragged grid: one path per (pixel, light), holes interpolated
        dict(name="trace_single_odd", kind="trace", H=501, W=389, K=12, C=3, spp=1, bounces=2, shared=False,
             fill=True),
        # subtract + photometric stereo, odd pixel count, FP32 images
        dict(name="normals_odd", kind="normals", H=501, W=333, K=12, C=3, f16=False),
        # subtract + photometric stereo of the large configuration: 32 lights, FP16 images
        dict(name="normals_2048", kind="normals", H=2048, W=2048, K=32, C=3, f16=True),
        # surface from normals: the middle configuration, and a ragged one
        dict(name="integrate_512", kind="integrate", H=512, W=512),
        dict(name="integrate_odd", kind="integrate", H=637, W=899),
        # classic photometric stereo of the large configuration (iteration 0 of every job of that size)
        dict(name="classic_2048", kind="classic", H=2048, W=2048, K=32, C=3, f16=True, irls=0),
        # classic photometric stereo with the robust integration (three reweighting steps), ragged
        dict(name="classic_robust", kind="classic", H=375, W=421, K=8, C=3, f16=False, irls=3),
        # a batch of objects of sides 96 to 320, each with its own lights, samples and bounces
        dict(name="batch_12", kind="batch", objects=12, lo=96, hi=320, f16=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["trace", "trace", "trace", "normals", "integrate", "classic", "loop", "batch"])
    if kind == "trace":
        side, ratio = _log(rng, 48, 1500), rng.uniform(0.7, 1.4)
        H, W = side, max(32, int(side * ratio))
        K, bounces = rng.choice([3, 4, 6, 8, 12, 16, 24, 32]), rng.choice([1, 2, 2, 3])
        most = max(1, min(256, int(2.0e8 / (H * W * K * bounces))))
        shared = rng.random() < 0.3
        fill = not shared and rng.random() < 0.25
        spp = 1 if fill else _log(rng, 1, most)
        return dict(kind=kind, H=H, W=W, K=K, C=rng.choice([1, 3, 3]), spp=spp, bounces=bounces, shared=shared,
                    fill=fill)
    if kind == "normals":
        return dict(kind=kind, H=_log(rng, 40, 1800), W=_log(rng, 40, 1800), K=rng.randint(4, 32),
                    C=rng.choice([1, 3, 3]), f16=rng.random() < 0.5)
    if kind == "integrate":
        return dict(kind=kind, H=_log(rng, 32, 1024), W=_log(rng, 32, 1024))
    if kind == "classic":
        robust = rng.random() < 0.3
        top = 500 if robust else 2048
        return dict(kind=kind, H=_log(rng, 64, top), W=_log(rng, 64, top), K=rng.randint(4, 16),
                    C=rng.choice([1, 3]), f16=rng.random() < 0.5, irls=rng.randint(1, 3) if robust else 0)
    if kind == "loop":
        side = _log(rng, 48, 300)
        return dict(kind=kind, H=side, W=max(32, int(side * rng.uniform(0.7, 1.4))), K=rng.choice([8, 12, 16]),
                    C=rng.choice([1, 3]), spp=rng.choice([64, 128, 256]), bounces=rng.choice([1, 2]),
                    iters=rng.randint(1, 3), f16=rng.random() < 0.5)
    return dict(kind=kind, objects=rng.randint(4, 16), lo=_log(rng, 48, 110), hi=_log(rng, 160, 300),
                f16=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
def _scene(seed, H, W, K, C):
    """Depth (H, W), unit normals (3, H, W), albedo (C, H, W) on the GPU in FP64; lights, env on the host."""
    r = np.random.default_rng(seed)
    x = (torch.arange(W, device=DEV, dtype=torch.float64) + 0.5) / W
    y = (torch.arange(H, device=DEV, dtype=torch.float64) + 0.5) / W
    top = H / W
    side = math.sqrt(H * W)
    n_bumps = 20 if side <= 700 else 200
    z = torch.zeros(H, W, device=DEV, dtype=torch.float64)
    zx, zy = torch.zeros_like(z), torch.zeros_like(z)
    for _ in range(n_bumps):
        cx, cy, a, s = r.uniform(0, 1), r.uniform(0, top), r.uniform(-0.15, 0.15), r.uniform(0.02, 0.1)
        ex, ey = torch.exp(-(x - cx) ** 2 / (2 * s * s)), a * torch.exp(-(y - cy) ** 2 / (2 * s * s))
        z.addr_(ey, ex)
        zx.addr_(ey, -ex * (x - cx) / s ** 2)
        zy.addr_(-ey * (y - cy) / s ** 2, ex)
    for _ in range(4):  # spherical-cap bowls, half as deep as their opening radius
        rad = r.uniform(0.05, 0.15)
        R = rad * 1.25
        dx, dy = x - r.uniform(0.15, 0.85), (y - r.uniform(0.15, 0.85) * top)[:, None]
        r2 = dx * dx + dy * dy
        q = torch.sqrt(torch.clamp(R * R - r2, min=1e-12))
        inside = r2 < rad * rad
        z += torch.where(inside, (R - 0.5 * rad) - q, 0.0)
        zx += torch.where(inside, dx / q, 0.0)
        zy += torch.where(inside, dy / q, 0.0)
    n = torch.stack([-zx, -zy, torch.ones_like(z)])
    n /= n.norm(dim=0, keepdim=True)
    best = torch.full((H, W), math.inf, device=DEV, dtype=torch.float64)
    albedo = torch.zeros(C, H, W, device=DEV, dtype=torch.float64)
    for _ in range(16):
        d2 = (x - r.uniform(0, 1)) ** 2 + ((y - r.uniform(0, top)) ** 2)[:, None]
        val = torch.tensor(r.uniform(0.4, 0.9, C), device=DEV)
        closer = d2 < best
        best = torch.where(closer, d2, best)
        albedo = torch.where(closer, val[:, None, None], albedo)
    az = 2 * np.pi * (np.arange(K) + r.uniform(-0.25, 0.25, K)) / K
    el = np.radians(45 + r.uniform(-10, 10, K))
    lights = np.stack([np.cos(el) * np.cos(az), np.cos(el) * np.sin(az), np.sin(el)], 1).astype(np.float32)
    EH, EW = (32, 64) if side <= 700 else (64, 128)
    th = ((np.arange(EH) + 0.5) * np.pi / EH)[:, None]
    ph = (np.arange(EW) + 0.5) * 2 * np.pi / EW
    env = np.full((C, EH, EW), 0.2)
    for _ in range(8):
        f, g, psi, a = r.integers(0, 4), r.integers(0, 4), r.uniform(0, 2 * np.pi), r.uniform(0, 0.1, C)
        env += a[:, None, None] * np.cos(f * th + g * ph + psi)
    return dict(depth=z, normals=n, albedo=albedo, lights=lights, env=np.maximum(env, 0).astype(np.float32))


def _photos(sc, seed, f16):
    """Images of a scene (K, C, H, W) and the indirect light in them: direct light, an indirect part that grows
    with the surface's tilt, and noise."""
    K = len(sc["lights"])
    C, H, W = sc["albedo"].shape
    gen = torch.Generator(device=DEV).manual_seed(seed)
    L = torch.tensor(sc["lights"], device=DEV)
    rho, n = sc["albedo"].float(), sc["normals"].float()
    tilt = 1.0 - n[2]
    images = torch.empty(K, C, H, W, device=DEV, dtype=torch.float16 if f16 else torch.float32)
    lbar = torch.empty(K, C, H, W, device=DEV)
    for k in range(K):
        direct = torch.clamp(n[0] * L[k, 0] + n[1] * L[k, 1] + n[2] * L[k, 2], min=0)
        for c in range(C):
            lbar[k, c] = 0.15 + 0.02 * c + 0.2 * tilt * (1 + 0.3 * L[k, 0] * n[0])
            noise = torch.randn(H, W, device=DEV, generator=gen) * 0.002
            images[k, c] = (rho[c] * (direct + lbar[k, c]) + noise).to(images.dtype)
    return images, lbar


def _host(t):
    return t.float().cpu().numpy()


def _state(sc):
    """The scene as a context's estimate: depth, normals (H, W, 3), albedo on the host."""
    return dict(depth=_host(sc["depth"]), normals=_host(sc["normals"].permute(1, 2, 0).contiguous()),
                albedo=_host(sc["albedo"]))


def _options(case):
    opt = irtps.irtps_default_options()
    opt.sampling = 1 if case.get("shared") else 0
    opt.fill_holes = 1 if case.get("fill") else 0
    opt.irls_iters = case.get("irls", 0)
    return opt


def _empty(*shape, dtype=torch.float32):
    return torch.empty(*shape, device=DEV, dtype=dtype)


def _results(C, H, W):
    return dict(depth=_empty(H, W), normals=_empty(H, W, 4), albedo=_empty(C, H, W))


def _objects(case):
    """Sizes and trace settings of a batch."""
    r = np.random.default_rng(1000 * case["objects"] + case["lo"])
    return [dict(side=int(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]))))),
                 K=int(r.choice([8, 16, 32])), spp=int(r.choice([128, 256])), bounces=int(r.choice([1, 2])))
            for _ in range(case["objects"])]


def _dtype(case):
    return irtps.IRTPS_F16 if case["f16"] else irtps.IRTPS_F32


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed)
    if kind == "batch":
        s["objects"] = _objects(case)
        s["ctx"], s["images"], s["out"] = [], [], []
        for i, o in enumerate(s["objects"]):
            sc = _scene(seed * 64 + i, o["side"], o["side"], o["K"], 3)
            s["ctx"].append(irtps.Context(o["side"], o["side"], sc["lights"], sc["env"]))
            s["images"].append(_photos(sc, seed + i, case["f16"])[0])
            s["out"].append(_results(3, o["side"], o["side"]))
        s["batch"] = irtps.Batch(s["ctx"])
        torch.cuda.synchronize()
        return s
    H, W = case["H"], case["W"]
    K, C = case.get("K", 4), case.get("C", 1)
    sc = _scene(seed, H, W, K, C)
    ctx = s["ctx"] = irtps.Context(H, W, sc["lights"], sc["env"], _options(case))
    if kind == "trace":
        ctx.set_state(**_state(sc))
        s["out"] = dict(indirect=_empty(K, C, H, W))
        if case["fill"]:
            s["out"]["holes"] = _empty(K, H, W, dtype=torch.uint8)
    elif kind == "integrate":
        ctx.set_state(**_state(sc))
        s["out"] = dict(depth=_empty(H, W))
    elif kind == "normals":
        images, lbar = _photos(sc, seed, case["f16"])
        torch.cuda.synchronize()
        ctx.set_images(images, _dtype(case), on_device=True)
        ctx.set_state(albedo=_host(sc["albedo"]))
        ctx.set_indirect(lbar.cpu().numpy())
        s["out"] = dict(_results(C, H, W), valid=_empty(H, W, dtype=torch.uint8))
        del s["out"]["depth"]
    else:  # classic, loop
        s["images"] = _photos(sc, seed, case["f16"])[0]
        s["out"] = dict(_results(C, H, W), valid=_empty(H, W, dtype=torch.uint8))
    torch.cuda.synchronize()
    return s


def run(s):
    case, ctx, out = s["case"], s["ctx"], s["out"]
    kind = case["kind"]
    if kind == "trace":
        ctx.trace(case["spp"], case["bounces"], s["seed"], 0)
        ctx.indirect(out=out["indirect"])
        if case["fill"]:
            ctx.holes(out=out["holes"])
        return out
    if kind == "integrate":
        ctx.integrate()
        ctx.depth(out=out["depth"])
        return out
    if kind == "normals":
        ctx.solve_normals()
        ctx.normals(out=out["normals"])
        ctx.albedo(out=out["albedo"])
        ctx.valid(out=out["valid"])
        return out
    if kind == "batch":
        s["batch"].set_images(s["images"], _dtype(case), on_device=True)
        s["batch"].iterate(1, [o["spp"] for o in s["objects"]], [o["bounces"] for o in s["objects"]], s["seed"])
        for c, o in zip(ctx, out):
            c.depth(out=o["depth"])
            c.normals(out=o["normals"])
            c.albedo(out=o["albedo"])
        return out
    ctx.set_images(s["images"], _dtype(case), on_device=True)
    if kind == "loop":
        ctx.iterate(case["iters"], case["spp"], case["bounces"], s["seed"])
    ctx.depth(out=out["depth"])
    ctx.normals(out=out["normals"])
    ctx.albedo(out=out["albedo"])
    ctx.valid(out=out["valid"])
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _trace_work(P, K, C, spp, bounces, shared=False):
    """Surface, normals and albedo read once, the indirect light written once; per sampled path a direction
    (Philox4x32-10 and a cosine sample: 145 operations) and one environment lookup or hit shading (about 60)."""
    paths = P * spp * (1 if shared else K)
    return dict(bytes=P * (4 + 12 + 4 * C) + 4 * P * K * C, flops=paths * 205)


def _ps_work(P, K, C, f16, indirect):
    """Images (and the indirect light) read once, normals, albedo and validity written once."""
    return dict(bytes=P * (K * C * ((2 if f16 else 4) + (4 if indirect else 0)) + (4 * C if indirect else 0) +
                           16 + 4 * C + 1), flops=P * K * C * (8 if indirect else 6))


def _depth_work(H, W):
    """Normals in, surface out; two fast cosine transforms each way."""
    return dict(bytes=H * W * (16 + 4), flops=H * W * (5 * (math.log2(H) + math.log2(W)) + 12))


def _add(*ws):
    return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        ws = []
        for o in _objects(case):
            P = o["side"] ** 2
            ws += [_trace_work(P, o["K"], 3, o["spp"], o["bounces"]), _ps_work(P, o["K"], 3, case["f16"], False),
                   _ps_work(P, o["K"], 3, case["f16"], True), _depth_work(o["side"], o["side"]),
                   _depth_work(o["side"], o["side"])]
        return _add(*ws)
    H, W = case["H"], case["W"]
    P = H * W
    if kind == "integrate":
        return _depth_work(H, W)
    K, C = case["K"], case["C"]
    if kind == "trace":
        return _trace_work(P, K, C, case["spp"], case["bounces"], case["shared"])
    if kind == "normals":
        return _ps_work(P, K, C, case["f16"], True)
    w = [_ps_work(P, K, C, case["f16"], False)] + [_depth_work(H, W)] * (1 + case.get("irls", 0))
    for _ in range(case.get("iters", 0)):
        w += [_trace_work(P, K, C, case["spp"], case["bounces"]), _ps_work(P, K, C, case["f16"], True),
              _depth_work(H, W)]
    return _add(*w)


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _exact_ps(images, lbar, rho, lights, tau=(0.02, 0.98), cond_max=1e8):
    """Masked least squares per pixel in FP64; the row masks are defined in FP32 (each operation rounded)."""
    K, C, H, W = images.shape
    L = torch.tensor(lights, device=DEV, dtype=torch.float64)
    M = [torch.zeros(H, W, device=DEV, dtype=torch.float64) for _ in range(6)]
    R = torch.zeros(3, C, H, W, device=DEV, dtype=torch.float64)
    rows = torch.zeros(H, W, device=DEV, dtype=torch.int32)
    three = torch.full((H, W), 3.0, device=DEV)
    for k in range(K):
        a = images[k].float()
        f32 = a if lbar is None else a - rho * lbar[k]
        chat = f32[0] if C == 1 else ((f32[0] + f32[1]) + f32[2]) / three
        ok = (chat > tau[0]) & (chat < tau[1])
        exact = a.double() if lbar is None else a.double() - rho.double() * lbar[k].double()
        rows += ok
        w = ok.double()
        for e, (u, v) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
            M[e] += w * (L[k, u] * L[k, v])
        for u in range(3):
            R[u] += (w * L[k, u]) * exact
    m00, m01, m02, m11, m12, m22 = M
    a00, a01, a02 = m11 * m22 - m12 * m12, m02 * m12 - m01 * m22, m01 * m12 - m02 * m11
    a11, a12, a22 = m00 * m22 - m02 * m02, m01 * m02 - m00 * m12, m00 * m11 - m01 * m01
    det = m00 * a00 + m01 * a01 + m02 * a02

    def norm1(b00, b01, b02, b11, b12, b22):
        return torch.maximum(b00.abs() + b01.abs() + b02.abs(), torch.maximum(
            b01.abs() + b11.abs() + b12.abs(), b02.abs() + b12.abs() + b22.abs()))

    cond = norm1(*M) * norm1(a00, a01, a02, a11, a12, a22) / det.abs()
    ok = (rows >= 3) & (det != 0) & (cond <= cond_max)
    G = torch.stack([a00 * R[0] + a01 * R[1] + a02 * R[2], a01 * R[0] + a11 * R[1] + a12 * R[2],
                     a02 * R[0] + a12 * R[1] + a22 * R[2]]) / det
    s = G.sum(1)
    norm = s.norm(dim=0)
    ok &= torch.isfinite(norm) & (norm > 0)
    albedo = torch.where(ok, G.norm(dim=0), 0.0)
    n = torch.where(ok, s / norm, torch.tensor([0.0, 0.0, 1.0], device=DEV, dtype=torch.float64)[:, None, None])
    normals = torch.cat([n, albedo.mean(0, keepdim=True)]).permute(1, 2, 0).contiguous()
    return normals, albedo


def _dct(n):
    i = torch.arange(n, device=DEV, dtype=torch.float64)
    Q = torch.cos(math.pi * i[:, None] * (2 * i + 1) / (2 * n)) * math.sqrt(2.0 / n)
    Q[0] = math.sqrt(1.0 / n)
    return Q, 4 * torch.sin(math.pi * i / (2 * n)) ** 2


def _exact_depth(normals, irls=0, delta=0.05, nz_min=0.05):
    """Least-squares surface of (H, W, >= 3) normals (trapezoidal edge targets, mean 0), then Huber reweighting."""
    n = normals.double()
    H, W = n.shape[:2]
    h = 1.0 / W
    nz = torch.clamp(n[..., 2], min=float(np.float32(nz_min)))
    p, q = -n[..., 0] / nz, -n[..., 1] / nz
    sh, sv = 0.5 * (p[:, 1:] + p[:, :-1]), 0.5 * (q[1:] + q[:-1])  # target slopes of the edges
    (QH, mu), (QW, nu) = _dct(H), _dct(W)
    lam = mu[:, None] + nu
    lam[0, 0] = 1.0

    def div(eh, ev):
        b = torch.zeros(H, W, device=DEV, dtype=torch.float64)
        b[:, 1:] += eh
        b[:, :-1] -= eh
        b[1:] += ev
        b[:-1] -= ev
        return b

    def unit(b):
        t = QH @ b @ QW.T / lam
        t[0, 0] = 0.0
        return QH.T @ t @ QW

    x = unit(div(h * sh, h * sv))
    delta = float(np.float32(delta))
    for _ in range(irls):
        uh, uv = (torch.diff(x, dim=1) / h - sh).abs(), (torch.diff(x, dim=0) / h - sv).abs()
        wh, wv = torch.where(uh <= delta, 1.0, delta / uh), torch.where(uv <= delta, 1.0, delta / uv)

        def A(v):
            return div(wh * torch.diff(v, dim=1), wv * torch.diff(v, dim=0))

        b = div(wh * (h * sh), wv * (h * sv))
        r = b - A(x)
        bn, d, rz = b.norm(), None, None
        for _ in range(400):  # conjugate gradients, preconditioned by the unit-weight solve
            if not r.norm() > 1e-13 * bn:
                break
            z = unit(r)
            new = (r * z).sum()
            d = z if d is None else z + (new / rz) * d
            rz = new
            Ad = A(d)
            a = rz / (d * Ad).sum()
            x = x + a * d
            r = r - a * Ad
    return x - x.mean()


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("normals", "integrate", "classic"):
        return None  # a traced path's decisions have no value in 64 bits
    H, W = case["H"], case["W"]
    sc = _scene(seed, H, W, case.get("K", 4), case.get("C", 1))
    if kind == "integrate":
        return dict(depth=_exact_depth(sc["normals"].permute(1, 2, 0).float()))
    images, lbar = _photos(sc, seed, case["f16"])
    if kind == "normals":
        normals, albedo = _exact_ps(images, lbar, sc["albedo"].float(), sc["lights"])
        return dict(normals=normals, albedo=albedo, valid=None)
    normals, albedo = _exact_ps(images, None, None, sc["lights"])
    return dict(depth=_exact_depth(normals, case["irls"]), normals=normals, albedo=albedo, valid=None)
