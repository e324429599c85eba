"""Weighted (robust) solves whose weights the unit-weight transform does not follow: small Huber thresholds and
outliers, where the solve goes over to the multigrid preconditioner."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu

LIGHTS, ENV = scenes.ring_lights(3, 45.0), np.full((1, 2, 2), 0.1, np.float32)


def _normals(H, W):
    """A smooth surface with one normal in twenty replaced by an outlier."""
    rs = np.random.default_rng(H + 5 * W)
    X, Y = scenes.grid(H, W)
    n = scenes.normals_from_gradient(0.6 * np.sin(7 * X) * np.cos(5 * Y) + 0.4, 0.5 * np.cos(6 * X + 2 * Y) - 0.3)
    out = rs.random((H, W)) < 0.05
    v = rs.normal(size=(int(out.sum()), 3))
    v[:, 2] = np.abs(v[:, 2]) + 0.1
    n[out] = v / np.linalg.norm(v, axis=1, keepdims=True)
    return n.astype(np.float32)


def _options(lib, delta, iters, cap=None):
    opt = lib.irtps_default_options()
    opt.irls_iters, opt.irls_delta = iters, delta
    if cap:
        opt.cg_max_iter = cap
    return opt


@pytest.mark.parametrize("H,W,delta,cap", [(64, 64, 1e-4, None), (64, 64, 1e-6, None), (128, 128, 1e-3, 100),
                                           (33, 70, 1e-3, 100), (130, 97, 1e-4, None), (5, 300, 1e-3, None)])
def test_small_thresholds(lib, oracle_mod, H, W, delta, cap):
    """Within a few hundred iterations (the transform alone takes up to 2000 here), and within an iteration cap that
    the multigrid preconditioner by itself stays below."""
    n = _normals(H, W)
    with lib.Context(H, W, LIGHTS, ENV, _options(lib, delta, 1, cap)) as ctx:
        ctx.set_state(depth=np.zeros((H, W), np.float32), normals=n)
        ctx.integrate()
        d, st = ctx.depth(), ctx.stats()
    assert 0 < st["cg_rel_residual"] <= 1e-9 and st["cg_iterations"] <= 400, st
    want = oracle_mod.irls_solve(n.astype(np.float64), 1.0 / W, float(np.float32(delta)), 1)
    assert np.abs(d - want).max() <= 1e-4 * np.ptp(want)


def test_small_thresholds_in_a_batch(lib):
    """Objects that change the preconditioner beside ones that do not, against each alone."""
    sizes, deltas = [(64, 64), (40, 44), (2, 4100), (33, 70)], [1e-4, 0.5, 1e-3, 1e-3]
    images = [np.clip(np.einsum("kx,hwx->khw", LIGHTS, _normals(H, W)), 0.03, 0.97)[:, None].astype(np.float32)
              for H, W in sizes]
    single = []
    for (H, W), delta, a in zip(sizes, deltas, images):
        with lib.Context(H, W, LIGHTS, ENV, _options(lib, delta, 2)) as ctx:
            ctx.set_images(a)
            single.append(ctx.depth())
    ctxs = [lib.Context(H, W, LIGHTS, ENV, _options(lib, delta, 2)) for (H, W), delta in zip(sizes, deltas)]
    with lib.Batch(ctxs) as b:
        b.set_images(images)
        got, st = [c.depth() for c in ctxs], b.stats()
    for c in ctxs:
        c.close()
    assert 0 < st["cg_rel_residual"] <= 1e-9
    for s, g in zip(single, got):
        assert np.abs(g - s).max() <= 1e-4 * np.ptp(s)
