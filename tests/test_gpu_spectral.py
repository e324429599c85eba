"""The direct depth solve (fast cosine transforms in FP32, refined with FP64 residuals) at the lengths where its
parts meet: every radix, chirp-convolution (prime) lengths, one- to eight-column blocks, odd row and column
counts, the longest lines; and a batch that mixes direct and iterative solves."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _normals(H, W):
    rs = np.random.default_rng(H + 5 * W)
    X, Y = scenes.grid(H, W)
    gx = 0.6 * np.sin(7 * X) * np.cos(5 * Y) + rs.normal(0, 0.05, (H, W)) + 0.4
    gy = 0.5 * np.cos(6 * X + 2 * Y) + rs.normal(0, 0.05, (H, W)) - 0.3
    return scenes.normals_from_gradient(gx, gy).astype(np.float32)


def _context(lib, H, W):
    ctx = lib.Context(H, W, scenes.ring_lights(3, 45.0), np.zeros((1, 2, 2), np.float32))
    ctx.set_state(depth=np.zeros((H, W), np.float32), normals=_normals(H, W))
    return ctx


@pytest.mark.parametrize("H,W", [(2, 3), (3, 2), (7, 5), (11, 13), (49, 27), (31, 97), (121, 250), (63, 640),
                                 (1031, 64), (90, 2047), (1500, 1201), (4096, 3), (3, 4093)])
def test_direct_solve(lib, oracle_mod, H, W):
    with _context(lib, H, W) as ctx:
        ctx.integrate()
        d, st = ctx.depth(), ctx.stats()
        ctx.integrate()
        assert np.array_equal(ctx.depth(), d)  # no dependence on the current depth, no run-to-run change
    want = oracle_mod.poisson_solve(_normals(H, W).astype(np.float64), 1.0 / W)
    # the stored depth's FP32 rounding (2^-24 of the largest value), and the refined solve well below it
    assert np.abs(d - want).max() <= 2.0 ** -23 * np.abs(want).max()
    assert st["cg_iterations"] == 1 and st["cg_rel_residual"] <= 1e-10, st


def test_batch_mixes_direct_and_iterative(lib):
    sizes = [(40, 44), (2, 4100), (33, 70)]
    rs = np.random.default_rng(3)
    images = [rs.uniform(0.2, 0.6, (3, 1, H, W)).astype(np.float32) for H, W in sizes]
    lights, env = scenes.ring_lights(3, 45.0), np.full((1, 2, 2), 0.1, np.float32)
    single = []
    for (H, W), a in zip(sizes, images):
        with lib.Context(H, W, lights, env) as ctx:
            ctx.set_images(a)
            single.append((ctx.depth(), ctx.stats()["cg_iterations"]))
    ctxs = [lib.Context(H, W, lights, env) for H, W in sizes]
    with lib.Batch(ctxs) as b:
        b.set_images(images)
        got = [c.depth() for c in ctxs]
    for c in ctxs:
        c.close()
    assert [s[1] == 1 for s in single] == [True, False, True]
    for i in (0, 2):
        assert np.array_equal(got[i], single[i][0])
    assert np.abs(got[1] - single[1][0]).max() <= 1e-4 * np.ptp(single[1][0])


@pytest.mark.parametrize("H,W,iters", [(97, 101, 2), (256, 130, 3), (3, 700, 2)])
def test_weighted_solve_spectral_preconditioner(lib, oracle_mod, H, W, iters):
    """Robust integration whose weighted solves are preconditioned by the transform, alone and in a batch beside a
    grid it does not cover, against the oracle's weighted solves (the bar of every weighted solve test)."""
    n = _normals(H, W)
    n[H // 2:H // 2 + 3, W // 3:W // 3 + 9] = np.array([0.6, 0.0, 0.8], np.float32)
    opt = lib.irtps_default_options()
    opt.irls_iters = iters
    with lib.Context(H, W, scenes.ring_lights(3, 45.0), np.zeros((1, 2, 2), np.float32), opt) as ctx:
        ctx.set_state(depth=np.zeros((H, W), np.float32), normals=n)
        ctx.integrate()
        d, st = ctx.depth(), ctx.stats()
    want = oracle_mod.irls_solve(n.astype(np.float64), 1.0 / W, 0.05, iters)
    assert st["cg_rel_residual"] <= 1e-9 and st["cg_iterations"] <= 60, st
    assert np.abs(d - want).max() <= 1e-4 * np.ptp(want)


def test_weighted_batch_mixes_preconditioners(lib):
    sizes = [(40, 44), (2, 4100), (33, 70)]
    rs = np.random.default_rng(4)
    images = [rs.uniform(0.2, 0.6, (3, 1, H, W)).astype(np.float32) for H, W in sizes]
    lights, env = scenes.ring_lights(3, 45.0), np.full((1, 2, 2), 0.1, np.float32)
    opt = lib.irtps_default_options()
    opt.irls_iters = 2
    single = []
    for (H, W), a in zip(sizes, images):
        with lib.Context(H, W, lights, env, opt) as ctx:
            ctx.set_images(a)
            single.append(ctx.depth())
    ctxs = [lib.Context(H, W, lights, env, opt) for H, W in sizes]
    with lib.Batch(ctxs) as b:
        b.set_images(images)
        got = [c.depth() for c in ctxs]
    for c in ctxs:
        c.close()
    for s, g in zip(single, got):
        assert np.abs(g - s).max() <= 1e-4 * np.ptp(s)


@pytest.mark.parametrize("precond", [0, 1, 2])
@pytest.mark.parametrize("every,tol", [(1, 1e-9), (2, 1e-6), (7, 1e-9), (1000, 1e-9), (1000, 1e-3)])
def test_refresh_rules_of_weighted_solves(lib, oracle_mod, precond, every, tol):
    """Whenever the residual is refreshed (every so many iterations, or when the FP32 recursion says so), a solve ends
    on an FP64 residual within its tolerance; at 1e-9 the surface is the oracle's."""
    H, W = 61, 53
    n = _normals(H, W)
    n[20:24, 10:30] = np.array([0.6, 0.0, 0.8], np.float32)
    opt = lib.irtps_default_options()
    opt.irls_iters, opt.precond, opt.cg_check_every, opt.cg_tol = 2, precond, every, tol
    with lib.Context(H, W, scenes.ring_lights(3, 45.0), np.zeros((1, 2, 2), np.float32), opt) as ctx:
        ctx.set_state(depth=np.zeros((H, W), np.float32), normals=n)
        ctx.integrate()
        d, st = ctx.depth(), ctx.stats()
    assert 0 < st["cg_rel_residual"] <= tol
    if tol == 1e-9:
        want = oracle_mod.irls_solve(n.astype(np.float64), 1.0 / W, 0.05, 2)
        assert np.abs(d - want).max() <= 1e-4 * np.ptp(want)
