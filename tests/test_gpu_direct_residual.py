"""The direct depth solve refines until its FP64 residual is within the tolerance: smooth, noise-free slopes (whose
surface is largest against the right-hand side, so that FP32 transforms lose most) at lengths up to the longest, thin
grids, and tolerances next to what one or two refinements reach."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu

LIGHTS, ENV = scenes.ring_lights(3, 45.0), np.zeros((1, 2, 2), np.float32)


def _normals(H, W, kind):
    x, y = ((np.arange(W) + 0.5) / W)[None], ((np.arange(H) + 0.5) / H)[:, None]
    gx, gy = np.zeros((H, W)), np.zeros((H, W))
    if kind == "x":
        gx += np.sin(np.pi * x)
    elif kind == "y":
        gy += np.sin(np.pi * y)
    elif kind == "xy":
        gx += 0.6 * np.sin(np.pi * x)
        gy += 0.6 * np.sin(np.pi * y)
    else:
        gx += 0.3
        gy -= 0.2
    return scenes.normals_from_gradient(gx, gy).astype(np.float32)


def _context(lib, H, W, kind, tol):
    opt = lib.irtps_default_options()
    opt.cg_tol = tol
    ctx = lib.Context(H, W, LIGHTS, ENV, opt)
    ctx.set_state(depth=np.zeros((H, W), np.float32), normals=_normals(H, W, kind))
    return ctx


@pytest.mark.parametrize("H,W,kind,tol", [
    (2039, 2039, "xy", 1e-9), (4096, 4096, "xy", 1e-9), (3001, 4001, "xy", 1e-9), (4093, 4093, "tilt", 1e-9),
    (64, 3001, "x", 1e-9), (64, 4096, "x", 1e-9), (4096, 64, "y", 1e-9), (2, 4096, "x", 1e-9), (4093, 3, "y", 1e-9),
    (127, 127, "y", 1e-10), (128, 128, "xy", 1e-10), (128, 2, "y", 1e-10), (512, 512, "xy", 1e-10),
    (1021, 1021, "xy", 1.5e-10)])
def test_smooth_surfaces_reach_the_tolerance(lib, oracle_mod, H, W, kind, tol):
    with _context(lib, H, W, kind, tol) as ctx:
        ctx.integrate()
        d, st = ctx.depth(), ctx.stats()
    assert 0 < st["cg_rel_residual"] <= tol and st["cg_iterations"] == 1, st
    want = oracle_mod.poisson_solve(_normals(H, W, kind).astype(np.float64), 1.0 / W)
    # the stored depth's FP32 rounding; the residual's share is below it: a relative residual of 1e-9 moves a smooth
    # surface, made of the lowest modes, by as little
    assert np.abs(d - want).max() <= 2.0 ** -23 * np.abs(want).max()


def test_tolerance_out_of_reach_is_an_error(lib):
    with _context(lib, 48, 40, "xy", 1e-18) as ctx:
        with pytest.raises(lib.IrtpsError) as e:
            ctx.integrate()
        assert e.value.code == lib.IRTPS_ENUMERIC
        d = ctx.depth()
    with _context(lib, 48, 40, "xy", 1e-9) as ctx:
        ctx.integrate()
        assert np.abs(ctx.depth() - d).max() <= 2.0 ** -22 * np.abs(d).max()


def _photos(H, W):
    """Images of a smooth surface, every row valid."""
    x = ((np.arange(W) + 0.5) / W)[None] + np.zeros((H, 1))
    n = scenes.normals_from_gradient(0.3 * np.sin(np.pi * x), 0 * x)
    return 0.9 * np.einsum("kx,hwx->khw", LIGHTS, n)[:, None].astype(np.float32)


@pytest.mark.parametrize("sizes,tols", [([(4, 4096), (61, 70)], (1e-9, 1e-9)),
                                        ([(64, 3001), (127, 127), (2, 300)], (1e-9, 1e-10, 1e-9))])
def test_batches_reach_the_tolerance(lib, sizes, tols):
    """As alone, bit for bit."""
    single = []
    for (H, W), tol in zip(sizes, tols):
        with _context(lib, H, W, "x", tol) as ctx:
            ctx.set_images(_photos(H, W))
            single.append(ctx.depth())
    ctxs = [_context(lib, H, W, "x", tol) for (H, W), tol in zip(sizes, tols)]
    with lib.Batch(ctxs) as b:
        b.set_images([_photos(H, W) for H, W in sizes])
        got, rel = [c.depth() for c in ctxs], b.stats()["cg_rel_residual"]
    for c in ctxs:
        c.close()
    assert 0 < rel <= max(tols)
    for g, s in zip(got, single):
        assert np.array_equal(g, s)
