"""The plane-bounded march against the oracle's plain cell walk, bit for bit, where its parts meet: tile
edges of the pyramid build (32 cells, levels 5 and 6), grids of one cell across, steep and rough surfaces
(planes far from flat), rays along grid lines, and primary rays near their own cell's planes."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _surface(kind, H, W):
    rng = np.random.default_rng(H * 1000 + W)
    x, y = np.meshgrid((np.arange(W) + 0.5) / W, (np.arange(H) + 0.5) / W)
    if kind == "rough":
        z = rng.uniform(-0.2, 0.2, (H, W))
    elif kind == "slope":
        z = 1.5 * x - 2.0 * y + 0.02 * np.sin(40 * x) * np.cos(30 * y)
    else:  # terraces: flat cells beside vertical steps
        z = 0.05 * np.floor(6 * x) - 0.04 * np.floor(5 * y)
    gy, gx = np.gradient(z, 1.0 / W) if min(H, W) > 1 else (np.zeros_like(z), np.zeros_like(z))
    n = np.stack([-gx, -gy, np.ones_like(z)], -1)
    return z.astype(np.float32), (n / np.linalg.norm(n, axis=-1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("H,W", [(2, 2), (2, 66), (33, 34), (65, 33), (34, 129), (97, 66)])
@pytest.mark.parametrize("kind", ["rough", "slope", "terrace"])
def test_march_is_the_cell_walk(lib, oracle_mod, kind, H, W):
    depth, normals = _surface(kind, H, W)
    rng = np.random.default_rng(7)
    albedo = rng.uniform(0.3, 0.9, (1, H, W)).astype(np.float32)
    # two lights in the planes of the axes: their shadow rays have an exact zero in x or y
    lights = np.array([[0.6, 0.0, 0.8], [0.0, -0.8, 0.6], [0.36, 0.48, 0.8]], np.float32)
    env = np.full((1, 2, 4), 0.3, np.float32)
    rays = []
    for _ in range(600):
        i, j = rng.integers(0, H), rng.integers(0, W)
        d = rng.normal(size=3) * [W, W, 0.3]
        d[: 2] *= rng.choice([0.0, 1.0], 2, p=[0.15, 0.85])
        rays.append([j, i, depth[i, j] + 1e-3 / W, *d])
        rays.append([rng.uniform(0, W - 1), i, depth.max() + rng.uniform(-0.2, 0.1), *d])
    rays = np.array(rays, np.float32)
    pix = rng.integers(0, H * W, min(H * W, 400)).astype(np.int32)
    with lib.Context(H, W, lights, env) as ctx:
        ctx.set_state(depth, normals, albedo)
        t, tri = ctx.probe_rays(rays)
        lbar, rec = ctx.trace_pixels(pix, 16, 3, 11, 2, records=True)
        ctx.set_tuning(0, 3)
        assert np.array_equal(ctx.probe_rays(rays)[1], tri)
    t_o, tri_o = oracle_mod.intersect(depth, rays.astype(np.float64), fp32=True, brute=False)
    assert np.array_equal(tri, tri_o)
    hit = tri >= 0
    assert np.array_equal(t[hit], t_o[hit].astype(np.float32))
    want, rec_o, _ = oracle_mod.trace(depth, normals, albedo, lights, env, 16, 3, 11, 2, fp32=True, pixels=pix,
                                      records=True)
    assert np.array_equal(rec, rec_o)
    assert np.abs(lbar - want).max() <= 1e-4 * np.abs(want).max()
