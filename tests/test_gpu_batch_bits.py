"""An object of a batch has the results it has alone, whatever objects are beside it."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _photos(lights, H, W):
    x, y = ((np.arange(W) + 0.5) / W)[None], ((np.arange(H) + 0.5) / H)[:, None]
    n = scenes.normals_from_gradient(0.3 * np.sin(np.pi * x) + 0 * y, 0.2 * np.sin(np.pi * y) + 0 * x)
    return 0.9 * np.einsum("kx,hwx->khw", lights, n)[:, None].astype(np.float32)


@pytest.mark.parametrize("beside", [(200, 200, 1e-9), (60, 50, 1e-11)])
def test_direct_solves_keep_their_own_refinements(lib, beside):
    """Small objects beside one whose size or tolerance asks for more refinement steps: the same depth, bit for bit,
    and the same residual (up to the order of its sum), which the steps would lower by a thousand."""
    lights, env = scenes.ring_lights(3, 45.0), np.full((1, 2, 2), 0.1, np.float32)
    small = [(127, 127), (100, 128), (113, 109)]
    sizes = small + [beside[:2]]
    images = [_photos(lights, H, W) for H, W in sizes]

    def context(i):
        opt = lib.irtps_default_options()
        if i == len(small):
            opt.cg_tol = beside[2]
        return lib.Context(*sizes[i], lights, env, opt)

    single = []
    for i in range(len(sizes)):
        with context(i) as ctx:
            ctx.set_images(images[i])
            single.append((ctx.depth(), ctx.stats()["cg_rel_residual"]))
    worst = max(s[1] for s in single)
    assert worst in [s[1] for s in single[:-1]]  # the last object's residual hides none of the others
    ctxs = [context(i) for i in range(len(sizes))]
    with lib.Batch(ctxs) as b:
        b.set_images(images)
        got, rel = [c.depth() for c in ctxs], b.stats()["cg_rel_residual"]
    for c in ctxs:
        c.close()
    assert abs(rel - worst) <= 1e-4 * worst
    for g, s in zip(got, single):
        assert np.array_equal(g, s[0])
