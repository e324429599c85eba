"""Small objects: the samples of a (pixel, light) item are spread over several lanes and summed in sample order, so
no bit may depend on whether a launch was large enough to go unsplit."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _ctx(lib, sc, lights, fill=0):
    opt = lib.irtps_default_options()
    opt.fill_holes = fill
    ctx = lib.Context(sc.H, sc.W, lights, sc.env, opt)
    ctx.set_state(sc.depth, sc.normals, sc.albedo)
    return ctx


@pytest.mark.parametrize("C", [1, 3])
@pytest.mark.parametrize("spp,fill", [(3, 0), (4, 1), (7, 0), (33, 0)])
def test_split_and_unsplit_agree_bit_for_bit(lib, C, spp, fill):
    sc = scenes.mixed(71, 97, 101, K=64, C=C)  # 64 lights: 627 k items, unsplit; 3 lights: 29 k, split
    got = []
    for K in (3, 64):
        with _ctx(lib, sc, sc.lights[:K], fill) as ctx:
            ctx.trace(spp, 2, 9, 1)
            got.append((ctx.indirect()[:3], ctx.holes()[:3] if fill else None))
    assert got[0][0].any() and np.array_equal(got[0][0], got[1][0])
    if fill:
        assert got[0][1].any() and np.array_equal(got[0][1], got[1][1])


def test_long_pixel_lists_are_not_split(lib):
    """A list may name a pixel many times: 600 k items of a 32 x 32 object, whose own trace is split."""
    sc = scenes.mixed(72, 32, 32, K=3, C=3)
    pix = np.random.default_rng(1).integers(0, 32 * 32, 200_000).astype(np.int32)
    with _ctx(lib, sc, sc.lights) as ctx:
        ctx.trace(16, 1, 5, 0)
        whole = ctx.indirect().reshape(3, 3, -1)
        listed = ctx.trace_pixels(pix, 16, 1, 5, 0)[0].reshape(3, 3, -1)
    assert np.array_equal(listed, whole[:, :, pix])


def test_batch_splits_within_its_room(lib):
    """Four objects of 79 MB of sample radiances each: the first three are split, the last is not."""
    scs = [scenes.mixed(73 + i, 100, 101, K=16, C=1) for i in range(4)]
    rng = np.random.default_rng(2)
    A = [rng.uniform(0.1, 0.9, (16, 1, 100, 101)).astype(np.float32) for _ in scs]
    ctxs = [lib.Context(sc.H, sc.W, sc.lights, sc.env) for sc in scs]
    try:
        for c, a in zip(ctxs, A):
            c.set_images(a)
        with lib.Batch(ctxs) as b:
            b.iterate(1, [128] * 4, [1] * 4, 3)
        got = [c.indirect() for c in ctxs]
    finally:
        for c in ctxs:
            c.close()
    for i, sc in enumerate(scs):
        with lib.Context(sc.H, sc.W, sc.lights, sc.env) as c:
            c.set_object(i)
            c.set_images(A[i])
            c.iterate(1, 128, 1, 3)
            assert np.array_equal(got[i], c.indirect()), i
