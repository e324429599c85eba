"""Contexts of different sizes on different host threads (one context per thread): what one launch asks of a kernel,
its shared memory above all, must not depend on what another thread's context asked of the same kernel."""
import threading

import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _normals(H, W):
    X, Y = scenes.grid(H, W)
    n = scenes.normals_from_gradient(0.6 * np.sin(7 * X) * np.cos(5 * Y) + 0.4, 0.5 * np.cos(6 * X + 2 * Y) - 0.3)
    n[H // 2:H // 2 + 3, W // 3:W // 3 + 9] = np.array([0.6, 0.0, 0.8])
    return n.astype(np.float32)


def _context(lib, H, W, irls):
    opt = lib.irtps_default_options()
    opt.irls_iters = irls
    ctx = lib.Context(H, W, scenes.ring_lights(3, 45.0), np.zeros((1, 2, 2), np.float32), opt)
    ctx.set_state(depth=np.zeros((H, W), np.float32), normals=_normals(H, W))
    return ctx


def _together(jobs):
    """Runs every job in a thread of its own, all started at once; the exceptions they ended with."""
    gate, errors = threading.Barrier(len(jobs)), []

    def body(job):
        gate.wait()
        try:
            job()
        except Exception as e:  # reported to the caller
            errors.append(e)

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


# robust solves of any two sizes; least-squares solves whose column blocks take more than 48 KB
@pytest.mark.parametrize("irls,sizes,calls", [(1, [(24, 31), (160, 127), (60, 64)], 150),
                                              (0, [(740, 1220), (1030, 1300)], 150)])
def test_contexts_of_two_sizes_on_threads(lib, irls, sizes, calls):
    ctxs = [_context(lib, H, W, irls) for H, W in sizes]
    want = []
    for c in ctxs:
        c.integrate()
        want.append(c.depth())
    got = [None] * len(ctxs)

    def job(i):
        def run():
            for _ in range(calls):
                ctxs[i].integrate()
            got[i] = ctxs[i].depth()
        return run

    errors = _together([job(i) for i in range(len(ctxs))])
    for c in ctxs:
        c.close()
    assert not errors, errors
    for g, w in zip(got, want):
        if irls:  # warm-started from the last surface: the solver's tolerance
            assert np.abs(g - w).max() <= 1e-6 * np.ptp(w)
        else:
            assert np.array_equal(g, w)


def test_batches_of_two_sizes_on_threads(lib):
    opt = lib.irtps_default_options()
    opt.irls_iters = 1
    rs = np.random.default_rng(8)
    lights, env = scenes.ring_lights(3, 45.0), np.full((1, 2, 2), 0.1, np.float32)
    sets = [[(40, 44), (33, 20)], [(150, 251), (64, 90)]]
    images = [[rs.uniform(0.2, 0.6, (3, 1, H, W)).astype(np.float32) for H, W in s] for s in sets]
    ctxs = [[lib.Context(H, W, lights, env, opt) for H, W in s] for s in sets]
    batches = [lib.Batch(c) for c in ctxs]
    want = []
    for b, c, a in zip(batches, ctxs, images):
        b.set_images(a)
        want.append([x.depth() for x in c])

    def job(i):
        def run():
            for _ in range(60):
                batches[i].set_images(images[i])
        return run

    errors = _together([job(0), job(1)])
    got = [[x.depth() for x in c] for c in ctxs] if not errors else None
    for b in batches:
        b.close()
    for c in ctxs:
        for x in c:
            x.close()
    assert not errors, errors
    for g, w in zip(got, want):
        for x, y in zip(g, w):
            assert np.array_equal(x, y)
