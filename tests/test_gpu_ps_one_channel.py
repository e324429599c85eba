"""One channel: masked systems have the same normals and albedo alone and in a batch, bit for bit."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spread", [0.5, 1e-2, 1e-3])
@pytest.mark.parametrize("f16", [False, True])
def test_one_channel_masked_systems(lib, spread, f16):
    """One channel, half of the pixels left with a cluster of lights (condition numbers from 1e1 to 1e6): the
    refined and the FP64 solves give the same normals and albedo alone and in a batch."""
    rng = np.random.default_rng(12)
    H, W, K = 90, 83, 10
    L = scenes.ring_lights(K, 50.0)
    L[:4] = np.array([0.3, 0.2, 0.93]) + spread * rng.normal(size=(4, 3))
    L = L.astype(np.float32)
    n = rng.normal(size=(H, W, 3)) * 0.2 + [0.1, 0.1, 1.0]
    n /= np.linalg.norm(n, axis=-1, keepdims=True)
    A = np.einsum("kx,hwx->khw", L.astype(np.float64), n)[:, None] * rng.uniform(0.5, 0.7, (1, 1, H, W))
    A = np.clip(A, 0.03, 0.97) + rng.normal(0, 1e-3, (K, 1, H, W))
    A[4:, :, : H // 2] = 0.0
    A = A.astype(np.float16 if f16 else np.float32)
    dtype, env = lib.IRTPS_F16 if f16 else lib.IRTPS_F32, np.zeros((1, 2, 2), np.float32)
    with lib.Context(H, W, L, env) as ctx:
        ctx.set_images(A, dtype)
        want = (ctx.normals(), ctx.albedo(), ctx.valid())
    assert want[2].mean() > 0.9
    with lib.Context(H, W, L, env) as ctx, lib.Batch([ctx]) as b:
        b.set_images([A], dtype)
        got = (ctx.normals(), ctx.albedo(), ctx.valid())
    for g, w in zip(got, want):
        assert np.array_equal(g, w)
