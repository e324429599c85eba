"""Row masks at their bounds: channel sums within a few ulp of 3 tau, where the division by 3 decides; and masked
systems from well to hopelessly conditioned, whose matrices are summed in fixed point."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def _near(rng, tau, shape):
    """Float32 channel triples whose FP32 mean lies within a few ulp of tau."""
    a = (tau * rng.uniform(0.5, 1.5, shape)).astype(np.float32)
    b = (tau * rng.uniform(0.5, 1.5, shape)).astype(np.float32)
    c = (np.float32(3 * tau) - a - b).astype(np.float32)
    steps = rng.integers(-6, 7, shape)
    return a, b, (c.view(np.int32) + steps.astype(np.int32)).view(np.float32)


@pytest.mark.parametrize("tau_lo,tau_hi", [(0.02, 0.98), (0.1, 0.5), (1.0 / 3.0, 0.75)])
def test_row_masks_at_the_bounds(lib, oracle_mod, tau_lo, tau_hi):
    H, W, rng = 37, 53, np.random.default_rng(5)
    A = np.empty((3, 3, H, W), np.float32)
    A[0] = np.stack(_near(rng, tau_lo, (H, W)))
    A[1] = np.stack(_near(rng, tau_hi, (H, W)))
    A[2] = 0.5 * (tau_lo + tau_hi)
    opt = lib.irtps_default_options()
    opt.tau_lo, opt.tau_hi = tau_lo, tau_hi
    with lib.Context(H, W, scenes.ring_lights(3, 45.0), np.zeros((3, 2, 2), np.float32), opt) as ctx:
        ctx.set_images(A)
        got = ctx.valid().astype(bool)
    lo, hi = np.float32(tau_lo), np.float32(tau_hi)
    mean = ((A[:, 0] + A[:, 1]) + A[:, 2]) / np.float32(3.0)
    rows = (mean > lo) & (mean < hi)
    assert 0.2 < rows[0].mean() < 0.8 and 0.2 < rows[1].mean() < 0.8  # both sides of the bounds
    assert np.array_equal(got, rows.all(axis=0))  # three lights: a pixel needs all its rows


@pytest.mark.parametrize("spread", [0.5, 1e-2, 1e-3, 3e-5])
@pytest.mark.parametrize("f16", [False, True])
def test_masked_systems_of_any_condition(lib, oracle_mod, spread, f16):
    """Ten lights, four of them in a cluster of the given spread (condition numbers 1e1 to 1e9 when only the cluster
    stays valid), two far off unit length; whole pixel classes see only the cluster."""
    rng = np.random.default_rng(11)
    H, W, K, C = 23, 41, 10, 3
    L = scenes.ring_lights(K, 50.0)
    base = np.array([0.3, 0.2, 0.93])
    L[:4] = base + spread * rng.normal(size=(4, 3))
    L = L.astype(np.float32)
    n = rng.normal(size=(H, W, 3)) * 0.2 + [0.1, 0.1, 1.0]
    n /= np.linalg.norm(n, axis=-1, keepdims=True)
    A = np.einsum("kx,hwx->khw", L.astype(np.float64), n)[:, None] * rng.uniform(0.5, 0.7, (1, C, H, W))
    A = np.clip(A, 0.03, 0.97) + rng.normal(0, 1e-3, (K, C, H, W))
    A[4:, :, : H // 2] = 0.0  # only the cluster's rows stay valid there
    A = A.astype(np.float16 if f16 else np.float32)
    with lib.Context(H, W, L, np.zeros((C, 2, 2), np.float32)) as ctx:
        ctx.set_images(A, lib.IRTPS_F16 if f16 else lib.IRTPS_F32)
        got, nn, rho = ctx.valid().astype(bool).ravel(), ctx.normals()[..., :3].reshape(-1, 3), ctx.albedo()
    I = A.astype(np.float32).reshape(K, C, -1)
    zero = np.zeros((C, H * W), np.float32)
    rows = oracle_mod.valid_rows(I, zero, np.zeros_like(I))
    # the 64-bit solve; the 1e-3 deg bar of the masked PS tests, and the FP32 output rounding for the albedo
    M = np.einsum("kp,kx,ky->pxy", rows.astype(np.float64), L.astype(np.float64), L.astype(np.float64))
    R = np.einsum("kp,kx,kcp->pcx", rows.astype(np.float64), L.astype(np.float64), I.astype(np.float64))
    with np.errstate(all="ignore"):
        cond = np.array([np.linalg.cond(m, 1) if r >= 3 else np.inf for m, r in zip(M, rows.sum(0))])
    sure = np.abs(np.log(cond / 1e8)) > 1e-6
    want_ok = cond <= 1e8
    assert np.array_equal(got[sure], want_ok[sure])
    ok = got & want_ok
    assert ok.sum() > 100
    G = np.linalg.solve(M[ok], R[ok].transpose(0, 2, 1))
    s = G.sum(-1)
    err = oracle_mod.angular_error_deg(nn[ok], s / np.linalg.norm(s, axis=-1, keepdims=True))
    assert err.max() < 1e-3
    a = np.linalg.norm(G, axis=1)
    assert np.abs(rho.reshape(C, -1).T[ok] - a).max() < 1e-5 * max(1.0, a.max())
