"""The Boris rotation of the push kernels over the whole range of its angle: a
uniform B_z from nothing to where 1 + t^2 (t = q B dt / (2 m gamma)) leaves the
normal range of its FP32 reciprocal (2^126) and where it overflows, particles at
rest and with momenta to 30 mc, E = 0, one step.  The momenta match the
textbook rotation in FP64: at most 12 roundings of 2^-24 on terms of at most
2 |u| (1.5e-6 |u|).  Past the overflow 2 / (1 + t^2) is 0, as FP32 division
gives it: the particle goes straight on and the step reports nothing."""
import numpy as np
import pytest

from _gpu_helpers import ctx_from, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [1, 2, 3])
@pytest.mark.parametrize("b", [0.0, 1e-3, 1.0, 7.0, 50.0, 1e4, 1e9, 1e15, 5e19, 1e20, 1.2e20, 1e24])
def test_rotation(shape, b):
    require_gpu()
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(3)
    n = 16
    x = rng.random((400, 3)) * n
    u = rng.normal(0, 1.0, x.shape) * 10.0 ** rng.uniform(-2, 1, (400, 1))
    u[:20] = 0.0
    u = u.astype(np.float32).astype(np.float64)
    B = np.zeros((3, n, n, n))
    B[2] = np.float32(b)
    box = W.BoxInit(n, n, n, particles=[(x, u, np.full(400, 1e-12))], B=B)
    wl = W.Workload("boris_range", W.DT_HALF_COURANT, [W.SpeciesDef("e", -1.0, 1.0, shape)], [box])
    ctx = ctx_from(wl, sc=(8, 4, 4), threads_per_sc=256)
    try:
        ctx.step(1)
        p = ctx.read_particles(0, 0, ids=True)
    finally:
        ctx.close()
    got = p["u"][np.argsort(p["id"])]
    t = -0.5 * wl.dt * np.float64(np.float32(b)) / np.sqrt(1.0 + (u * u).sum(1))
    over = t * t > 2.0 * float(np.finfo(np.float32).max)
    near = (t * t > 0.99 * float(np.finfo(np.float32).max)) & ~over  # either side of the overflow
    assert over.all() if b == 1e24 else not over.any()
    s = np.where(over, 0.0, 2.0 * t / (1.0 + t * t))
    up = u + np.stack([u[:, 1] * t, -u[:, 0] * t, 0.0 * t], 1)
    want = u + np.stack([up[:, 1] * s, -up[:, 0] * s, 0.0 * s], 1)
    err = np.sqrt(((got - want) ** 2).sum(1))
    size = np.sqrt((u * u).sum(1))
    assert np.all(err[~near] <= 1.5e-6 * size[~near]), float(np.max(err[~near] / np.maximum(size[~near], 1e-30)))
    assert np.all(np.abs(np.sqrt((got * got).sum(1)) - size) <= 1.5e-6 * size)
