"""A small load, some steps (which capture the step's graphs), then a load a
hundred thousand times as large into preset buffers, which nothing reallocates:
the frame maintenance takes no longer than that of a context that was loaded at
once, so no launch of the graphs is left at the size that the first load had."""
import numpy as np
import pytest

from _gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


def _frames_ms(first, n=64, ppc=24):
    from paper_1606_02862_gb300 import pic, workloads as W

    rng = np.random.default_rng(5)
    x = rng.random((n ** 3 * ppc, 3)) * n
    u = rng.normal(0, 0.5, x.shape)
    w = np.full(x.shape[0], 1e-9)
    ctx = pic.Context([(n, n, n)], (1.0, 1.0, 1.0), W.DT_HALF_COURANT, [pic.Species(-1.0, 1.0, 2)], sc=(8, 8, 8),
                      threads_per_sc=256, pool_frames=40000, move_capacity=1 << 23, sort_every=1000)
    try:
        if first:
            ctx.load_particles(0, 0, x[:first], u[:first], w[:first])
            ctx.step(4)
            assert ctx.info(pic.INFO_GRAPH_ACTIVE) == 1
        ctx.load_particles(0, 0, x[first:], u[first:], w[first:])
        ctx.step(4)
        best = np.inf
        for _ in range(5):
            ctx.stage_timing(True)
            ctx.step(4)
            ms, steps = ctx.stage_times()
            best = min(best, ms[1] / steps)
        assert ctx.count_particles(0, 0) == x.shape[0]
        return best
    finally:
        ctx.close()


def test_larger_load_after_capture():
    require_gpu()
    at_once = _frames_ms(0)
    later = _frames_ms(64)
    print("frames ms per step: loaded at once", at_once, "after a small load", later)
    assert later < 1.5 * at_once + 0.02
