"""The plain FP64 push's deposit on the union of the old and the new support:
particles at rest and at offsets on, just below and just above the cell faces
and half-cell lines, moving either way along every axis (so that each axis
in turn takes the window's extra node), across every seam of a box of uneven
edges, with both gathers, against the FP64 oracle: only the order of FP64
operations differs (1e-11 of the largest value, as in the parity tests)."""
import numpy as np
import pytest

from _gpu_helpers import compare_box, ctx_from, oracle_state_from_gpu, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ec", [False, True])
@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("n", [(4, 4, 4), (6, 5, 9)])
def test_crossings(orc, n, shape, ec):
    require_gpu()
    from paper_1606_02862_gb300 import pic
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(7)
    N = np.array(n, dtype=float)
    edge = np.array([0.0, 1e-9, 0.1, 0.5 - 1e-9, 0.5, 0.5 + 1e-9, 0.9, 1.0 - 1e-9])
    x = np.floor(rng.random((600, 3)) * N) + rng.choice(edge, (600, 3))
    u = rng.choice([-1.5, -1e-6, 0.0, 1e-6, 1.5], (600, 3))
    box = W.BoxInit(*n, particles=[(x, u, 0.01 + 0.01 * rng.random(600))],
                    E=rng.normal(0, 1e-2, (3, n[2], n[1], n[0])), B=rng.normal(0, 1e-2, (3, n[2], n[1], n[0])))
    wl = W.Workload("plain_crossings", W.DT_HALF_COURANT, [W.SpeciesDef("e", -1.0, 1.0, shape, ec=ec)], [box])
    ctx = ctx_from(wl, precision=pic.PRECISION_FP64_PLAIN)
    try:
        st, ids = oracle_state_from_gpu(orc, ctx, wl, 0)
        ctx.step(1)
        st.step(1)
        compare_box(st, ids, ctx, wl, 0, tol_field=1e-11, tol_x=1e-11, tol_u=1e-11)
    finally:
        ctx.close()
