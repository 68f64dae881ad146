"""FP64 diagnostics and the charge density of the mixed form for every shape
(CIC, TSC, PCS), two species, particles on cell faces, at half cells and
across every seam of the box, against the FP64 oracle on the state read back.
Both add the same FP64 terms in another order: 1e-12 of the largest."""
import numpy as np
import pytest

from _gpu_helpers import ctx_from, oracle_state_from_gpu, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [1, 2, 3])
@pytest.mark.parametrize("n,sc,threads", [((8, 8, 8), (4, 4, 4), 128), ((24, 12, 16), (8, 4, 4), 256)])
def test_diagnostics_and_rho(orc, shape, n, sc, threads):
    require_gpu()
    from paper_1606_02862_gb300 import pic
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(shape)
    N = np.array(n, dtype=float)
    parts = []
    for _ in range(2):
        x = np.concatenate([rng.random((300, 3)) * N, np.floor(rng.random((60, 3)) * N),
                            np.floor(rng.random((60, 3)) * N) + 0.5, np.zeros((1, 3)), N[None] - 1e-3])
        parts.append((x, rng.normal(0, 0.7, x.shape), 0.01 * rng.random(x.shape[0])))
    box = W.BoxInit(*n, particles=parts, E=rng.normal(0, 1e-2, (3, n[2], n[1], n[0])), rho_bg=0.003)
    sp = [W.SpeciesDef("e", -1.0, 1.0, shape), W.SpeciesDef("p", 1.0, 1836.0, shape, mobile=False)]
    wl = W.Workload("diag_test", W.DT_HALF_COURANT, sp, [box])
    ctx = ctx_from(wl, sc=sc, threads_per_sc=threads)
    try:
        ctx.set_background(0, 0.003)
        st, _ = oracle_state_from_gpu(orc, ctx, wl, 0)
        rho = ctx.read_fields(0, pic.FIELD_RHO)
        ref = st.rho()
        assert np.max(np.abs(rho - ref)) <= 1e-12 * np.max(np.abs(ref))
        got, want = ctx.diagnostics(0), st.diagnostics()
        for k in range(4):
            assert abs(got[k] - want[k]) <= 1e-12 * max(1.0, abs(want[k])), (k, got[k], want[k])
    finally:
        ctx.close()
