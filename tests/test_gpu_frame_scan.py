"""Frame maintenance at the edge between its one-block scan (at most 4096
lists) and the three-kernel one: 1024 supercells with 1, 4 (4096 lists) and 5
species, fast particles that change supercell on every step.  Particles keep
their ids, and a step from the read-back state matches the FP64 oracle."""
import numpy as np
import pytest

from _gpu_helpers import compare_box, ctx_from, oracle_state_from_gpu, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("species", [1, 4, 5])
def test_scan(orc, species):
    require_gpu()
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(species)
    n = (64, 64, 16)
    parts, sp = [], []
    for s in range(species):
        x = rng.random((900, 3)) * np.array(n, dtype=float)
        parts.append((x, rng.normal(0, 2.0, x.shape), np.full(900, 0.01)))
        sp.append(W.SpeciesDef(f"s{s}", -1.0 if s % 2 else 1.0, 1.0 + s, 2))
    box = W.BoxInit(*n, particles=parts, E=rng.normal(0, 1e-2, (3, n[2], n[1], n[0])))
    wl = W.Workload("scan_test", W.DT_HALF_COURANT, sp, [box])
    ctx = ctx_from(wl)
    try:
        ctx.step(5)
        st, ids = oracle_state_from_gpu(orc, ctx, wl, 0)
        assert all(np.array_equal(i, np.arange(900)) for i in ids)
        ctx.step(1)
        st.step(1)
        compare_box(st, ids, ctx, wl, 0, tol_field=1e-5, tol_x=1e-5, tol_u=1e-5)
    finally:
        ctx.close()
