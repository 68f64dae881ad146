"""The push's work items: the list of supercells that hold mobile particles,
rewritten by every frame maintenance.  Fast particles in an otherwise empty
box (every few steps a supercell empties and another fills), an empty box
and an immobile species beside it, and a moving-window shift, each followed
against the FP64 oracle from a read-back state at the per-step tolerance of
the parity tests."""
import numpy as np
import pytest

from _gpu_helpers import compare_box, ctx_from, oracle_state_from_gpu, require_gpu

pytestmark = pytest.mark.gpu

TOL = dict(tol_field=1e-5, tol_x=1e-5, tol_u=1e-5)


def _sparse(nbox=2):
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(31)
    n = 16
    x = np.array([[0.2, 0.3, 15.9], [15.7, 8.1, 3.95], [7.99, 0.01, 7.9], [4.5, 4.5, 4.5]])
    u = np.array([[-2.0, -1.5, 2.5], [3.0, 0.1, 0.4], [1.0, -3.0, 1.0], [0.0, 0.0, 0.0]])
    ions = W.uniform_in_cells(rng, n, n, n, 1)[::97]
    none = (np.empty((0, 3)), np.empty((0, 3)), np.empty(0))
    still = (ions, np.zeros_like(ions), np.full(ions.shape[0], 0.01))
    E = rng.normal(0, 1e-2, (3, n, n, n))
    boxes = [W.BoxInit(n, n, n, particles=[(x, u, np.full(4, 0.01)), still], E=E)]
    boxes += [W.BoxInit(n, n, n, particles=[none, still], E=E) for _ in range(nbox - 1)]
    sp = [W.SpeciesDef("e", -1.0, 1.0, 2), W.SpeciesDef("frozen", 1.0, 1836.0, 2, mobile=False)]
    return W.Workload("sparse_test", W.DT_HALF_COURANT, sp, boxes)


def test_supercells_empty_and_fill(orc):
    require_gpu()
    wl = _sparse()
    ctx = ctx_from(wl)
    try:
        for _ in range(4):
            ctx.step(4)
            states = [oracle_state_from_gpu(orc, ctx, wl, b) for b in range(2)]
            ctx.step(1)
            for b, (st, ids) in enumerate(states):
                st.step(1)
                compare_box(st, ids, ctx, wl, b, **TOL)
    finally:
        ctx.close()


def test_items_after_a_window_shift(orc):
    require_gpu()
    wl = _sparse(1)
    ctx = ctx_from(wl)
    try:
        ctx.step(2)
        ctx.shift_window(0, 4)
        st, ids = oracle_state_from_gpu(orc, ctx, wl, 0)
        assert 0 < st.species[0].x.shape[0] <= 4
        ctx.step(1)
        st.step(1)
        compare_box(st, ids, ctx, wl, 0, **TOL)
    finally:
        ctx.close()
