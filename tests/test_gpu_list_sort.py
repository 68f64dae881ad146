"""The sort of the frame lists (TSC, PCS: whole lists in runs of at most 1536
particles, by the frame maintenance; CIC: chunk by chunk in the push): one
supercell holds n particles, n at the edges of a chunk (256), of a run and of
two and three runs, the others a few.  The particles are the same after sorts
on every step (ids, weights), and one step from the read-back state matches
the FP64 oracle at the per-step tolerance of the parity tests."""
import numpy as np
import pytest

from _gpu_helpers import compare_box, ctx_from, oracle_state_from_gpu, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,sc,threads", [(2, (8, 4, 4), 256), (2, (4, 4, 4), 64), (2, (8, 8, 8), 256),
                                              (3, (8, 4, 4), 256), (1, (4, 4, 4), 128)])
@pytest.mark.parametrize("n", [1, 255, 257, 1536, 1537, 3200])
def test_sorted_lists(orc, n, shape, sc, threads):
    require_gpu()
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(100 + n)
    N = 16
    x = np.concatenate([8.0 + rng.random((n, 3)) * np.array([min(sc[0], 8), 4.0, 4.0]),
                        rng.random((40, 3)) * N])
    u = rng.normal(0, 0.1, x.shape)
    w = 0.01 + 0.01 * rng.random(x.shape[0])
    box = W.BoxInit(N, N, N, particles=[(x, u, w)], E=rng.normal(0, 1e-2, (3, N, N, N)), rho_bg=0.01)
    wl = W.Workload("sort_test", W.DT_HALF_COURANT, [W.SpeciesDef("e", -1.0, 1.0, shape)], [box])
    ctx = ctx_from(wl, sc=sc, threads_per_sc=threads, sort_every=1)
    try:
        ctx.step(3)
        p = ctx.read_particles(0, 0, ids=True)
        o = np.argsort(p["id"])
        assert np.array_equal(p["id"][o], np.arange(x.shape[0]))
        assert np.array_equal(p["w"][o], w.astype(np.float32).astype(np.float64))
        st, ids = oracle_state_from_gpu(orc, ctx, wl, 0)
        ctx.step(1)
        st.step(1)
        compare_box(st, ids, ctx, wl, 0, tol_field=1e-5, tol_x=1e-5, tol_u=1e-5)
    finally:
        ctx.close()


def test_resting_lists_are_left_alone(orc):
    """A species at rest beside a fast one, a sort due on every step: the lists
    that nothing joins keep their order, the others are sorted, and both match
    the FP64 oracle over the next step."""
    require_gpu()
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(8)
    N = 16
    xs = [rng.random((900, 3)) * N for _ in range(2)]
    us = [rng.normal(0, 0.5, (900, 3)), np.zeros((900, 3))]
    box = W.BoxInit(N, N, N, particles=[(x, u, np.full(900, 0.01)) for x, u in zip(xs, us)])
    sp = [W.SpeciesDef("e", -1.0, 1.0, 2), W.SpeciesDef("i", 1.0, 1e9, 2)]
    wl = W.Workload("rest_test", W.DT_HALF_COURANT, sp, [box])
    ctx = ctx_from(wl, sc=(8, 4, 4), threads_per_sc=256, sort_every=1)
    try:
        ctx.step(1)
        before = [ctx.read_particles(0, s, ids=True)["id"] for s in range(2)]
        ctx.step(3)
        after = [ctx.read_particles(0, s, ids=True)["id"] for s in range(2)]
        assert np.array_equal(before[1], after[1])
        assert not np.array_equal(before[0], after[0])
        assert np.array_equal(np.sort(after[0]), np.sort(before[0]))
        st, ids = oracle_state_from_gpu(orc, ctx, wl, 0)
        ctx.step(1)
        st.step(1)
        compare_box(st, ids, ctx, wl, 0, tol_field=1e-5, tol_x=1e-5, tol_u=1e-5)
    finally:
        ctx.close()


@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("shape", [2, 3])
def test_arrivals_between_sorts(shape, shift):
    """Particles at rest, and a few that enter the next supercell along y in the
    second step and stay there; a sort is due on the fourth step, in which none
    arrives.  It takes up the lists that they joined (a window shift in between
    moves the lists by a row): every list is in order of its nodes (PCS: cells).
    On the eighth step no list has been joined since, and all keep their order."""
    require_gpu()
    from paper_1606_02862_gb300 import pic, workloads as W

    rng = np.random.default_rng(21)
    N = 16
    sc = (8, 4, 4)
    x = rng.random((1500, 3)) * N
    u = np.zeros_like(x)
    v = 0.2 / W.DT_HALF_COURANT
    x[:60, 1] = 4.0 * rng.integers(1, 4, 60) - 0.3  # past the face in the second step
    u[:60, 1] = v / np.sqrt(1.0 - v * v)
    box = W.BoxInit(N, N, N, particles=[(x, u, np.full(1500, 1e-12))])
    wl = W.Workload("between", W.DT_HALF_COURANT, [W.SpeciesDef("e", -1.0, 1.0, shape)], [box])
    ctx = ctx_from(wl, sc=sc, threads_per_sc=256, sort_every=4)

    def lists():
        p = ctx.read_particles(0, 0, ids=True)
        home = np.floor(p["x"] / np.array(sc)).astype(int)
        g = home[:, 0] + 2 * (home[:, 1] + 4 * home[:, 2])
        node = np.floor(p["x"] + (0.5 if shape == 2 else 0.0)).astype(int) - home * np.array(sc)
        return p["id"], g, node[:, 0] + 9 * (node[:, 1] + 5 * node[:, 2])

    try:
        ctx.step(3)
        if shift:
            ctx.shift_window(0, 4)
        _, g, key = lists()
        assert any(np.any(np.diff(key[g == k]) < 0) for k in range(32))  # arrivals at the lists' ends
        ctx.step(1)
        ids, g, key = lists()
        assert np.all(np.diff(g) >= 0)  # read back list after list
        for k in range(32):
            assert np.all(np.diff(key[g == k]) >= 0), k
        ctx.step(4)
        assert np.array_equal(lists()[0], ids)
        assert ctx.info(pic.INFO_STEPS) == 8
    finally:
        ctx.close()
