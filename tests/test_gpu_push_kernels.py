"""The push kernels of one shape and the one for any mix: contexts whose mobile
species call for each of them, with a supercell that holds several chunks of
unequal weights (the deposit tile is folded when its term counter or a chunk's
scale asks for it) and momenta from rest to 50 mc (the kernels' own 1/sqrt and
1/x).  One step from the read-back state matches the FP64 oracle at the
per-step tolerance of the parity tests, J also within the rounding of its
fixed-point sums: a chunk's terms stay below 2^21 units, their largest (at most
a weight at the speed of light) above 2^20, so each of n terms of a node is off
by at most h = max(w) 2^-21, and their sum by 5 h sqrt(n / 3) at five standard
deviations.  (At 1e-5 alone PCS failed at 1.0e-5 to 1.3e-5 of max |J|: with
weights over two decades the largest term is large against J.)"""
import numpy as np
import pytest

from _gpu_helpers import compare_box, ctx_from, oracle_state_from_gpu, require_gpu

pytestmark = pytest.mark.gpu

# (shape, energy-conserving, mobile) of each species
MIXES = {"cic": [(1, False, True)], "tsc": [(2, False, True)], "pcs": [(3, False, True)],
         "tsc+frozen cic": [(2, False, True), (1, False, False)],
         "cic+frozen pcs": [(1, False, True), (3, False, False)],
         "cic+tsc": [(1, False, True), (2, False, True)],
         "tsc+pcs": [(2, False, True), (3, False, True)],
         "tsc ec": [(2, True, True)]}


@pytest.mark.parametrize("sc,threads", [((8, 4, 4), 256), ((4, 4, 4), 128)])
@pytest.mark.parametrize("mix", list(MIXES))
def test_one_step(orc, mix, sc, threads):
    require_gpu()
    from paper_1606_02862_gb300 import pic, workloads as W

    rng = np.random.default_rng(77)
    N = 16
    sp, parts = [], []
    for k, (shape, ec, mobile) in enumerate(MIXES[mix]):
        sp.append(W.SpeciesDef("s%d" % k, -1.0 if k == 0 else 1.0, 1.0, shape, mobile=mobile, ec=ec))
        x = np.concatenate([8.0 + rng.random((1500, 3)) * 4.0, rng.random((300, 3)) * N])
        u = rng.normal(0, 0.1, x.shape)
        u[::50] *= 0.0
        u[7::50] *= 500.0
        w = 10.0 ** rng.uniform(-4, -2, x.shape[0])
        parts.append((x, u if mobile else np.zeros_like(u), w))
    box = W.BoxInit(N, N, N, particles=parts, E=rng.normal(0, 1e-2, (3, N, N, N)), rho_bg=0.01)
    wl = W.Workload("push_kernels", W.DT_HALF_COURANT, sp, [box])
    ctx = ctx_from(wl, sc=sc, threads_per_sc=threads)
    try:
        for _ in range(2):
            st, ids = oracle_state_from_gpu(orc, ctx, wl, 0)
            ctx.step(1)
            st.step(1)
            compare_box(st, ids, ctx, wl, 0, tol_field=1e-5, tol_x=1e-5, tol_u=1e-5, check_j=False)
            J = ctx.read_fields(0, pic.FIELD_J)
            rounding = sum(5.0 * p[2].max() * 2.0 ** -21 * np.sqrt(p[0].shape[0] / 3.0) for p in parts)
            assert np.max(np.abs(J - st.J)) <= 1e-5 * np.max(np.abs(st.J)) + rounding
    finally:
        ctx.close()
