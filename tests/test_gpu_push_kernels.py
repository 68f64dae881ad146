"""The push kernels of one shape and the one for any mix: contexts whose mobile
species call for each of them, with a supercell that holds several chunks of
unequal weights (the deposit tile is folded when its term counter or a chunk's
scale asks for it), momenta from rest to 50 mc, and B of either sign around 10,
so that particles turn by anything up to nearly pi in a step (1 + t^2 over
several binades; the kernels' 2 / x and 1 / sqrt(x) by themselves:
test_gpu_quotients.py).  The species drift at 0.3 mc, so that J is large
against one particle's part in it (without a drift the rounding of the fixed-
point sums alone, half a unit of 2^-20 of a chunk's largest term, came to 1e-5 of
max |J|: the weights span two decades).  One step from the read-back state
matches the FP64 oracle at the per-step tolerance of the parity tests."""
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
    from paper_1606_02862_gb300 import workloads as W

    rng = np.random.default_rng(77)
    N = 16
    sp, parts = [], []
    for k, (shape, ec, mobile) in enumerate(MIXES[mix]):
        sp.append(W.SpeciesDef("s%d" % k, -1.0 if k == 0 else 1.0, 1.0, shape, mobile=mobile, ec=ec))
        x = np.concatenate([8.0 + rng.random((1500, 3)) * 4.0, rng.random((300, 3)) * N])
        u = rng.normal(0, 0.1, x.shape) + np.array([0.3 * sp[-1].q, 0.0, 0.0])
        u[::50] *= 0.0
        u[7::50] *= 500.0
        w = 10.0 ** rng.uniform(-4, -2, x.shape[0])
        parts.append((x, u if mobile else np.zeros_like(u), w))
    box = W.BoxInit(N, N, N, particles=parts, E=rng.normal(0, 1e-2, (3, N, N, N)), B=rng.normal(0, 20.0, (3, N, N, N)),
                   rho_bg=0.01)
    wl = W.Workload("push_kernels", W.DT_HALF_COURANT, sp, [box])
    ctx = ctx_from(wl, sc=sc, threads_per_sc=threads)
    try:
        for _ in range(2):
            st, ids = oracle_state_from_gpu(orc, ctx, wl, 0)
            ctx.step(1)
            st.step(1)
            errs = compare_box(st, ids, ctx, wl, 0, tol_field=1e-5, tol_x=1e-5, tol_u=1e-5)
            print(mix, sc, errs)
    finally:
        ctx.close()
