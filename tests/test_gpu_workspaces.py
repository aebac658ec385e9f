"""Workspaces a context keeps between calls, in the orders a caller may use
them (each result compared with that of a context that saw no other call)."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2403_04946_gb300 import binding, build
    build.build()
    return binding


def test_evaluation_staging_survives_growth_of_the_tensor_core_scratch(B):
    """Points and moments read before and after a mixed rounding that grows
    the tensor-core scratch (a factor of 4096 rows): the evaluation staging
    must stay the context's own."""
    d, n, r = 3, 128, 33
    cores = synthetic.random_tt_cores(d, n, [1, r, r, 1], seed=5)
    idx = synthetic.random_probe_indices(d, n, 40, seed=6)

    def fresh():
        ctx = B.Context(d=d, n=n, nu=0.01, tol=1e-7, rank_cap=r, L=6.0, precision=B.HOPF_MIXED)
        return ctx, ctx.tt_from_host(cores, max_rank=r)

    ctx, t = fresh()
    want = ctx.hopf_eval_points(t, idx)
    want_mean, want_cov, _ = ctx.hopf_eval_moments(t)
    big = ctx.tt_create(6 * r)
    ctx.hopf_apply_op(t, big)
    ctx.tt_round(big, 1e-7, r)
    others = [ctx.tt_create(4) for _ in range(4)]  # would take freed staging over
    for _ in range(2):
        assert np.array_equal(ctx.hopf_eval_points(t, idx), want)
        mean, cov, _ = ctx.hopf_eval_moments(t)
        assert np.array_equal(mean, want_mean) and np.array_equal(cov, want_cov)
    for x in others + [big, t]:
        ctx.tt_free(x)
    ctx.close()
