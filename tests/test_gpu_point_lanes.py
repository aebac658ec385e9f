"""Point evaluation in every split of the columns over lanes: ranks of each
remainder to 32 columns (1, 2, 3 to 4, 5 to 8, 9 to 16, 17 to 24, 25 to 31, none)
with row vectors shorter and longer than the lanes, largest ranks on either side
of the CTA sizes (4, 8, 24, 48), few points and many; and the moments on either
side of the rule that takes them from points.

Tolerance: d r eps = 7 * 100 * 2.2e-16 = 1.6e-13 of the product of magnitudes:
1e-12 of it, as in the other evaluation tests; the moments' differences are of
the size of the values: 1e-11 of the largest."""
import numpy as np
import pytest

from oracle import tt
import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2403_04946_gb300 import binding, build
    build.build()
    return binding


CASES = [[1, 2, 3, 4, 4, 1], [2, 5, 6, 7, 8, 3], [1, 8, 9, 16, 5, 2], [9, 2, 17, 1, 10, 23], [24, 3, 22, 17, 18, 24],
         [25, 31, 1, 32, 4, 30], [33, 1, 34, 36, 2, 29], [40, 48, 5, 41, 47, 12], [49, 50, 33, 64, 2, 63],
         [66, 70, 1, 81, 96, 95], [97, 100, 3, 66, 99, 98]]


@pytest.mark.parametrize("ranks", CASES, ids=str)
@pytest.mark.parametrize("npts", [1, 304, 700])
def test_points(B, ranks, npts):
    d, n = len(ranks) + 1, 12
    x = synthetic.random_tt_cores(d, n, [1] + ranks + [1], seed=sum(ranks), scale=2.0)
    idx = synthetic.random_probe_indices(d, n, npts, seed=npts)
    ctx = B.Context(d=d, n=n, nu=0.01, tol=1e-9, rank_cap=max(ranks), L=3.0)
    t = ctx.tt_from_host(x)
    got, want = ctx.hopf_eval_points(t, idx), tt.evaluate(x, idx)
    assert np.max(np.abs(got - want)) < 1e-12 * np.max(np.abs(tt.evaluate([np.abs(c) for c in x], idx)))
    ctx.tt_free(t)
    ctx.close()


# 1 + 2 d + 2 d (d - 1) points of d r^2 multiply-adds against 2.4e6, and r against 48
@pytest.mark.parametrize("d,n,ranks", [(4, 6, [6, 48, 6]), (4, 6, [6, 49, 6]), (16, 8, [8] + [16] * 13 + [8]),
                                       (16, 8, [8] + [18] * 13 + [8]), (3, 4, [1, 1]), (20, 10, [9] * 19)])
def test_moments_from_points_and_from_chains(B, d, n, ranks):
    L = 3.0
    x = synthetic.random_tt_cores(d, n, [1] + ranks + [1], seed=d + n + max(ranks), scale=2.0)
    ctx = B.Context(d=d, n=n, nu=0.01, tol=1e-9, rank_cap=max(ranks), L=L)
    t = ctx.tt_from_host(x)
    mean, cov, _ = ctx.hopf_eval_moments(t)
    wmean, wcov = tt.moments(x, n, L, 2.0 * L / n)
    assert np.max(np.abs(mean - wmean)) < 1e-11 * np.max(np.abs(wmean))
    assert np.max(np.abs(cov - wcov)) < 1e-11 * np.max(np.abs(wcov))
    ctx.tt_free(t)
    ctx.close()
