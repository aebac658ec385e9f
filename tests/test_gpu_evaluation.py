"""Point and moment evaluation at the edges of their kernels: ranks around the
lanes per column (4 .. 32), ranks that split a chain of the moments over 1 to
8 CTAs, uneven ranks, the smallest tensor.

Tolerances: a value is a product of d vector-matrix products of at most r
terms each, in FP64 in another order than numpy's: d r eps = 9 * 130 * 2.2e-16
= 2.6e-13 of the product of magnitudes; 1e-12 of that product.  The entries
are independent, so the differences behind the moments are as large as the
values: 1e-11 of the largest moment."""
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


def state(d, n, ranks, seed):
    return synthetic.random_tt_cores(d, n, [1] + list(ranks) + [1], seed=seed, scale=2.0)


CASES = [(3, 4, [1, 1]), (3, 8, [2, 7]), (5, 12, [3, 9, 17, 8]), (4, 10, [33, 16, 31]), (6, 8, [5, 64, 65, 32, 4]),
         (3, 6, [130, 97]), (9, 8, [8, 34, 40, 36, 33, 37, 12, 3])]


@pytest.mark.parametrize("d,n,ranks", CASES)
@pytest.mark.parametrize("npts", [1, 400])
def test_points_match_the_oracle(B, d, n, ranks, npts):
    x = state(d, n, ranks, seed=d + n)
    idx = synthetic.random_probe_indices(d, n, npts, seed=npts)
    ctx = B.Context(d=d, n=n, nu=0.01, tol=1e-9, rank_cap=max(ranks), L=3.0)
    t = ctx.tt_from_host(x)
    got = ctx.hopf_eval_points(t, idx)
    want = tt.evaluate(x, idx)
    assert np.max(np.abs(got - want)) < 1e-12 * np.max(np.abs(tt.evaluate([np.abs(c) for c in x], idx)))
    np.testing.assert_array_equal(ctx.hopf_eval_points_noalloc(t, idx), got)
    ctx.tt_free(t)
    ctx.close()


@pytest.mark.parametrize("d,n,ranks", CASES)
def test_moments_match_the_oracle(B, d, n, ranks):
    L = 3.0
    x = state(d, n, ranks, seed=7 * d + n)
    ctx = B.Context(d=d, n=n, nu=0.01, tol=1e-9, rank_cap=max(ranks), L=L)
    t = ctx.tt_from_host(x)
    mean, cov, _ = ctx.hopf_eval_moments(t)
    wmean, wcov = tt.moments(x, n, L, 2.0 * L / n)
    assert np.max(np.abs(mean - wmean)) < 1e-11 * np.max(np.abs(wmean))
    assert np.max(np.abs(cov - wcov)) < 1e-11 * np.max(np.abs(wcov))
    ctx.tt_free(t)
    ctx.close()
