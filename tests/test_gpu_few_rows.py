"""FP64 factorisations whose CTAs hold few rows: eight lanes along the rows up
to 24 rows per CTA, a warp along them beyond (the count of CTAs sets the rows:
576 rows on 72, 64, 36, 24 and 23 CTAs are 8, 9, 16, 24 and 26 each), with one
to three panels and remainders in the last.  At tol = 0 the rounding keeps
every value and leaves every core but the last left-orthonormal: the 1e-12 of
the other FP64 rounding tests."""
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


def check(B, n, ranks, ctas):
    x = synthetic.random_tt_cores(len(ranks) - 1, n, ranks, seed=n + ranks[2] + ctas)
    ctx = B.Context(d=len(ranks) - 1, n=n, nu=0.02, tol=0.0, rank_cap=max(ranks), L=4.0)
    ctx.hopf_set_max_ctas(ctas)
    t = ctx.tt_from_host(x, max_rank=max(ranks))
    ctx.tt_round(t, 0.0, max(ranks), forced_ranks=ranks)
    got = ctx.tt_to_host(t)
    assert tt.diff_norm(got, x) < 1e-12 * tt.norm(x)
    for C in got[:-1]:
        V = tt.V(C)
        assert np.abs(V.conj().T @ V - np.eye(V.shape[1])).max() < 1e-12
    ctx.tt_free(t)
    ctx.close()


@pytest.mark.parametrize("ctas", [72, 64, 36, 24, 23])
@pytest.mark.parametrize("r", [1, 31, 40, 70])
def test_rows_per_cta(B, ctas, r):
    check(B, 24, [1, 24, r, 24, 1], ctas)
