"""FP64 roundings whose tall factors take the digit products (2048 rows and
more than 32 columns, or 1024 rows and 64 columns): row counts at the threshold
and between K-chunks, column counts with a remainder in the last panel,
magnitudes graded over the columns, a wide factor through its LQ.

At tol = 0 the rounding keeps every value, so the tensor must come back and
every core but the last must be left-orthonormal.  The products are accurate
to about one unit of FP64 rounding of |A||B| and everything else is FP64:
the bar is the 1e-12 of the other FP64 rounding tests."""
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


@pytest.mark.parametrize("graded", [False, True])
@pytest.mark.parametrize("n,r1,r2", [(64, 33, 32), (64, 64, 33), (66, 100, 37), (130, 97, 64), (64, 50, 31),
                                     (32, 64, 32), (34, 70, 31)])
def test_fp64_rounding_through_the_digit_products(B, n, r1, r2, graded):
    d = 4
    ranks = [1, min(n, r1), r1, r2, 1]
    x = synthetic.random_tt_cores(d, n, ranks, seed=n + r1)
    if graded:
        x[1] = np.asfortranarray(x[1] * np.logspace(0, -10, r1))
        x[2] = np.asfortranarray(x[2] * np.logspace(0, -10, r2))
    ctx = B.Context(d=d, n=n, nu=0.02, tol=0.0, rank_cap=max(ranks), L=4.0)
    t = ctx.tt_from_host(x, max_rank=max(ranks))
    ctx.tt_round(t, 0.0, max(ranks), forced_ranks=ranks)
    got = ctx.tt_to_host(t)
    assert tt.diff_norm(got, x) < 1e-12 * tt.norm(x)
    for C in got[:-1]:
        V = tt.V(C)
        assert np.abs(V.conj().T @ V - np.eye(V.shape[1])).max() < 1e-12
    ctx.tt_free(t)
    ctx.close()


def test_wide_factor_through_its_lq(B):
    """Bond 1 of rank 1100 at n = 80: the first flattening is 80 x 1100, its LQ a
    QR of 1100 x 80."""
    n = 80
    x = synthetic.random_tt_cores(3, n, [1, 1100, 30, 1], seed=2)
    ctx = B.Context(d=3, n=n, nu=0.02, tol=0.0, rank_cap=1100, L=4.0)
    t = ctx.tt_from_host(x, max_rank=1100)
    ctx.tt_round(t, 0.0, 1100, forced_ranks=[1, n, 30, 1])
    got = ctx.tt_to_host(t)
    assert tt.diff_norm(got, x) < 1e-12 * tt.norm(x)
    ctx.tt_free(t)
    ctx.close()


def test_fp64_step_with_digit_products_matches_the_oracle(B):
    """One RK4 step at n = 64, rank 40 (factors of up to 2560 x 240 rows and
    columns, merges and projections included) against the oracle with its
    ranks replayed; the bar of the FP64 step tests."""
    from oracle import model
    d, n, r = 4, 64, 40
    x, _ = synthetic.saturated_tt_cores(d, n, r, seed=3)
    L, nu, dt, tol = 6.0, 0.02, 1e-4, 1e-8
    log = []
    want, _ = tt.rk4_step(x, dt, model.mpo_blocks(d, n, L, nu), model.mpo_bond_dims(d), tol, r, record=log)
    ctx = B.Context(d=d, n=n, nu=nu, tol=tol, rank_cap=r, L=L)
    t = ctx.tt_from_host(x, max_rank=r)
    ctx.hopf_step(t, dt, 1, replay=np.array(log))
    assert tt.diff_norm(ctx.tt_to_host(t), want) < 1e-10 * tt.norm(want)
    ctx.tt_free(t)
    ctx.close()


@pytest.mark.parametrize("where", ["interior", "last"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_value_that_is_not_finite_is_reported(B, where, bad):
    """An infinity or a NaN in a core survives the digit products: the rounding
    reports it (HOPF_ENUMERIC), as it does through FP64 products, and the
    context keeps working."""
    d, n = 4, 64
    ranks = [1, 48, 48, 40, 1]
    x = synthetic.random_tt_cores(d, n, ranks, seed=11)
    ctx = B.Context(d=d, n=n, nu=0.02, tol=1e-10, rank_cap=48, L=4.0)
    y = [c.copy(order="F") for c in x]
    y[1 if where == "interior" else 3][5 % y[3].shape[0], 7, 0] = bad
    t = ctx.tt_from_host(y, max_rank=48)
    with pytest.raises(B.HopfError) as e:
        ctx.tt_round(t, 1e-10, 48)
    assert e.value.status == B.HOPF_ENUMERIC
    ctx.tt_set_from_host(t, cores=x)
    ctx.tt_round(t, 0.0, 48, forced_ranks=ranks)
    assert tt.diff_norm(ctx.tt_to_host(t), x) < 1e-12 * tt.norm(x)
    ctx.tt_free(t)
    ctx.close()
