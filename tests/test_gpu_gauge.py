"""FP64 contexts do not depend on the gauge of a bond: a tensor with D on one
side of a bond and 1 / D on the other is the same tensor.  D are powers of two
(exact, so the inputs agree to the last bit of their product) over up to 16
decades, growing, falling or mixed along the bond, on one bond or on all; the
factors are tall enough for the digit products (1024 rows and 64 columns, 2048
and 33), whose merges contract over that bond.

Tolerance: the rounding at tol = 0 is backward stable against |A||B|, which the
gauge leaves as it is: the 1e-12 of the other FP64 rounding tests; a step's
result moves by its roundings' tolerance of 1e-12 at most eight times: 1e-10 as
in the FP64 step tests."""
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


def gauge(cores, kind, decades, bonds, rng):
    out = [c.copy() for c in cores]
    for k in bonds:
        r = out[k].shape[0]
        u = np.arange(r) / max(r - 1, 1)
        e = {"grow": u, "fall": -u, "mixed": rng.random(r) - 0.5}[kind] * decades
        D = 2.0 ** np.round(e / np.log10(2.0))
        out[k - 1] = out[k - 1] * D
        out[k] = out[k] / D[:, None, None]
    return [np.asfortranarray(c) for c in out]


@pytest.mark.parametrize("kind,decades,bonds", [("grow", 0, [2]), ("grow", 8, [2]), ("fall", 12, [2]), ("mixed", 16, [2]),
                                                ("grow", 12, [1, 2, 3]), ("mixed", 14, [1, 2, 3])])
@pytest.mark.parametrize("n,ranks", [(64, [1, 48, 64, 40, 1]), (66, [1, 40, 130, 35, 1])])
def test_rounding_does_not_see_the_gauge(B, n, ranks, kind, decades, bonds):
    x = synthetic.random_tt_cores(4, n, ranks, seed=n)
    y = gauge(x, kind, decades, bonds, np.random.default_rng(1))
    ctx = B.Context(d=4, n=n, nu=0.02, tol=0.0, rank_cap=max(ranks), L=4.0)
    t = ctx.tt_from_host(y, max_rank=max(ranks))
    ctx.tt_round(t, 0.0, max(ranks), forced_ranks=ranks)
    got = ctx.tt_to_host(t)
    assert tt.diff_norm(got, x) < 1e-12 * tt.norm(x)
    ctx.tt_free(t)
    ctx.close()


def test_a_bond_that_one_side_does_not_use(B):
    """Zero columns on one side under large rows on the other: the rows meet only
    zeros and must not set the scale of what the others are cut at."""
    n, ranks = 64, [1, 48, 64, 40, 1]
    x = synthetic.random_tt_cores(4, n, ranks, seed=4)
    x[1][:, :, 5:9] = 0.0
    y = [c.copy(order="F") for c in x]
    y[2][5:9] *= 2.0 ** 60
    ctx = B.Context(d=4, n=n, nu=0.02, tol=0.0, rank_cap=64, L=4.0)
    t = ctx.tt_from_host(y, max_rank=64)
    ctx.tt_round(t, 0.0, 64, forced_ranks=[1, 48, 60, 40, 1])
    assert tt.diff_norm(ctx.tt_to_host(t), x) < 1e-12 * tt.norm(x)
    ctx.tt_free(t)
    ctx.close()


@pytest.mark.parametrize("kind,decades", [("grow", 12), ("mixed", 12)])
def test_step_does_not_see_the_gauge(B, kind, decades):
    """The operator's six-block merges: an Euler step of a state and of the same
    state in another gauge."""
    d, n, r = 4, 64, 33
    x, _ = synthetic.saturated_tt_cores(d, n, r, seed=3)
    out = []
    for y in (x, gauge(x, kind, decades, [1, 2, 3], np.random.default_rng(2))):
        ctx = B.Context(d=d, n=n, nu=0.02, tol=1e-12, rank_cap=r, L=6.0)
        t = ctx.tt_from_host(y, max_rank=r)
        ctx.hopf_step_scheme(t, B.HOPF_EULER, 1e-4, 1)
        out.append(ctx.tt_to_host(t))
        ctx.tt_free(t)
        ctx.close()
    assert tt.diff_norm(out[1], out[0]) < 1e-10 * tt.norm(out[0])
