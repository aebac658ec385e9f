"""The dense products of a rounding (merges, projections) in every tile size
(8, 16, 32 and 64 wide: the largest that gives each SM a tile), with edges
that the tiles do not divide.  The rounding at tol = 0 reproduces the tensor;
FP64 to 1e-12 as in the other rounding tests, double-float to 1e-11 (2^-48
per operation)."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,r", [(4, 3), (6, 9), (10, 17), (22, 35), (30, 60), (40, 100)])
def test_rounding_in_every_tile_size(B, n, r, precision):
    d = 4
    ranks = [1, min(r, n), r, min(r, n), 1]
    x = synthetic.random_tt_cores(d, n, ranks, seed=r)
    ctx = B.Context(d=d, n=n, nu=0.02, tol=0.0, rank_cap=r, L=4.0, precision=precision)
    ctx.hopf_set_qr_method(B.HOPF_QR_DOUBLEFLOAT)
    t = ctx.tt_from_host(x, max_rank=r)
    ctx.tt_round(t, 0.0, r, forced_ranks=ranks)
    assert tt.diff_norm(ctx.tt_to_host(t), x) < (1e-11 if precision else 1e-12) * tt.norm(x)
    ctx.tt_free(t)
    ctx.close()
