"""Singular values and left vectors of a bond factor through tt_round: spectra
that decide which path the vectors take (separate values, values equal in
groups, a group at rounding level), at sizes around the kernels' edges.

Tolerance: the rounding is backward stable, so with the cut in a gap of a
factor of ten the result moves by about n eps sigma_1 / (sigma_cut - next) *
sigma_cut, at most 514 * 2.2e-16 * 1.1 * 10 = 1.3e-12 of the norm; 1e-11
leaves room for the sweeps around it.  Orthonormality: the columns are
products of n reflections, n eps = 1.1e-13; 1e-12 as in the other tests."""
import numpy as np
import pytest

from oracle import tt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2403_04946_gb300 import binding, build
    build.build()
    return binding


def spectrum(kind, n):
    if kind == "decaying":
        return np.logspace(0, -15, n)
    if kind == "groups":  # five equal values at each level, levels a factor of ten apart
        return 10.0 ** -(np.arange(n) // 5 % 14).astype(float)
    if kind == "equal":
        return np.ones(n)
    if kind == "close":  # neighbours 1e-9 apart: orthogonal only after the correction
        return np.logspace(0, -3, (n + 1) // 2).repeat(2)[:n] * (1.0 + 1e-9 * (np.arange(n) % 2))
    s = np.logspace(0, -4, n)  # "deficient"
    s[(n + 1) // 2:] = 0.0
    return s


@pytest.mark.parametrize("kind", ["decaying", "groups", "equal", "close", "deficient"])
@pytest.mark.parametrize("n", [1, 2, 33, 64, 130, 512, 514])
def test_left_vectors_of_a_planted_spectrum(B, n, kind):
    rng = np.random.default_rng(n)
    m, q = n + 2 + n % 2, 2
    m = max(m, 4)
    s = np.sort(spectrum(kind, n))[::-1]
    cgauss = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
    Ul = np.linalg.qr(cgauss(m, n))[0]
    Vr = np.linalg.qr(cgauss(m * q, n))[0]  # orthonormal rows of the rest: the bond's values are s
    last = np.linalg.qr(cgauss(m, q))[0]
    cores = [np.asfortranarray((Ul * s).reshape(1, m, n)),
             np.asfortranarray(Vr.conj().T.reshape(n, m, q)), np.asfortranarray(last.T.reshape(q, m, 1))]
    # cut inside a gap: below the last value above 3e-6 of the largest
    keep = int(np.sum(s > 3e-6))
    forced = [1, keep, q, 1]
    want, _, wdisc = tt.round_tt(cores, 0.0, n, forced)
    ctx = B.Context(d=3, n=m, nu=0.05, tol=0.0, rank_cap=n, L=3.0)
    t = ctx.tt_from_host(cores, max_rank=max(n, q))
    disc, _ = ctx.tt_round(t, 0.0, n, forced_ranks=forced)
    got = ctx.tt_to_host(t)
    V = tt.V(got[0])
    assert np.abs(V.conj().T @ V - np.eye(V.shape[1])).max() < 1e-12
    # the kept part of a decaying spectrum has its neighbours close to the cut
    bar = 1e-11 if kind != "decaying" else 1e-11 + 10 * n * 2.3e-16
    assert tt.diff_norm(got, want) < bar * np.linalg.norm(s)
    assert abs(disc - wdisc) < 1e-6 * wdisc + 1e-13 * np.linalg.norm(s)
    ctx.tt_free(t)
    ctx.close()
