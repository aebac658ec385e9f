"""The tiled dense products in each tile size: shapes whose tiles of 64, 32, 16
are just enough for 152 SMs (13 x 13 tiles or 14 x 13), one below, with remainders
in every direction, and the smallest.

Against extended precision, real and imaginary parts entry by entry, relative to
|A||B|: FP64 chains of two multiply-adds per term, K 2^-52; double-float products
and sums lose a few 2^-48 each, K 2^-45."""
import numpy as np
import pytest

import native_probes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probes(tmp_path_factory):
    return native_probes.load(tmp_path_factory.mktemp("probes"))


SHAPES = [(830, 780), (420, 400), (200, 215), (50, 45), (1, 1), (9, 1300)]


@pytest.mark.parametrize("M,N", SHAPES)
@pytest.mark.parametrize("K", [1, 17, 64])
@pytest.mark.parametrize("kind", ["rh", "rblk", "uh", "rh_mixed", "rblk_mixed"])
def test_products(probes, M, N, K, kind):
    rng = np.random.default_rng(M + N + K)
    cgauss = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    mixed = kind.endswith("mixed")
    if kind == "uh":
        A, R = cgauss(K, M), cgauss(K, N)
        got = probes.gemm(A, R, uh=True)
        L, R2 = A.conj().T, R
    else:
        coff = 5 if kind.startswith("rblk") else 0
        A, R = cgauss(M, K), cgauss(N, coff + K)
        got = probes.gemm(A, R, coff=coff, mixed=mixed)  # below the trapezoid R holds anything
        L, R2 = A, np.triu(R)[:, coff:].conj().T
    lr, li, rr, ri = (x.astype(np.longdouble) for x in (L.real, L.imag, R2.real, R2.imag))
    bar = K * 2.0 ** (-45 if mixed else -52) * (np.abs(L) @ np.abs(R2))
    assert (np.abs(got.real - (lr @ rr - li @ ri)) <= bar).all()
    assert (np.abs(got.imag - (lr @ ri + li @ rr)) <= bar).all()
