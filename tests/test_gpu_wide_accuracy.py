"""The eight-digit product by itself, and the reciprocals of the FP64 chains.

Exact: integers whose long products cancel to short sums need every digit level
(38 + 30 bits: levels 0 to 7), the carry of the two lowest levels and the
fixed-point sum re + im; the result is an integer below 2^53 and must come out
as it is.  (Without the balance: it moves two columns that cancel by different
powers of two, so that their low digits can fall on either side of the cut.)

Accuracy, against extended precision: a chunk's product is rounded once, the
chunks' partial sums are FP64 additions: (1 + chunks) 2^-53 of |A||B|, entry by
entry; the cut of an operand is 2^-63 of the row's largest entry on either side
and the dropped pairs weigh 8 2^-64, with the three products of a complex one
less than K 2^-58 of the product of the largest entries."""
import numpy as np
import pytest

import native_probes

pytestmark = pytest.mark.gpu

KS = [1, 63, 64, 65, 127, 128, 129, 257]
SHAPES = [(1, 1), (130, 33), (127, 31), (257, 65)]


@pytest.fixture(scope="module")
def probes(tmp_path_factory):
    return native_probes.load(tmp_path_factory.mktemp("probes"))


def cgauss(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def reference(A, B):
    """A B^T and |A||B|^T in extended precision (real parts and imaginary parts)."""
    L = np.longdouble
    ar, ai, br, bi = (x.astype(L) for x in (A.real, A.imag, B.real, B.imag))
    re, im = ar @ br.T - ai @ bi.T, ar @ bi.T + ai @ br.T
    return re, im, (np.abs(A) @ np.abs(B).T)


def check(got, re, im, mag, cut, chunks):
    bar = (1 + (chunks if chunks > 1 else 0)) * 2.0 ** -53 * mag + cut
    assert (np.abs(got.real.astype(np.longdouble) - re) <= bar).all()
    assert (np.abs(got.imag.astype(np.longdouble) - im) <= bar).all()


def top(X, axis):
    return np.maximum(np.abs(X.real), np.abs(X.imag)).max(axis=axis)


@pytest.mark.parametrize("K", [2, 64, 128, 130, 384])
@pytest.mark.parametrize("M,N", SHAPES)
def test_cancelling_integers_are_exact(probes, M, N, K):
    rng = np.random.default_rng(M + N + K)
    ints = lambda bits, *sh: rng.integers(-2 ** bits + 1, 2 ** bits, sh)
    ar, ai = ints(38, M, K // 2), ints(38, M, K // 2)
    dr, di = ints(7, M, K // 2), ints(7, M, K // 2)
    br, bi = ints(30, N, K // 2), ints(30, N, K // 2)
    A = np.empty((M, K), complex)
    B = np.empty((N, K), complex)
    A[:, 0::2], A[:, 1::2] = ar + 1j * ai, (dr - ar) + 1j * (di - ai)
    B[:, 0::2] = B[:, 1::2] = br + 1j * bi
    want = (dr @ br.T - di @ bi.T) + 1j * (dr @ bi.T + di @ br.T)  # int64, below 2^46
    np.testing.assert_array_equal(probes.wide_product(A, B), want)


@pytest.mark.parametrize("K", KS)
@pytest.mark.parametrize("M,N", SHAPES)
@pytest.mark.parametrize("kind", ["plain", "opposite", "below_two", "graded_rows", "zero_rows"])
def test_accuracy(probes, M, N, K, kind):
    rng = np.random.default_rng(3 * M + N + K)
    A, B = cgauss(rng, M, K), cgauss(rng, N, K)
    if kind == "opposite":  # re + im far below re and im
        A = A.real * (1 - 1j) + 1e-12j * A.imag
        B = B.real * (1 - 1j) + 1e-9 * B.imag
    elif kind == "below_two":  # largest magnitudes just below a power of two
        A = np.sign(A.real) * (2.0 - 2.0 ** -52) + 1j * np.sign(A.imag) * (1.0 - 2.0 ** -53)
        B = np.sign(B.real) * (2.0 - 2.0 ** -52) - 1j * np.sign(B.imag) * (2.0 - 2.0 ** -52)
    elif kind == "graded_rows":
        A *= 10.0 ** rng.uniform(-100, 100, M)[:, None]
        B *= 10.0 ** rng.uniform(-100, 100, N)[:, None]
    elif kind == "zero_rows":
        A[:: 2] = 0.0
        B[:, ::3] = 0.0
    re, im, mag = reference(A, B)
    cut = K * 2.0 ** -58 * np.outer(top(A, 1), top(B, 1))
    chunks = (K + 127) // 128
    check(probes.wide_product(A, B), re, im, mag, cut, chunks)
    # transposed store, and the product subtracted from what is there
    C0 = cgauss(rng, M, N) * (mag + (mag == 0))
    got = probes.wide_product(A, B, C0=C0, alpha=-1.0, transposed=True)
    check(got, C0.real - re, C0.imag - im, 2 * mag + np.abs(C0), cut, chunks)


@pytest.mark.parametrize("K", [2, 64, 129, 257])
@pytest.mark.parametrize("decades", [8, 16, 200])
def test_accuracy_does_not_depend_on_the_gauge(probes, K, decades):
    """Columns of A times D and of B over D, with the balance."""
    rng = np.random.default_rng(K + decades)
    M, N = 130, 33
    A, B = cgauss(rng, M, K), cgauss(rng, N, K)
    D = 2.0 ** np.round(decades * np.log2(10.0) * (rng.random(K) - 0.5))
    re, im, mag = reference(A, B)
    # half a power of two is lost on either side where the exponents' sum is odd
    cut = 4 * K * 2.0 ** -58 * (top(A, 0) * top(B, 0)).max()
    check(probes.wide_product(A * D, B / D, balance=True), re, im, mag, cut, (K + 127) // 128)


@pytest.mark.parametrize("balance", [False, True])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1j * np.inf])
def test_what_is_not_finite_stays_in_its_row(probes, balance, bad):
    rng = np.random.default_rng(8)
    M, N, K = 40, 35, 200
    A, B = cgauss(rng, M, K), cgauss(rng, N, K)
    clean = A.copy()
    clean[:, 150] = 0.0  # (the balance leaves the column's maximum to the finite rows)
    A[:, 150] = 0.0
    A[3, 150] = bad
    got = probes.wide_product(A, B, balance=balance)
    assert np.isnan(got[3]).all()
    keep = np.arange(M) != 3
    re, im, mag = reference(clean[keep], B)
    check(got[keep], re, im, mag, K * 2.0 ** -58 * np.outer(top(clean[keep], 1), top(B, 1)), 2)


def test_reciprocals(probes):
    """1 / x: the seed's 2^-20 to the third power is far below the last bit, so
    what is left is one rounding, half a unit and a little; 1 / sqrt(x) has x y
    rounded as well: one unit.  All binades of the stated range, its ends, and
    mantissas next to powers of two."""
    rng = np.random.default_rng(0)
    e = np.concatenate([np.arange(-962, 963), rng.integers(-962, 963, 200000)])
    m = np.concatenate([np.ones(1925), 1.0 + rng.random(199990),
                        [1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5, 4 / 3, np.sqrt(2), 1.0 + 2.0 ** -20, 1.25, 1.75, 1.1]])
    x = np.ldexp(m, e) * rng.choice([-1.0, 1.0], m.size)
    x = np.concatenate([x, [1e-290, 1e290, -1e290]])
    r, s = probes.reciprocals(x)
    X = x.astype(np.longdouble)
    for got, want, units in ((r, 1 / X, 0.51), (s, 1 / np.sqrt(np.abs(X)), 1.01)):
        unit = np.spacing(np.abs(want).astype(np.float64))
        assert np.abs((got - want) / unit).max() <= units


def test_reflector_is_unitary(probes):
    """tau, scale and beta of the FP64 panels' reflector over the range of its
    fast forms (|alpha|^2 + |x|^2 from 2^-928 to 2^929) and beyond the ends:
    |tau|^2 |v|^2 = 2 Re tau with |v|^2 = 1 + |scale|^2 |x|^2, and |beta| the
    norm.  About twenty roundings of at most a unit of 2^-53 each enter either
    side: 16 eps."""
    rng = np.random.default_rng(1)
    n = 40000
    al = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 10.0 ** rng.uniform(-8, 8, n)
    s2 = 10.0 ** rng.uniform(-16, 16, n)
    al[::17], s2[::19], al[::23] = 0.0, 0.0, al[::23].real
    e = rng.integers(-490, 490, n)
    edge = np.array([-465, -464, -463, 463, 464, 465, 466])
    e[: n // 2] = edge[rng.integers(0, edge.size, n // 2)]
    scale_to = np.sqrt(np.abs(al) ** 2 + s2) + (al == 0) * (s2 == 0)
    al, s2 = al / scale_to, s2 / scale_to ** 2
    al, s2 = al * 2.0 ** e, np.ldexp(s2, 2 * e)
    tau, sc, beta = probes.house(al, s2)
    L = np.longdouble
    norm = np.sqrt(al.real.astype(L) ** 2 + al.imag.astype(L) ** 2 + s2.astype(L))
    none = (s2 == 0) & (al.imag == 0)
    eps = np.finfo(float).eps
    assert (tau[none] == 0).all() and (sc[none] == 0).all() and (beta[none] == al.real[none]).all()
    k = ~none
    assert (np.abs(np.abs(beta[k]) - norm[k]) <= 16 * eps * norm[k]).all()
    assert (np.signbit(beta[k]) != (al.real[k] < 0)).all()
    t2 = tau.real.astype(L) ** 2 + tau.imag.astype(L) ** 2
    v2 = 1 + (sc.real.astype(L) ** 2 + sc.imag.astype(L) ** 2) * s2.astype(L)
    assert (np.abs(t2 * v2 - 2 * tau.real)[k] <= 16 * eps * 2 * tau.real[k]).all()
