"""Eight-digit products at the ends of the FP64 range: results in the highest
binade, overflow, results and operands below the normal range."""
import numpy as np
import pytest

import native_probes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probes(tmp_path_factory):
    return native_probes.load(tmp_path_factory.mktemp("probes"))


@pytest.mark.parametrize("balance", [False, True])
@pytest.mark.parametrize("ea,eb", [(1023, 0), (511, 512), (0, 1023), (1000, 24), (-1074, 0), (-537, -537), (-1022, -52),
                                   (-1000, -60), (-1060, 30), (-600, -474), (-700, -700)])
def test_single_products_at_the_ends_of_the_range(probes, balance, ea, eb):
    """One term, so the result is a single rounding of the exact product, numpy's
    own (the factors have 8 bits: exact unless the range cuts)."""
    a = np.ldexp(np.array([1.0, 1.25, -1.9921875, 0.0])[:, None], ea) + 0j
    b = np.ldexp(np.array([1.0, -1.5, 1.9921875])[:, None], eb) + 0j
    with np.errstate(all="ignore"):
        want = (a.real @ b.real.T)
    got = probes.wide_product(a, b, balance=balance)
    fin = np.isfinite(want)
    np.testing.assert_array_equal(got.real[~fin], want[~fin])
    assert (got.imag[fin] == 0).all()
    # below the normal range a tie may go away from zero instead of to even: one unit of 2^-1074
    assert np.abs(got.real[fin] - want[fin]).max() <= (5e-324 if ea + eb < -1014 else 0.0)


def test_sums_below_the_normal_range(probes):
    """Integers times 2^-1070 against integers: exact."""
    rng = np.random.default_rng(0)
    A = rng.integers(-9, 10, (5, 40)) + 1j * rng.integers(-9, 10, (5, 40))
    B = rng.integers(-9, 10, (4, 40)) + 1j * rng.integers(-9, 10, (4, 40))
    got = probes.wide_product(A * 2.0 ** -1070, B)
    np.testing.assert_array_equal(got, (A @ B.T) * 2.0 ** -1070)
