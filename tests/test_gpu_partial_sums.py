"""Partial sums of the digit products' K-chunks: the buffer stays bounded, and a
product that runs in groups of columns gives the same bits."""
import numpy as np
import pytest

import native_probes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probes(tmp_path_factory):
    return native_probes.load(tmp_path_factory.mktemp("probes"))


@pytest.mark.parametrize("digits,chunk", [(0, 128), (5, 192)])
@pytest.mark.parametrize("M,N,K", [(327680, 2560, 2560), (65536, 18432, 512), (128, 384, 49152), (1, 1, 129)])
def test_buffer_is_bounded(probes, digits, chunk, M, N, K):
    """A merge of 2560 columns, the six blocks of a rank-512 state, a panel's
    products, the smallest: never more than all of the partial sums, 1 GiB, or
    those of one tile's columns; none for a single chunk."""
    nz = -(-K // chunk)
    got = probes.lib.probe_part_bytes(M, N, K, digits)
    assert got == (min(16 * nz * M * N, max(1 << 30, 16 * nz * M * 32)) if nz > 1 else 0)


@pytest.mark.parametrize("digits,K", [(0, 129), (0, 700), (5, 193), (5, 700)])
@pytest.mark.parametrize("N", [33, 64, 130])
@pytest.mark.parametrize("transposed,accumulate", [(False, False), (True, True)])
def test_groups_of_columns_give_the_same_bits(probes, digits, K, N, transposed, accumulate):
    rng = np.random.default_rng(K + N)
    M = 70
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((N, K)) + 1j * rng.standard_normal((N, K))
    kw = dict(C0=np.ones((M, N)), alpha=-1.0) if accumulate else {}
    whole = probes.wide_product(A, B, transposed=transposed, digits=digits, **kw)
    nz = -(-K // (192 if digits else 128))
    for cols in (32, 64 + 5):
        got = probes.wide_product(A, B, transposed=transposed, digits=digits, max_part=nz * M * cols, **kw)
        np.testing.assert_array_equal(got, whole)
