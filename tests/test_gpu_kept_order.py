"""Mixed contexts with digit products keep their order of operations: a step,
roundings, a step from the library's own initial state and a sum with an
applied operator against recorded values (tests/golden/kept_order.txt, hex
floats; nvcc 13.0, GB300).

The five-digit products cut at 2^-40, so a changed last bit in a factor, a
bidiagonal or a singular vector shows in Phi at 1e-11 to 1e-10 and more in a
covariance; with the order kept the cores are the same to the last bit.
Tolerance: what remains is the read-out, a product of d vector-matrix products
of r terms in FP64, d r eps = 4 * 64 * 2.2e-16 = 6e-14 of the product of
magnitudes; the entries are independent, so values and differences are of that
size up to the factor of cancellation of a sum of r signed terms: 1e-12."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "kept_order.txt")
# d, n, ranks, powers of two over which the bonds' weights fall, what is done
CASES = {"step": (4, 128, [1, 64, 64, 64, 1], 20, "step"),
         "wide_factor": (3, 128, [1, 300, 64, 1], 30, "round"),
         "tall_factors": (4, 128, [1, 128, 300, 128, 1], 12, "round"),
         "init_step": (6, 32, [1, 32, 32, 32, 32, 32, 1], 0, "init"),
         "apply_sum": (4, 128, [1, 64, 64, 64, 1], 20, "apply")}


def read_out(name):
    """Mean, covariance and values near the centre, as one vector."""
    from paper_2403_04946_gb300 import binding as B
    d, n, ranks, decay, what = CASES[name]
    rng = np.random.default_rng(5)
    cores = []
    for a, b in zip(ranks[:-1], ranks[1:]):
        c = rng.standard_normal((a, n, b)) + 1j * rng.standard_normal((a, n, b))
        # exact weights: the same input bits on every machine
        cores.append(np.asfortranarray(c * 2.0 ** -np.floor(decay * np.arange(b) / max(b - 1, 1))))
    idx = rng.integers(n // 4, 3 * n // 4, size=(12, d)).astype(np.int32)
    cap = min(64, max(ranks))
    ctx = B.Context(d=d, n=n, nu=0.01, tol=1e-7, rank_cap=cap, L=12.4, precision=B.HOPF_MIXED)
    if what == "init":
        t = ctx.hopf_init_gaussian(np.linspace(-0.125, 0.25, d), np.eye(d) * 0.5 + 0.25)
    else:
        t = ctx.tt_from_host(cores, max_rank=max(ranks))
    if what == "apply":  # x + dt G x by hand
        g, s = ctx.tt_create(6 * cap), ctx.tt_create(7 * cap)
        ctx.hopf_apply_op(t, g)
        ctx.tt_sum([t, g], np.array([1.0, 2.0 ** -16]), s)
        ctx.tt_free(g)
        ctx.tt_free(t)
        t = s
    if what in ("step", "init"):
        ctx.hopf_step(t, 1.2e-5, 1)
    else:
        ctx.tt_round(t, 1e-7, cap)
    mean, cov, _ = ctx.hopf_eval_moments(t)
    phi = ctx.hopf_eval_points(t, idx)
    ctx.tt_free(t)
    ctx.close()
    return [np.ravel(mean), np.ravel(cov), phi.real, phi.imag]


def recorded(name):
    with open(GOLDEN) as f:
        rows = [line.split() for line in f if line.startswith(name + " ")]
    return [np.array([float.fromhex(v) for v in r[1:]]) for r in rows]


@pytest.mark.parametrize("name", CASES)
def test_outputs_are_the_recorded_ones(name):
    for got, want in zip(read_out(name), recorded(name), strict=True):
        assert np.max(np.abs(got - want)) < 1e-12 * np.max(np.abs(want))


def test_factor_whose_solver_arrays_fit_once():
    """A bond factor of 1200 columns: the serial vectors' factors have one
    buffer in shared memory.  Against the FP64 rounding of the same tensor; the
    cut products are good to 2^-40 of their operands, a tenth of the rounding
    tolerance is the bar."""
    from paper_2403_04946_gb300 import binding as B
    from oracle import tt
    d, n, ranks = 4, 64, [1, 64, 1200, 64, 1]
    rng = np.random.default_rng(3)
    cores = []
    for a, b in zip(ranks[:-1], ranks[1:]):
        c = rng.standard_normal((a, n, b)) + 1j * rng.standard_normal((a, n, b))
        cores.append(np.asfortranarray(c * 2.0 ** -np.floor(16 * np.arange(b) / max(b - 1, 1))))
    out = []
    for precision in (B.HOPF_MIXED, B.HOPF_FP64):
        ctx = B.Context(d=d, n=n, nu=0.01, tol=1e-7, rank_cap=90, L=6.0, precision=precision)
        t = ctx.tt_from_host(cores, max_rank=1200)
        ctx.tt_round(t, 1e-7, 90, forced_ranks=[1, 60, 90, 60, 1])
        out.append(ctx.tt_to_host(t))
        ctx.tt_free(t)
        ctx.close()
    for C in out[0][:-1]:
        V = tt.V(C)
        assert np.abs(V.conj().T @ V - np.eye(V.shape[1])).max() < 1e-9
    assert tt.diff_norm(out[0], out[1]) < 1e-8 * tt.norm(out[1])
