"""GPU: the panel kernel divides a pivot row by the pivot's reciprocal and two
corrections where the operands' exponents lie within 2^+-500, by a / b elsewhere;
every quotient must be IEEE's.

One row and one pivot per solve: T[0][j] = A[0][j] / A[0][q] for every column (the
last one is the rhs), read back from the tableau after one pivot and compared with
numpy's division.  Pivots and numerators have exponents at, inside and outside the
limits, significands next to 1 and 2, of few bits, of runs of ones and random, and
signed zeros among the numerators.
"""
import numpy as np
import pytest

from paper_1804_04737_gb300 import capi
from paper_1804_04737_gb300.build import build_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    capi.load_library()


def _significands(rng, count):
    """In [1, 2): 1 + k ulp, 2 - k ulp, few bits, runs of ones, random."""
    k = rng.integers(0, 5, size=count)
    few = rng.integers(0, 1 << 8, size=count).astype(np.uint64) << np.uint64(44)
    lo, hi = rng.integers(0, 27, size=count), rng.integers(27, 53, size=count)
    ones = ((np.uint64(1) << hi.astype(np.uint64)) - (np.uint64(1) << lo.astype(np.uint64))) & np.uint64(2 ** 52 - 1)
    kinds = [k.astype(np.uint64), np.uint64(2 ** 52 - 1) - k.astype(np.uint64), few, ones,
             rng.integers(0, 1 << 52, size=count).astype(np.uint64)]
    pick = rng.integers(0, len(kinds), size=count)
    frac = np.choose(pick, kinds)
    return (np.uint64(1023 << 52) | frac).view(np.float64)


def _values(rng, exps, count):
    v = np.ldexp(_significands(rng, count), rng.choice(exps, size=count))
    return v * rng.choice([-1.0, 1.0], size=count)


# exponents of pivot and numerators (the limits are +-500; quotients stay normal)
@pytest.mark.parametrize("pivot", [0, 1, 499, 500, 501, -499, -500, -501, -640])
@pytest.mark.parametrize("dual", [False, True])
def test_pivot_row_is_the_ieee_quotient(dual, pivot):
    m, n, r = 760, 3000, 411  # (n <= 4 m: the panel kernel's; the other rows are zero)
    for seed in range(4):
        rng = np.random.default_rng(1000 * seed + abs(pivot) + 7 * dual)
        near = [e for e in (-501, -500, -499, -1, 0, 1, 499, 500, 501) if -1021 < e - pivot < 1021]
        row = _values(rng, near, n)
        row[rng.integers(0, n, size=40)] *= 0.0
        q = int(rng.integers(0, n))
        p = float(np.ldexp(_significands(rng, 1)[0], pivot))
        A, b, slack = np.zeros((m, n)), np.zeros(m), np.zeros(m)
        b[r] = abs(_values(rng, near, 1)[0])
        slack[r] = 1.0
        if not dual:  # only column q has a positive objective entry, and only row r can leave
            row[q] = p
            A[r], c, sense = row, np.full(n, -1.0), capi.LP_MAX_LE
            c[q] = 1.0
            T0, piv = np.concatenate([row, slack, b[r:r + 1]]), p
        else:  # the form's row is [-A | 1 | -b]: it leaves, and only column q can enter
            A[r], c, sense = -np.abs(row), np.ones(n), capi.LP_MIN_GE
            A[r, q] = p
            T0, piv = np.concatenate([-A[r], slack, -b[r:r + 1]]), -p
        h = capi.lp_create(capi.lp_options_default(max_iters=1, eps_d=1e-300, eps_p=1e-300, eps_r=1e-300))
        try:
            capi.lp_load(h, A, b, c, sense)
            capi.lp_solve(h)
            _, st, it = capi.lp_result(h)
            got = capi.lp_get_tableau(h, m, n)[r]
        finally:
            capi.lp_destroy(h)
        assert it == 1 and st in (capi.LP_ITER_LIMIT, capi.LP_OPTIMAL)
        want = T0 / piv
        bad = np.flatnonzero(got.view(np.uint64) != want.view(np.uint64))
        assert bad.size == 0, (bad[:5], T0[bad[:5]], piv)
