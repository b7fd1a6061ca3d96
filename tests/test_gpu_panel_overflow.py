"""GPU: solves whose entries overflow, on the panel kernel and on the one that
updates the tableau every pivot (pipeline 0).

Finite data of widely spread exponents; within 60 pivots most of the tableaus hold
infinities and NaN, so panels get every column, rows turn non-finite, and ratios
and objective entries with them.  Status, pivots, basis and tableau are the same
bits (a NaN is a NaN); in turn and overlapped, columns left out where they may be.
"""
import numpy as np
import pytest

from paper_1804_04737_gb300 import capi, lpgen
from paper_1804_04737_gb300.build import build_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    capi.load_library()


def _bits(a):
    u = np.array(a, dtype=np.float64).view(np.uint64)
    u[np.isnan(u.view(np.float64))] = 0x7ff8000000000000
    return u


def _run(A, b, c, sense, **opts):
    m, n = A.shape
    h = capi.lp_create(capi.lp_options_default(max_iters=60, trace_cap=60, eps_d=1e-300, eps_p=1e-300, eps_r=1e-300,
                                               **opts))
    try:
        capi.lp_load(h, A, b, c, sense)
        capi.lp_solve(h)
        _, st, it = capi.lp_result(h)
        tp, tq = capi.lp_get_trace(h, 60)
        return st, it, list(tp), list(tq), list(capi.lp_get_basis(h, m)), capi.lp_get_tableau(h, m, n)
    finally:
        capi.lp_destroy(h)


@pytest.mark.parametrize("e", [500, 700, 850, 1000])
@pytest.mark.parametrize("sense", [capi.LP_MAX_LE, capi.LP_MIN_GE])
@pytest.mark.parametrize("m,n", [(20, 30), (90, 70), (601, 1203), (1100, 300)])
def test_overflowing_solves_agree(m, n, sense, e):
    for seed in range(3):
        rng = np.random.default_rng(10 * seed + e)

        def spread(*shape):
            return np.ldexp(rng.uniform(0.5, 1.0, shape), rng.integers(-e, e, size=shape))

        A, b, c = spread(m, n) * (rng.random((m, n)) < 0.9), spread(m), spread(n)
        if sense == capi.LP_MIN_GE:
            A, b, c = lpgen.dual_of(A, b, c)
        want = _run(A, b, c, sense, pipeline=0)
        for zero_skip in (1, 2):
            got = _run(A, b, c, sense, zero_skip=zero_skip)
            assert got[:5] == want[:5]
            assert np.array_equal(_bits(got[5]), _bits(want[5]))
