"""GPU: the body refresh's products run over groups of four tableau columns
that are not all basic slacks.  Shapes at the edges of the groups (the number
of structurals modulo 4, a last group cut by the rhs column, rows of A on and
off 32 bytes) and of the tiles, in both forms, against the definition, with
the bound of the refresh's own test (one FP32 rounding plus 1e-10 of the row)."""
import numpy as np
import pytest

import oracle
from paper_1804_04737_gb300 import capi, lpgen
from paper_1804_04737_gb300.build import build_library
from test_gpu_ozaki import _fp32_stopped

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    capi.load_library()


@pytest.mark.parametrize("sense", [capi.LP_MAX_LE, capi.LP_MIN_GE])
@pytest.mark.parametrize("m,n", [(1, 1), (3, 2), (2, 5), (7, 4), (33, 30), (61, 64), (66, 63), (130, 129),
                                 (129, 260), (515, 512)])
def test_refresh_at_group_edges(m, n, sense):
    for gen in (lpgen.dense_lp, lpgen.paper_lp):
        A, b, c = gen(m, n, seed=m)
        if sense == capi.LP_MIN_GE:
            A, b, c = lpgen.dual_of(A, b, c)
        mm = A.shape[0]
        st, total, *_ = _fp32_stopped(A, b, c, sense, 10 ** 9)
        assert st == capi.LP_OPTIMAL
        for k in sorted({1, total // 2, total - 1} - {0, -1}):
            if k >= total:
                continue
            _, it, basis, T, nre, _ = _fp32_stopped(A, b, c, sense, k)
            assert it == k and nre >= 1
            R = oracle.reinvert(A, b, c, basis, sense=sense)[:mm, :-1]
            want = R.astype(np.float32).astype(np.float64)
            tol = (np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
                   + 1e-10 * np.abs(R).max(axis=1, keepdims=True))
            assert np.all(np.abs(T[:mm, :-1] - want) <= tol)
            unit = T[:mm, basis]
            assert np.array_equal(unit, np.eye(mm)) and not np.any(np.signbit(unit))
