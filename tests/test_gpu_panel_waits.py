"""GPU: the panel kernel's waits run out (short lp_options.spin_timeout_cycles).

A solve whose waits run out ends in LP_TIMEOUT wherever it then is: at an
exchange of records, at a tagged value, at the group's barrier, with a panel
under way on the overlapped kernel's other warps or without.  With a limit that
some runs meet the results are the oracle's.  The context stays usable: a handle
with the default limit then solves the same LP.
"""
import os

import pytest

import oracle
from paper_1804_04737_gb300 import capi, lpgen
from paper_1804_04737_gb300.build import build_library
from test_gpu_parity import Run, _oracle, assert_same

pytestmark = pytest.mark.gpu

MAX_LE, MIN_GE = capi.LP_MAX_LE, capi.LP_MIN_GE


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    capi.load_library()
    oracle.set_threads(os.cpu_count() or 1)
    yield
    oracle.set_threads(1)


# (in turn on many CTAs and on two, overlapped from 2^20 tableau elements on)
@pytest.mark.parametrize("limit", [1, 300, 1500, 4000, 20000])
@pytest.mark.parametrize("sense", [MAX_LE, MIN_GE])
@pytest.mark.parametrize("m,n,ctas", [(90, 70, 0), (300, 200, 2), (601, 1203, 0), (1203, 601, 20)])
def test_waits_that_run_out(m, n, ctas, sense, limit):
    A, b, c = lpgen.dense_lp(m, n, seed=3)
    if sense == MIN_GE:
        A, b, c = lpgen.dual_of(A, b, c)
    o = _oracle(A, b, c, sense)
    h = capi.lp_create(capi.lp_options_default(ctas=ctas, spin_timeout_cycles=limit))
    try:
        capi.lp_load(h, A, b, c, sense)
        capi.lp_solve(h)
        obj, st, it = capi.lp_result(h)
        if st == capi.LP_TIMEOUT:
            assert it <= o.iters
            with pytest.raises(capi.LpError) as e:
                capi.lp_solve(h)
            assert e.value.code == capi.LP_ERR_STATE
        else:
            assert limit > 1 and st == o.status and it == o.iters and obj == o.obj
    finally:
        capi.lp_destroy(h)
    assert_same(Run(A, b, c, sense, ctas=ctas), o)
