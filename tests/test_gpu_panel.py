"""GPU: the panel kernel (the default of single solves) at the edges of its split.

Each CTA owns a slice of the rows and a strip of the columns, selects on
entries formed on demand and applies up to 16 pending pivots at a time; the
pivots and every bit of the tableau must be the oracle's where slices are
empty, uneven or one element wide, where a call ends inside, at the end or
just after a panel, in both forms, with basic columns left out of the panels
and without, and where the ratios' single-precision keys leave their range.
"""
import os

import numpy as np
import pytest

import oracle
from paper_1804_04737_gb300 import capi, lpgen
from paper_1804_04737_gb300.build import build_library
from test_gpu_parity import Run, _bits, _oracle, assert_same

pytestmark = pytest.mark.gpu

MAX_LE, MIN_GE = capi.LP_MAX_LE, capi.LP_MIN_GE


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    capi.load_library()
    oracle.set_threads(os.cpu_count() or 1)
    yield
    oracle.set_threads(1)


@pytest.mark.parametrize("zero_skip", [0, 1, 2])
@pytest.mark.parametrize("sense", [MAX_LE, MIN_GE])
@pytest.mark.parametrize("m,n,ctas", [(1, 1, 0), (2, 1, 0), (1, 40, 0), (40, 1, 0), (17, 33, 5),
                                      (31, 32, 152), (130, 90, 152), (305, 40, 1), (40, 305, 1),
                                      (305, 700, 2), (611, 310, 0), (90, 2600, 9)])
def test_slices_bitwise(m, n, ctas, sense, zero_skip):
    for A, b, c in (lpgen.dense_lp(m, n, seed=m + n), lpgen.paper_lp(m, n, seed=m + n)):
        if sense == MIN_GE:
            A, b, c = lpgen.dual_of(A, b, c)
            c = np.abs(c)
        assert_same(Run(A, b, c, sense, ctas=ctas, zero_skip=zero_skip, time_limit_s=60.0),
                    _oracle(A, b, c, sense))


@pytest.mark.parametrize("chunk", [1, 15, 16, 17, 33])
@pytest.mark.parametrize("kind", ["primal", "dual", "phase1"])
def test_calls_that_end_around_a_panel(chunk, kind):
    """Resumed in calls of `chunk` pivots: each call applies what is pending,
    so the next one starts from the tableau alone."""
    A, b, c = lpgen.paper_lp(150, 170, seed=4) if kind != "phase1" else lpgen.dense_lp(120, 90, seed=1)
    sense = MAX_LE
    if kind == "dual":
        A, b, c = lpgen.dual_of(A, b, c)
        sense = MIN_GE
    if kind == "phase1":
        A, b = lpgen.with_ge_rows(A, b, 0.1, seed=2)
    o = _oracle(A, b, c, sense)
    m, n = A.shape
    h = capi.lp_create(capi.lp_options_default(max_iters=chunk))
    try:
        capi.lp_load(h, A, b, c, sense)
        for _ in range(o.iters + 2):
            capi.lp_solve(h)
            x, y = np.empty(n), np.empty(m)
            obj, st, it = capi.lp_result(h, x, y)
            if st != capi.LP_ITER_LIMIT:
                break
        assert st == o.status and it == o.iters and _bits([obj])[0] == _bits([o.obj])[0]
        assert np.array_equal(_bits(x), _bits(o.x)) and np.array_equal(_bits(y), _bits(o.y))
        assert np.array_equal(_bits(capi.lp_get_tableau(h, m, n)), _bits(o.T))
    finally:
        capi.lp_destroy(h)


@pytest.mark.parametrize("sense", [MAX_LE, MIN_GE])
@pytest.mark.parametrize("e", [40, 61, 200])
def test_ratio_keys_out_of_range(e, sense):
    """Rows and columns scaled by 2^+-e: all, some or none of the ratios'
    operands lie within the keys' range of exponents (2^+-60)."""
    from test_gpu_scaled import scaled_lp
    (A, b, c), eps, _ = scaled_lp(90, 110, e, seed=e)
    if sense == MIN_GE:
        A, b, c = lpgen.dual_of(A, b, c)
        eps = {"eps_d": eps["eps_r"], "eps_p": eps["eps_p"], "eps_r": eps["eps_d"]}
    assert_same(Run(A, b, c, sense, zero_skip=2, **eps), _oracle(A, b, c, sense, **eps))


# overlapped panels: from 2^20 tableau elements on (fewer than 450000 per CTA)
@pytest.mark.parametrize("zero_skip", [0, 2])
@pytest.mark.parametrize("sense", [MAX_LE, MIN_GE])
@pytest.mark.parametrize("m,n,ctas", [(30, 36000, 0), (1500, 10, 0), (601, 1203, 0), (701, 800, 3),
                                      (1023, 515, 152), (150, 8001, 20)])
def test_overlapped_panels_bitwise(m, n, ctas, sense, zero_skip):
    """Few rows or columns per CTA, uneven slices, few pivots (the copy of the
    tableau still running when the pivots end) and many."""
    m1, n1 = (m, n) if sense == MAX_LE else (n, m)
    for A, b, c in (lpgen.dense_lp(m1, n1, seed=m + n), lpgen.paper_lp(m1, n1, seed=5)):
        if sense == MIN_GE:
            A, b, c = lpgen.dual_of(A, b, c)
        kw = dict(max_iters=200)
        assert_same(Run(A, b, c, sense, ctas=ctas, zero_skip=zero_skip, time_limit_s=60.0, **kw),
                    _oracle(A, b, c, sense, **kw))


@pytest.mark.parametrize("chunk", [1, 7, 8, 9, 16, 17, 24, 25])
@pytest.mark.parametrize("kind", ["primal", "dual", "phase1"])
def test_overlapped_calls_that_end_around_a_panel(chunk, kind):
    """Calls of `chunk` pivots: ending with none, one or two panels begun, in
    either buffer."""
    m, n, sense = 600, 1200, MAX_LE
    A, b, c = lpgen.dense_lp(m, n, seed=9)
    if kind == "dual":
        A, b, c = lpgen.dual_of(A, b, c)
        sense = MIN_GE
    if kind == "phase1":
        A, b = lpgen.with_ge_rows(A, b, 0.02, seed=2)
    calls = 6
    h = capi.lp_create(capi.lp_options_default(max_iters=chunk))
    try:
        capi.lp_load(h, A, b, c, sense)
        for k in range(calls):
            capi.lp_solve(h)
            _, st, it = capi.lp_result(h)
            if st != capi.LP_ITER_LIMIT:
                break
        o = _oracle(A, b, c, sense, max_iters=chunk * (k + 1))
        assert st == o.status and it == o.iters
        assert np.array_equal(capi.lp_get_basis(h, A.shape[0]), o.basis)
        assert np.array_equal(_bits(capi.lp_get_tableau(h, *A.shape)), _bits(o.T))
    finally:
        capi.lp_destroy(h)


@pytest.mark.parametrize("sense", [MAX_LE, MIN_GE])
@pytest.mark.parametrize("m,n", [(40, 30), (130, 90), (760, 690)])
def test_captured_solve_runs_again(m, n, sense):
    """A captured lp_solve_async, 7 pivots a run, run until the LP is solved,
    then again after other LPs of the shape are loaded and begun (the largest
    with overlapped panels): the values that carry tags are then those of earlier
    runs of the same launch."""
    import torch
    stream = torch.cuda.Stream()
    h = capi.lp_create(capi.lp_options_default(cuda_stream=stream, max_iters=7))
    graph = None
    try:
        for seed in (1, 2, 1):
            A, b, c = lpgen.paper_lp(m, n, seed=seed)
            if sense == MIN_GE:
                A, b, c = lpgen.dual_of(*lpgen.dense_lp(n, m, seed=seed))
            capi.lp_load(h, A, b, c, sense)
            torch.cuda.synchronize()
            if graph is None:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    capi.lp_solve_async(h)
                first = 1
            else:
                capi.lp_solve(h)
                first = 2
            o = oracle.solve(A, b, c, sense=sense)
            x, y = np.empty(A.shape[1]), np.empty(A.shape[0])
            for run in range(first, o.iters // 7 + 3):
                with torch.cuda.stream(stream):
                    graph.replay()
                obj, st, it = capi.lp_result(h, x, y)
                assert it == min(7 * run, o.iters)
                if st != capi.LP_ITER_LIMIT:
                    break
            assert st == o.status and it == o.iters and _bits([obj])[0] == _bits([o.obj])[0]
            assert np.array_equal(_bits(x), _bits(o.x)) and np.array_equal(_bits(y), _bits(o.y))
    finally:
        torch.cuda.synchronize()
        del graph
        capi.lp_destroy(h)
