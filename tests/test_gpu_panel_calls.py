"""GPU: the rules that choose between the panel kernel's two forms and the others.

A call of fewer than 16 pivots (more on larger tableaus) runs its panels in turn,
a longer one overlapped, on the same tableau; LPs of fewer than 64 rows or
columns run them in turn; wide LPs of few rows or of long rows go to the kernels
that split the columns.  Whatever the call takes, its pivots and every bit of the
tableau are the oracle's.
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


def _lp(kind, m, n):
    A, b, c = lpgen.dense_lp(m, n, seed=9)
    if kind == "dual":
        return (*lpgen.dual_of(A, b, c), MIN_GE)
    if kind == "phase1":  # (the call that ends Phase 1 goes on with what is left of its pivots)
        A, b = lpgen.with_ge_rows(A, b, 0.02, seed=2)
    return A, b, c, MAX_LE


@pytest.mark.parametrize("chunk", [2, 15, 16, 18, 20, 21, 31])
@pytest.mark.parametrize("kind", ["primal", "dual", "phase1"])
def test_calls_of_few_and_many_pivots(chunk, kind):
    A, b, c, sense = _lp(kind, 600, 1200)
    h = capi.lp_create(capi.lp_options_default(max_iters=chunk))
    try:
        capi.lp_load(h, A, b, c, sense)
        for k in range(5):
            capi.lp_solve(h)
            _, st, it = capi.lp_result(h)
            if st != capi.LP_ITER_LIMIT:
                break
        o = oracle.solve(A, b, c, sense=sense, max_iters=chunk * (k + 1), keep_tableau=True)
        assert st == o.status and it == o.iters
        assert np.array_equal(capi.lp_get_basis(h, A.shape[0]), o.basis)
        assert np.array_equal(_bits(capi.lp_get_tableau(h, *A.shape)), _bits(o.T))
    finally:
        capi.lp_destroy(h)


@pytest.mark.parametrize("kind", ["primal", "dual"])
def test_captured_overlapped_solve_runs_again(kind):
    """A captured call of 19 pivots (overlapped), run again and again, also once
    other LPs of the shape were loaded and begun."""
    import torch
    m, n = (760, 690) if kind == "primal" else (690, 760)
    stream = torch.cuda.Stream()
    h = capi.lp_create(capi.lp_options_default(cuda_stream=stream, max_iters=19))
    graph = None
    try:
        for seed in (1, 2, 1):
            A, b, c = lpgen.paper_lp(m, n, seed=seed)
            sense = MAX_LE
            if kind == "dual":
                A, b, c = lpgen.dual_of(*lpgen.dense_lp(m, n, seed=seed))
                sense = MIN_GE
            capi.lp_load(h, A, b, c, sense)
            torch.cuda.synchronize()
            first = 1
            if graph is None:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    capi.lp_solve_async(h)
            else:
                capi.lp_solve(h)
                first = 2
            o = oracle.solve(A, b, c, sense=sense)
            x, y = np.empty(A.shape[1]), np.empty(A.shape[0])
            for run in range(first, o.iters // 19 + 3):
                with torch.cuda.stream(stream):
                    graph.replay()
                obj, st, it = capi.lp_result(h, x, y)
                assert it == min(19 * run, o.iters)
                if st != capi.LP_ITER_LIMIT:
                    break
            assert st == o.status and it == o.iters and _bits([obj])[0] == _bits([o.obj])[0]
            assert np.array_equal(_bits(x), _bits(o.x)) and np.array_equal(_bits(y), _bits(o.y))
    finally:
        torch.cuda.synchronize()
        del graph
        capi.lp_destroy(h)


# either side of 64 columns and of 64 rows (overlapped from 2^20 elements on); of 16
# rows; and of the wide rule's bound on the columns per CTA, on all CTAs and on two
@pytest.mark.parametrize("zero_skip", [1, 2])
@pytest.mark.parametrize("sense", [MAX_LE, MIN_GE])
@pytest.mark.parametrize("m,n,ctas", [(1100, 63, 0), (1100, 64, 0), (63, 16600, 0), (64, 16600, 0), (15, 400, 0),
                                      (16, 400, 0), (20, 81, 0), (20, 3000, 0), (150, 8100, 0), (150, 8600, 0),
                                      (160, 6000, 0), (17, 310, 2), (17, 330, 2), (20, 379, 2),
                                      (20, 381, 2)])
def test_either_side_of_the_rules(m, n, ctas, sense, zero_skip):
    m1, n1 = (m, n) if sense == MAX_LE else (n, m)
    A, b, c = lpgen.dense_lp(m1, n1, seed=m + n)
    if sense == MIN_GE:
        A, b, c = lpgen.dual_of(A, b, c)
    for kw in ({}, {"max_iters": 13}):
        assert_same(Run(A, b, c, sense, ctas=ctas, zero_skip=zero_skip, **kw), _oracle(A, b, c, sense, **kw))
