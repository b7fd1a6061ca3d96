"""GPU: the kernels a batch may take give the oracle's bits, whichever takes it.

lp_batch_stats tells which it was: the panel kernel has CTAs of 256 threads, the
kernel that updates the tableau every pivot the threads asked for (512).
"""
import os
import subprocess
import sys

import pytest

import oracle
from paper_1804_04737_gb300 import capi, lpgen
from paper_1804_04737_gb300.build import build_library
from test_gpu_batch import _check_against_oracle

pytestmark = pytest.mark.gpu

PANEL, EVERY_PIVOT = 256, 512


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    capi.load_library()
    oracle.set_threads(os.cpu_count() or 1)
    yield
    oracle.set_threads(1)


def _lps(shapes, dual=False):
    lps = []
    for k, (m, n) in enumerate(shapes):
        if dual:
            lps.append((*lpgen.dual_of(*lpgen.dense_lp(n, m, seed=k)), capi.LP_MIN_GE))
        else:
            lps.append((*lpgen.dense_lp(m, n, seed=k), capi.LP_MAX_LE))
    return lps


def _solve(lps, kernel, **opts):
    _check_against_oracle(lps, capi.lp_solve_batch(lps, capi.lp_options_default(**opts), want_xy=True))
    assert capi.lp_batch_stats()[3] == kernel


@pytest.mark.parametrize("zero_skip", [0, 1, 2])
@pytest.mark.parametrize("dual", [False, True])
def test_zero_skip(dual, zero_skip):
    """Batches leave out the columns that stay basic whatever is asked."""
    _solve(_lps([(60, 50), (9, 30), (200, 40), (33, 17)], dual), PANEL, zero_skip=zero_skip)


@pytest.mark.parametrize("dual", [False, True])
def test_few_wide_lps(dual):
    """Most of the tableau elements in wide LPs with long rows, fewer than two
    CTAs per SM: the column split; otherwise panels."""
    wide, square = (30, 1500), (150, 140)
    _solve(_lps([wide, (40, 40), (9, 1200)], dual), EVERY_PIVOT)
    _solve(_lps([wide, square, square, square], dual), PANEL)
    _solve(_lps([(30, 350), (6, 300)], dual), PANEL)
    _solve(_lps([(30, 450)], dual), EVERY_PIVOT if dual else PANEL)
    _solve(_lps([(12, 1100)] * 320, dual), PANEL)


def test_one_lp_past_the_panel_kernels_shared_memory():
    """It takes the whole batch with it."""
    _solve(_lps([(400, 400), (2, 30000), (9, 20)]), PANEL)
    _solve(_lps([(400, 400), (2, 50000), (9, 20)]), EVERY_PIVOT)


NO_ROOM = """
import sys
sys.path[:0] = [%r, %r]
import numpy as np
import torch
from paper_1804_04737_gb300 import capi, lpgen
from test_gpu_batch import _check_against_oracle
few = [(*lpgen.dense_lp(8, 8, seed=1), capi.LP_MAX_LE)]
capi.lp_solve_batch(few)
lps = [(*lpgen.dense_lp(1, 4000, seed=k), capi.LP_MAX_LE) for k in range(40)] * 100
held = torch.empty(torch.cuda.mem_get_info()[0] - (1800 << 20), dtype=torch.uint8, device="cuda")
obj, st, it, xs, ys = capi.lp_solve_batch(lps, want_xy=True)
print("threads", capi.lp_batch_stats()[3])
_check_against_oracle(lps[:40], (obj[:40], st[:40], it[:40], xs[:40], ys[:40]))
assert all(np.array_equal(xs[k], xs[k %% 40]) for k in range(len(lps)))
del held
torch.cuda.empty_cache()
capi.lp_solve_batch(lps)
print("threads", capi.lp_batch_stats()[3])
"""


def test_no_room_for_the_panels():
    """4000 LPs of 1 x 4000 take 0.5 GB, and 3 GB more for the pending rows and
    columns of the panel kernel: with 1.8 GB free they run without it."""
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-c", NO_ROOM % (os.path.dirname(here), here)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["threads", str(EVERY_PIVOT), "threads", str(PANEL)]


@pytest.mark.parametrize("kernel,shapes", [(PANEL, [(60, 50), (9, 30), (200, 40)]), (EVERY_PIVOT, [(2, 1500)] * 3)])
def test_autotune_on_either_kernel(kernel, shapes):
    """The choice names the CTA size it was timed with: the panel kernel's one
    size, or one of two."""
    lps = _lps(shapes)
    _solve(lps, kernel)
    best = capi.lp_batch_autotune(lps)
    assert best.threads in ((256,) if kernel == PANEL else (256, 512))
    _check_against_oracle(lps, capi.lp_solve_batch(lps, best, want_xy=True))
    assert capi.lp_batch_stats()[3] == best.threads
