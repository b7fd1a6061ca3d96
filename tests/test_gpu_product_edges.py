"""GPU: lp_dgemm_emulated at the sizes where its kernels change or split.

Integer matrices whose products are exact in FP64 (entries below 2^10), so the
result is numpy's bit for bit, on either side of the sizes where the row
exponents of B go from a warp to a block per row (256 columns; a row for each
eight SMs' warps).
"""
import ctypes

import numpy as np
import pytest

from paper_1804_04737_gb300 import capi
from paper_1804_04737_gb300.build import build_library

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_library()
    capi.load_library()


def _ints(rng, m, n):
    return rng.integers(-1000, 1001, size=(m, n)).astype(np.float64)


@pytest.mark.parametrize("N", [255, 256, 257, 513])
@pytest.mark.parametrize("K", [1, 16, 1215, 1216, 1217])
def test_row_exponents(N, K):
    rng = np.random.default_rng(N + K)
    A, B = _ints(rng, 40, K), _ints(rng, K, N)
    B *= 2.0 ** rng.integers(-8, 9, size=(1, N))  # (every sum stays exact)
    C = torch.empty((40, N), dtype=torch.float64, device="cuda")
    capi.lp_dgemm_emulated(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C)
    assert np.array_equal(C.cpu().numpy(), A @ B)
