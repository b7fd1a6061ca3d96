"""GPU: lp_dgemm_emulated at the sizes where its kernels change or split.

Integer matrices whose products are exact in FP64 (entries below 2^10), so the
result is numpy's bit for bit, on either side of the sizes where the row
exponents of B go from a warp to a block per row (256 columns; a row for each
eight SMs' warps), and where its results, exchanged between the lanes of a warp
so that 16 columns of a row are written together, end inside such a piece.
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


@pytest.mark.parametrize("K", [1, 64, 65, 449])
@pytest.mark.parametrize("M", [1, 15, 16, 17, 31, 33, 127, 129])
def test_ragged_results_and_pitches(M, K):
    """Results of every width around a piece, a warp's columns and a tile, in a
    matrix with a longer pitch that starts 8 bytes off a 16-byte boundary: the
    entries around them keep their bits."""
    lib = capi.load_library()
    rng = np.random.default_rng(M + K)
    A = _ints(rng, M, K)
    tA = torch.from_numpy(A).cuda()
    for N in (1, 15, 16, 17, 47, 63, 64, 65, 130):
        B = _ints(rng, K, N)
        tB = torch.from_numpy(B).cuda()
        for pitch in (N, N + 3):
            mem = torch.full((M * pitch + 10,), np.nan, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            assert lib.lp_dgemm_emulated(M, N, K, tA.data_ptr(), K, tB.data_ptr(), N,
                                         mem.data_ptr() + 40, pitch, None) == 0
            got = mem.cpu().numpy()
            want = np.full(M * pitch + 10, np.nan)
            np.lib.stride_tricks.as_strided(want[5:], (M, N), (8 * pitch, 8))[:] = A @ B
            assert np.array_equal(got, want, equal_nan=True)
