"""GPU: request inputs copied by helper threads, at the sizes where the copy splits.

From 1 MB the rows of A are copied in pieces of 256 KB by the submitting
thread and the server's helpers; below that by the submitting thread alone.
Shapes lie close to either side of the threshold, on whole pieces and off them, and come from one or three submitting threads; the caller's array is
overwritten as soon as the submission returns.
"""
import threading

import numpy as np
import pytest

import oracle
from paper_1804_04737_gb300 import capi, lpgen
from test_gpu_serve import _check, _lib  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu

SHAPES = [(510, 257), (257, 510), (256, 512), (512, 256), (257, 511), (512, 320), (700, 701)]


@pytest.mark.parametrize("clients", [1, 3])
@pytest.mark.parametrize("lanes", [0, 3])
def test_copied_inputs_match_oracle(lanes, clients):
    lps = [(*lpgen.dense_lp(m, n, seed=m), capi.LP_MAX_LE) for m, n in SHAPES]
    srv = capi.lp_server_create(capi.lp_options_default(lanes=lanes), hbm_budget_bytes=4 << 30,
                                max_slots=32)
    got, errs = {}, []

    def client(j):
        try:
            mine = [(j, k) for k in range(len(lps))][j:] + [(j, k) for k in range(j)]
            tickets = []
            for key in mine:
                A, b, c, sense = lps[key[1]]
                A = A.copy()
                tickets.append(capi.lp_server_submit(srv, A, b, c, sense))
                A.fill(np.nan)
            for key, t in zip(mine, tickets):
                got[key] = capi.lp_server_wait(srv, t, *lps[key[1]][0].shape)
        except Exception as e:  # noqa: BLE001
            errs.append(e)

    try:
        ths = [threading.Thread(target=client, args=(j,)) for j in range(clients)]
        [t.start() for t in ths]
        [t.join() for t in ths]
        assert not errs
    finally:
        capi.lp_server_destroy(srv)
    assert len(got) == clients * len(lps)
    for (_, k), res in got.items():
        _check(lps[k], res)
