"""GPU: loads where the device, or a server's slice of its arena, has room for the
tableau but not for the second buffer of the overlapped panels: the panels run in
turn, with the same bits."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_1804_04737_gb300 import capi, lpgen
from paper_1804_04737_gb300.build import build_library

pytestmark = pytest.mark.gpu

TIGHT = """
import sys
sys.path.insert(0, %r)
import numpy as np
import torch
from paper_1804_04737_gb300 import capi
g = torch.Generator(device="cuda")
g.manual_seed(1)
ints = lambda lo, hi, s: torch.randint(lo, hi, s, generator=g, device="cuda").to(torch.float64)
n = 5000
A, b, c = (t.cpu() for t in (ints(1, 1001, (n, n)), ints(1000, 100001, (n,)), ints(1, 101, (n,))))
torch.cuda.empty_cache()
def solve():
    h = capi.lp_create(capi.lp_options_default(max_iters=120))
    capi.lp_load(h, A, b, c, capi.LP_MAX_LE)
    capi.lp_solve(h)
    x, y = np.empty(n), np.empty(n)
    r = capi.lp_result(h, x, y)
    capi.lp_destroy(h)
    return x, y, r
small = capi.solve(A[:700, :900].contiguous(), b[:700].contiguous(), c[:900].contiguous())
want = solve()
held = torch.empty(torch.cuda.mem_get_info()[0] - (900 << 20), dtype=torch.uint8, device="cuda")
got = solve()
assert want[2] == got[2], (want[2], got[2])
assert all(np.array_equal(a.view(np.uint64), w.view(np.uint64)) for a, w in zip(got[:2], want[:2]))
print("same")
"""


def test_room_for_the_tableau_only():
    """5000 x 5000: 0.2 GB of inputs and 0.4 of tableau with 0.9 free."""
    build_library()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", TIGHT % root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == ["same"]


@pytest.mark.parametrize("mib", [26, 30, 40, 60, 90, 150])
def test_lanes_of_small_slices(mib):
    """LPs of overlapped size (7.9 MB of tableau, 4.8 of inputs) on three lanes: a
    slice of the budget holds none of them, the tableau alone, or both buffers."""
    build_library()
    capi.load_library()
    oracle.set_threads(os.cpu_count() or 1)
    lps = [(*lpgen.dense_lp(600, 1000, seed=k), capi.LP_MAX_LE) for k in range(4)]
    lps += [(*lpgen.dual_of(*lpgen.dense_lp(1000, 600, seed=k)), capi.LP_MIN_GE) for k in range(2)]
    srv = capi.lp_server_create(capi.lp_options_default(), hbm_budget_bytes=mib << 20, max_slots=16)
    try:
        tickets = [capi.lp_server_submit(srv, *lp) for lp in lps]
        got = [capi.lp_server_wait(srv, t, *lp[0].shape) for t, lp in zip(tickets, lps)]
    finally:
        capi.lp_server_destroy(srv)
        oracle.set_threads(1)
    for (A, b, c, sense), (obj, st, it, x, y, *_) in zip(lps, got):
        o = oracle.solve(A, b, c, sense=sense)
        assert st == o.status and it == o.iters and obj == o.obj
        assert np.array_equal(x.view(np.uint64), o.x.view(np.uint64))
        assert np.array_equal(y.view(np.uint64), o.y.view(np.uint64))
