"""lp_batch_autotune's file, on the CPU: a choice is taken only for the kernel it
was timed on.  (Without a device, a call that finds no choice fails.)"""
import ctypes

import numpy as np
import pytest

from paper_1804_04737_gb300 import capi
from paper_1804_04737_gb300.build import build_library


def _signature(shapes):
    h = 1469598103934665603
    for v in sorted((m << 32) | n for m, n in shapes):
        for i in range(8):
            h = ((h ^ ((v >> (8 * i)) & 0xff)) * 1099511628211) % (1 << 64)
    return h


def _tune(shapes, path, precision):
    lib = capi.load_library()
    m, n = (np.array(v, dtype=np.int32) for v in zip(*shapes))
    none = (ctypes.c_void_p * len(shapes))()
    o, best = capi.lp_options_default(precision=precision), capi.lp_options_default()
    e = lib.lp_batch_autotune(len(shapes), m.ctypes.data, n.ctypes.data, none, none, none, None,
                              ctypes.byref(o), str(path).encode(), ctypes.byref(best))
    return (best.group_elems, best.threads) if e == 0 else None


# (rows and columns of which no CTA's slice fits the panel kernel's shared memory: the last)
@pytest.mark.parametrize("precision,prec", [(capi.LP_FP64, "fp64"), (capi.LP_FP32_REINV, "fp32")])
@pytest.mark.parametrize("shapes,panel", [([(30, 20), (5, 7)], True), ([(30, 20), (5, 70000)], False)])
def test_a_choice_is_the_kernels_own(tmp_path, shapes, panel, precision, prec):
    build_library()
    tail = "c%d-%016x" % (len(shapes), _signature(shapes))
    f = tmp_path / "tune.txt"
    f.write_text("fp64-%s 65536 512 8.9000\n" % tail)
    assert _tune(shapes, f, precision) == (None if panel else (65536, 512))
    with open(f, "a") as out:
        out.write("panel-%s-%s 262144 256 5.8000\n" % (prec, tail))
    assert _tune(shapes, f, precision) == (262144, 256)
