"""Which cycles have their own kernel: the plan's count on both sides of the limits (four tables,
seven conditioning chunks, the widest sketch), and rows that it must have taken, because
their value is 0 while the terms of the generic path are beyond int128."""
import ctypes as C

import numpy as np
import pytest
import torch

from host_probe import compile_probe
from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import pipeline as P
from test_gpu_wide import _fill, _one_row_tables, _run

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "estimate.cuh"
extern "C" int64_t cycles(const void* plan) { return static_cast<const cmpk::EstPlanHdr*>(plan)->n_cyc; }
"""


@pytest.fixture(scope="module")
def cycles(tmp_path_factory):
    f = compile_probe(tmp_path_factory.mktemp("probe"), SOURCE).cycles
    f.restype, f.argtypes = C.c_int64, [C.c_void_p]
    return f


@pytest.mark.parametrize("n,w,chunk,flags,want", [
    (4, 64, 8, 0, 1), (4, 63, 9, 0, 0), (4, 64, 9, 0, 1), (4, 448, 0, 0, 0), (4, 449, 0, 0, 1), (5, 4096, 0, 0, 1),
    (4, 4097, 0, 0, 0), (3, 1024, 0, 0, 0), (4, 1024, 256, 0, 0), (4, 1024, 0, K.CMP_EST_GENERIC_ONLY, 0),
    (4, 1024, 0, K.CMP_EST_CACHE_MESSAGES, 1)])
def test_plans_hold_the_cycles(cycles, n, w, chunk, flags, want):
    dw = _one_row_tables(list(range(n)), [(i + 1) % n for i in range(n)], n, 2, w)
    est = P.DeviceEstimator(dw, [(1 << n) - 1, 0b11], cfg=K.cmp_estimate_cfg.make(flags=flags, cond_chunk=chunk))
    assert cycles(est.plan_host.ctypes.data) == want


def test_rows_whose_terms_alone_leave_int128(cycles):
    """Every sketch 2^31 - 1, but one of +-(2^31 - 2) in equal numbers: the smaller magnitude is
    the merged value of its table, so every row estimate is 0.  Each conditioning value's own
    term is about 2^154 when that sketch is on the conditioned edge."""
    n, w, big = 4, 1024, 2**31 - 1
    eu, ev = [0, 1, 2, 0], [1, 2, 3, 3]
    beyond = 0
    for e in range(n):
        dw = _one_row_tables(eu, ev, n, 2, w)
        _fill(dw, lambda s: np.full(s, big))
        t, k = dw.wl.sketch_of(e, 0)
        alternating = (torch.arange(w, device="cuda", dtype=torch.int32) % 2 * 2 - 1) * (big - 1)
        dw.tables[t].counters[k] = alternating
        est, st = _run(dw, [0b1111], flags=K.CMP_EST_NO_WIDE)
        assert cycles(est.plan_host.ctypes.data) == 1
        assert st == 0 and float(est.est[0]) == 0.0 and est.row_values()[0] == [0, 0]
        gen, st = _run(dw, [0b1111], flags=K.CMP_EST_NO_WIDE | K.CMP_EST_GENERIC_ONLY)
        beyond += st == K.CMP_EOVERFLOW and bool(np.isnan(float(gen.est[0])))
    assert beyond > 0  # the generic path cannot have given those zeros
