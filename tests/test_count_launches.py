"""The counting pass's launches as a plan lays them out, on the host: the one that the presence-
bitmap or the unique-key kernel runs beside has one CTA per SM, the others that select rows
have two."""
import ctypes as C

import numpy as np
import pytest

from host_probe import compile_probe

SOURCE = r"""
#include "internal.cuh"
extern "C" void fields(const void* plan, int64_t* out) {
  const cmpk::BuildPlanHdr& h = *static_cast<const cmpk::BuildPlanHdr*>(plan);
  for (int k = 0; k < 4; k++) out[k] = h.cnt_grid[k];
  out[4] = h.cnt_split;
}
"""
SMS = 152
ROWS = 40_000_000


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    from paper_2102_02440_gb300 import build_lib, compass as K
    build_lib.build()
    probe = compile_probe(tmp_path_factory.mktemp("probe"), SOURCE)

    def run(kinds):
        tabs = []
        for kind in kinds:
            uniq = kind in ("presence", "unique")
            flags = K.CMP_COL_DOMAIN | (K.CMP_COL_UNIQUE if uniq else 0)
            cols = (K.cmp_col * 2)(K.cmp_col(0x1000, 0, flags, 0, ROWS if uniq else 1_000_000), K.cmp_col(0x2000, 0, 0, 0, 0))
            preds = (K.cmp_pred * 1)(K.cmp_pred(1, 0, 0, 100, None, 0))
            n_preds = 1 if kind in ("predicates", "unique") else 0
            key, edge = (C.c_int32 * 1)(0), (C.c_int32 * 1)(0)
            t = K.cmp_table(ROWS, 2, n_preds, 1, 0, cols, preds, key, edge, 7, 0.1 if kind == "sample" else 0.0)
            t._keep = (cols, preds, key, edge)
            tabs.append(t)
        n, _ = K.cmp_build_plan_bytes(tabs, 11, 4096, None)
        buf = np.zeros(n, np.uint8)
        K.cmp_build_plan_encode(tabs, 11, 4096, 1, [0x3000] * len(tabs), 0x4000, None, buf.ctypes.data, n)
        out = (C.c_int64 * 5)()
        probe.fields(C.c_void_p(buf.ctypes.data), out)
        return list(out[:4]), out[4]
    return run


@pytest.mark.parametrize("kinds,grids", [
    (("presence", "whole"), (2, 1, 0, 0)),
    (("presence", "predicates"), (2, 0, 0, 1)),
    (("presence", "whole", "sample"), (2, 1, 1, 0)),
    (("presence", "whole", "sample", "predicates"), (2, 1, 2, 1)),
    (("unique", "whole"), (0, 1, 0, 0)),
    (("unique", "predicates"), (0, 0, 0, 1)),
    (("unique", "sample", "predicates"), (0, 0, 1, 2)),
    (("unique", "whole", "sample", "predicates"), (0, 1, 2, 2)),
    (("unique", "presence", "whole", "predicates"), (0, 1, 0, 2)),
    (("whole", "sample", "predicates"), (0, 2, 2, 2)),
    (("presence",), (0, 2, 0, 0)),
])
def test_ctas_per_sm_of_each_launch(plan, kinds, grids):
    got, split = plan(kinds)
    assert got == [g * SMS for g in grids]
    assert (split > 0) == (kinds[0] == "presence" and len(kinds) > 1)

