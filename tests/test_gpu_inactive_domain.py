"""Declared key domains that the counting pass turns down, where the domain does not start at a
multiple of four or comes after a column with another smallest key: one surviving key outside
the domain, and no surviving row at all (three predicates: the general selection).  Counters
and survivor counts equal the oracle's; integers, no tolerance."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from paper_2102_02440_gb300 import pipeline as P

pytestmark = pytest.mark.gpu


def _before(rng, n, edge):
    """An int64 column of small odd keys (smallest 7)."""
    key = 7 + 2 * rng.integers(0, 400, n)
    key[0] = 7
    return G.Table("before", [key.astype(np.int64)], [], [0], [edge])


def _turned_down(rng, n, edge, kind, base):
    key = (rng.integers(0, 900, n) + base).astype(np.int64)
    meta = ("domain", base, base + 900)
    if kind == "outside":
        key[n // 2] = base + 900
        return G.Table("outside", [key], [], [0], [edge], [meta])
    p = [rng.integers(0, 1000, n).astype(np.int32) for _ in range(3)]
    preds = [G.Pred(1, G.RANGE, 0, 500), G.Pred(2, G.RANGE, 0, 500), G.Pred(3, G.RANGE, 2000, 3000)]
    return G.Table("none", [key, *p], preds, [0], [edge], [meta, None, None, None])


@pytest.mark.parametrize("w", [256, 1000])
@pytest.mark.parametrize("base", [5, 6, 7, 8])
@pytest.mark.parametrize("kind", ["outside", "none"])
@pytest.mark.parametrize("alone", [True, False])
def test_turned_down_domains(orc, kind, base, w, alone):
    rng = np.random.default_rng(base)
    n = 3001
    tabs = [] if alone else [_before(rng, n, 0)]
    tabs.append(_turned_down(rng, n, len(tabs), kind, base))
    if not alone:
        tabs.append(_before(rng, n, len(tabs)))  # a column after it is hashed as ever
    e = list(range(len(tabs)))
    wl = G.Workload("down", tabs, [0] * len(e), [0] * len(e), 3, w, 99, 7)
    dw = P.DeviceWorkload(wl)
    for t in dw.tables:
        t.counters.fill_(77)
    dw.build_batched(K.cmp_build_cfg.make(aggregate=1))
    torch.cuda.synchronize()
    dw.check_status()
    surv = dw.survivors.cpu().numpy()
    for i, (t, dt) in enumerate(zip(tabs, dw.tables)):
        ref, m = orc.build_sketch(t, dw.hash_u64, 3, w)
        assert int(surv[i]) == m, t.name
        assert np.array_equal(dt.counters.cpu().numpy(), ref), t.name
