"""Hashing of counted keys in plans of few counters: private counters over fewer items, on both
sides of each limit of that rule (counters of the plan, key range, survivors per slot, slabs),
and shared ones whose warps begin at another pair each; keys of every form, declared and
undeclared columns, an even and an odd width.  Integers: equal to the oracle."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from paper_2102_02440_gb300 import pipeline as P

pytestmark = pytest.mark.gpu


def _same(orc, tabs, d, w):
    e = list(range(sum(len(t.key_col) for t in tabs)))
    wl = G.Workload("few", tabs, [0] * len(e), [0] * len(e), d, w, 99, 7)
    dw = P.DeviceWorkload(wl)
    for t in dw.tables:
        t.counters.fill_(77)
    dw.build_batched(K.cmp_build_cfg.make(aggregate=1))
    torch.cuda.synchronize()
    dw.check_status()
    for i, (t, dt) in enumerate(zip(tabs, dw.tables)):
        ref, n = orc.build_sketch(t, dw.hash_u64, d, w)
        assert int(dw.survivors[i].item()) == n
        assert np.array_equal(dt.counters.cpu().numpy(), ref), t.name


@pytest.mark.parametrize("base", [0, 1 << 30, (1 << 45) + 3, -(1 << 19)])
@pytest.mark.parametrize("declared", [False, True])
@pytest.mark.parametrize("d,w,n,span", [
    (5, 1024, 600_000, 300_000),     # one slab, private over fewer items
    (5, 1023, 600_000, 262_144),     # at the smallest range
    (5, 1024, 600_000, 262_143),     # below it: shared
    (1, 40, 400_000, 400_000),       # a single pair
    (11, 4096, 700_000, 300_000),    # three slabs, two survivors for each slot
    (11, 4096, 500_000, 300_000),    # fewer: shared
    (12, 4096, 700_000, 300_000),    # 48 K counters, three slabs
    (13, 4096, 700_000, 300_000),    # more: the other kernel
])
def test_one_column(orc, base, declared, d, w, n, span):
    rng = np.random.default_rng(n + w)
    key = rng.integers(0, span, n).astype(np.int64)
    key[:2] = 0, span - 1
    _same(orc, [G.Table("t", [key + base], [], [0], [0], [("domain", base, base + span)] if declared else [])], d, w)


@pytest.mark.parametrize("d", [3, 5, 16])
def test_columns_of_several_tables(orc, d):
    """3 to 16 rows of 1000 counters for three columns: 9,000 to 48,000."""
    rng = np.random.default_rng(d)
    tabs = []
    for i, (n, span) in enumerate([(500_000, 300_000), (20_000, 5_000), (400_000, 1_000_000)]):
        tabs.append(G.Table(f"t{i}", [rng.integers(0, span, n).astype(np.int32)], [], [0], [i]))
    _same(orc, tabs, d, 1000)
