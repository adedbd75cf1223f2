"""Keys on both sides of 2^31, where the hash arithmetic changes form, through every kernel
that hashes keys (the per-row build, the unique-key kernel with int32 and 16-bit counters,
the hashing pass of counted keys, the partition build), for widths that are and are not powers
of two; and the hashing pass's reading of the count array: key ranges that start at any slot
of a four-slot load, wrap around a masked array, end inside a load, fill a batch exactly, or
hold one key in thousands of slots.  Integers: equal to the oracle, no tolerance."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from paper_2102_02440_gb300 import pipeline as P

pytestmark = pytest.mark.gpu


def _check(orc, tabs, cfg, d=5, w=512):
    ne = 1 + max((e for t in tabs for e in t.edge_id), default=0)
    wl = G.Workload("small", tabs, [0] * ne, [0] * ne, d, w, 31337, 3)
    dw = P.DeviceWorkload(wl)
    dw.build_batched(cfg)
    torch.cuda.synchronize()
    dw.check_status()
    surv = dw.survivors.cpu().numpy()
    for i, (t, dt) in enumerate(zip(tabs, dw.tables)):
        ref, n = orc.build_sketch(t, dw.hash_u64, d, w)
        assert int(surv[i]) == n
        assert np.array_equal(dt.counters.cpu().numpy(), ref), t.name


@pytest.mark.parametrize("w", [512, 500, 40_000])
@pytest.mark.parametrize("cfg", [dict(aggregate=0, unique=-1), dict(aggregate=0, unique=-1, mode=1, pairs_per_slab=1),
                                 dict(aggregate=1), dict()])
def test_keys_around_the_limit_of_the_small_form(orc, w, cfg):
    rng = np.random.default_rng(w)
    n = 4099
    tabs = []
    for mid in (0, 1 << 29, (1 << 31) - 1, 1 << 31, 1 << 32, (1 << 61) - 2, -(1 << 31), -(1 << 62)):
        pk = rng.permutation(n).astype(np.int64) - n // 2 + mid
        tabs.append(G.Table(f"i64 {mid}", [pk], [], [0], [len(tabs)], [("unique", int(pk.min()), int(pk.max()) + 1)]))
        tabs.append(G.Table(f"fk {mid}", [rng.choice(pk, n)], [], [0], [len(tabs)]))
    hi = ((1 << 31) - 1 - rng.permutation(n)).astype(np.int32)
    tabs.append(G.Table("i32 top", [hi], [], [0], [len(tabs)], [("unique", int(hi.min()), 1 << 31)]))
    tabs.append(G.Table("i32 top fk", [rng.choice(hi, n), rng.choice(hi, n)], [], [0, 0, 1], [0, 1, 2]))
    if w == 40_000:
        tabs = tabs[4:8] + tabs[-2:]
    _check(orc, tabs, K.cmp_build_cfg.make(**cfg), w=w)


@pytest.mark.parametrize("first", [0, 1, 2, 3, 4093, (1 << 31) - 2500, -1234])
def test_count_array_ranges(orc, first):
    rng = np.random.default_rng(abs(first) + 1)
    tabs = []

    def add(name, key, meta=None):
        tabs.append(G.Table(name, [key.astype(np.int64)], [], [0], [len(tabs)], [meta] if meta else []))
    for span in (1, 2, 127, 128, 129, 2047, 2049):
        add(f"all {span}", np.concatenate([np.arange(span), rng.integers(0, span, 2500)]) + first)
    add("sparse", rng.choice(200_000, 40, replace=False).repeat(90) + first, ("domain", first - 3, first + 200_001))
    add("ends", np.array([0, 199_999]).repeat(2000) + first, ("domain", first, first + 200_000))
    _check(orc, tabs, K.cmp_build_cfg.make(aggregate=1))
