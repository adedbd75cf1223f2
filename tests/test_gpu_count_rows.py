"""Counting of tables without a selection: counters and survivor counts equal the oracle bit
for bit at the edges of the kernel's loads (columns that start off a 16-byte boundary, rows
before and after the last whole load, fewer rows than one load), for both key types, domains
that end at or beyond int32, more key columns than hot-key caches, a key outside its declared
domain, and tables on both sides of the smallest aggregated size.  Integers: no tolerance."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from paper_2102_02440_gb300 import pipeline as P

pytestmark = pytest.mark.gpu


def _tables(rng, rows):
    I32 = np.iinfo(np.int32)
    cols = [
        (G.zipf_keys(rng, rows, 900, 1.1), None),
        (G.zipf_keys(rng, rows, 900, 0.7), ("domain", 0, 900)),
        ((rng.integers(0, 700, rows) + (I32.max - 699)).astype(np.int32), ("domain", I32.max - 699, I32.max + 1)),
        ((rng.integers(0, 700, rows) + I32.min).astype(np.int32), ("domain", I32.min - 50, I32.min + 700)),
        (rng.integers(0, 5000, rows).astype(np.int64) - (1 << 40), ("domain", -(1 << 40), 5000 - (1 << 40))),
        (rng.integers(0, 300, rows).astype(np.int64) + (1 << 50), None),
    ]
    return [c for c, _ in cols], [m for _, m in cols]


def _check(orc, tabs, cfg, shift, d=3, w=256):
    eu = [0] * sum(len(t.key_col) for t in tabs)
    wl = G.Workload("count", tabs, eu, list(eu), d, w, 99, 7)
    # columns `shift` elements into their buffers
    cols = [[torch.cat([torch.zeros(shift, dtype=torch.from_numpy(c).dtype), torch.from_numpy(c)]).cuda()[shift:]
             for c in t.cols] for t in tabs]
    dw = P.DeviceWorkload(wl, cols_dev=cols)
    dw.build_batched(cfg)
    torch.cuda.synchronize()
    dw.check_status()
    surv = dw.survivors.cpu().numpy()
    for i, (t, dt) in enumerate(zip(tabs, dw.tables)):
        ref, n = orc.build_sketch(t, dw.hash_u64, d, w)
        assert int(surv[i]) == n
        assert np.array_equal(dt.counters.cpu().numpy(), ref), (t.name, shift)


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("rows", [1, 3, 7, 2049, 16385, 70_001])
def test_rows_before_and_after_whole_loads(orc, rows, shift):
    rng = np.random.default_rng(rows * 4 + shift)
    cols, meta = _tables(rng, rows)
    edges = list(range(len(cols)))
    _check(orc, [G.Table("t", cols, [], edges, edges, meta)], K.cmp_build_cfg.make(aggregate=1), shift)


def test_presence_beside_counts_and_a_key_outside_its_domain(orc):
    rng = np.random.default_rng(5)
    n = 40_003
    bad = G.zipf_keys(rng, n, 900, 1.0)
    bad[n - 1] = 900  # the last row, counted with the rows after the last whole load
    pk = (rng.permutation(2 * n)[:n] - 17).astype(np.int32)
    tabs = [G.Table("pk", [pk, G.zipf_keys(rng, n, 900, 1.0)], [], [0, 1], [0, 1], [("unique", -17, 2 * n - 17), None]),
            G.Table("bad", [bad], [], [0], [2], [("domain", 0, 900)])]
    _check(orc, tabs, K.cmp_build_cfg.make(aggregate=1), 1)


def test_both_sides_of_the_smallest_aggregated_table(orc):
    rng = np.random.default_rng(6)
    tabs = []
    for n in (8191, 8192, 8193, (1 << 18) - 1, 1 << 18):
        for dom in (16 * n, 16 * n + 1):
            e = len(tabs)
            key = rng.integers(0, dom, n).astype(np.int32)
            tabs.append(G.Table(f"n{n}", [key], [], [0], [e], [("domain", 0, dom)]))
    # keys far sparser than the rows, without a declared domain: per row when the array is too small
    for span in (1 << 16, 1 << 26):
        tabs.append(G.Table("sparse", [rng.integers(0, span, 9000).astype(np.int32)], [], [0], [len(tabs)]))
    _check(orc, tabs, None, 0)


@pytest.mark.parametrize("rate", [1e-4, 0.1, 0.5, 0.999])
@pytest.mark.parametrize("rows", [1, 31, 33, 2047, 70_001])
def test_sampled_rows(orc, rows, rate):
    """A row sample without predicates: few, some and nearly all rows kept per warp and buffer; the
    reference is the oracle over the rows the oracle's sampler picks."""
    from oracle import sample as S
    rng = np.random.default_rng(rows)
    cols, meta = _tables(rng, rows)
    edges = list(range(len(cols)))
    tab = G.Table("s", cols, [], edges, edges, meta)
    wl = G.Workload("count", [tab], [0] * 6, [0] * 6, 3, 256, 99, 7)
    dw = P.DeviceWorkload(wl, sample_rates=[rate], sample_seed=11)
    dw.build_batched(K.cmp_build_cfg.make(aggregate=1))
    torch.cuda.synchronize()
    dw.check_status()
    ref, n = orc.build_sketch(S.sampled_table(tab, 11, rate), dw.hash_u64, 3, 256)
    assert int(dw.survivors.cpu()[0]) == n
    assert np.array_equal(dw.tables[0].counters.cpu().numpy(), ref)


@pytest.mark.parametrize("domain", [True, False])
@pytest.mark.parametrize("n_tables", [10, 13])
@pytest.mark.parametrize("large", [False, True])
def test_small_tables_on_both_sides_of_the_work_they_need(orc, n_tables, domain, large):
    """10 tables of 120,000 keys for 12 sketch rows need fewer than 2^24 evaluations, 13 more."""
    rng = np.random.default_rng(n_tables)
    tabs = [G.Table(f"t{i}", [rng.integers(0, 9000, 120_000).astype(np.int32)], [], [0], [i],
                    [("domain", 0, 9000)] if domain else []) for i in range(n_tables)]
    if large:
        tabs.append(G.Table("large", [rng.integers(0, 9000, 1 << 18).astype(np.int32)], [], [0], [n_tables]))
    _check(orc, tabs, None, 0, d=12, w=128)
