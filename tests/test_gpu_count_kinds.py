"""Every kind of counted table in one build: presence columns, whole tables, row samples, samples
with predicates and predicates, each counted by its own launch from its own chunk counter; with
unique-key columns beside the counting pass and without (a split pass).  Counters and survivor
counts equal the oracle's; integers, no tolerance."""
import itertools

import numpy as np
import pytest
import torch

from oracle import sample as S
from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from paper_2102_02440_gb300 import pipeline as P

pytestmark = pytest.mark.gpu

KINDS = ["presence", "whole", "sample", "sample_pred", "pred"]


def _table(rng, kind, n, edge):
    fk = G.zipf_keys(rng, n, 3000, 1.0)
    p = rng.integers(0, 1000, n).astype(np.int32)
    preds = [G.Pred(1, G.RANGE, 0, 300)]
    if kind == "presence":
        return G.Table(kind, [rng.permutation(2 * n)[:n].astype(np.int32), fk], [], [0, 1], [edge, edge + 1],
                       [("unique", 0, 2 * n), ("domain", 0, 3000)])
    if kind == "unique":
        return G.Table(kind, [rng.permutation(n).astype(np.int32), p], preds, [0], [edge], [("unique", 0, n), None])
    return G.Table(kind, [fk, p], preds if kind.endswith("pred") else [], [0], [edge], [("domain", 0, 3000), None])


@pytest.mark.parametrize("unique", [False, True])
@pytest.mark.parametrize("leave_out", [None, *KINDS])
@pytest.mark.parametrize("rows", [5000, 70_001])
def test_kinds_together(orc, rows, leave_out, unique):
    rng = np.random.default_rng(rows)
    tabs, edge = [], 0
    for kind, _ in itertools.product([k for k in KINDS if k != leave_out] + ["unique"] * unique, range(2)):
        tabs.append(_table(rng, kind, rows + len(tabs), edge))
        edge += len(tabs[-1].key_col)
    wl = G.Workload("kinds", tabs, [0] * edge, [0] * edge, 3, 256, 99, 7)
    rates = [0.2 if t.name.startswith("sample") else 1.0 for t in tabs]
    dw = P.DeviceWorkload(wl, sample_rates=rates, sample_seed=11)
    for t in dw.tables:
        t.counters.fill_(77)
    for _ in range(2):  # (the workspace of the first build is the second one's)
        dw.build_batched(K.cmp_build_cfg.make(aggregate=1))
        torch.cuda.synchronize()
        dw.check_status()
        surv = dw.survivors.cpu().numpy()
        for i, (t, dt) in enumerate(zip(tabs, dw.tables)):
            ref, m = orc.build_sketch(S.sampled_table(t, 11 + i, rates[i]) if rates[i] < 1 else t, dw.hash_u64, 3, 256)
            assert int(surv[i]) == m, t.name
            assert np.array_equal(dt.counters.cpu().numpy(), ref), t.name
