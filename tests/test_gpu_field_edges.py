"""Hash functions whose folded sums meet the field's edges: coefficients 0, 1, p - 2 and p - 1 on
keys next to the multiples of p, 2^31 and the ends of int64, where a sum is p itself, or one
more or less, through every kernel that hashes keys of 2^31 and more.  Equal to the oracle."""
import itertools

import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from paper_2102_02440_gb300 import pipeline as P

pytestmark = pytest.mark.gpu

p = (1 << 61) - 1


def _params():
    """16 rows of (a, b, c0, c1, c2, c3)."""
    rows = list(itertools.product((1, p - 1), (0, 1, p - 1)))
    out = []
    for i in range(16):
        a, b = rows[i % len(rows)]
        out.append((a, b, (0, 1, p - 1, p - 2)[i % 4], (0, 1, p - 1)[i % 3], (0, p - 1)[i % 2], (0, 0, 1, p - 1, p - 2)[i % 5]))
    return np.array(out, np.uint64).reshape(1, 16, 6)


@pytest.mark.parametrize("w", [512, 500, 40_000])
@pytest.mark.parametrize("cfg", [dict(aggregate=0, unique=-1), dict(aggregate=0, unique=-1, mode=1, pairs_per_slab=1),
                                 dict(aggregate=1, unique=-1), dict()])
def test_sums_at_the_edges_of_the_field(orc, w, cfg):
    near = [k for m in (p, 2 * p, 3 * p, -p, -2 * p, 0, 1 << 31, 1 << 62, (1 << 63) - 1, -(1 << 63)) for k in range(m - 4, m + 5)
            if -(1 << 63) <= k < 1 << 63]
    near = np.unique(np.array(near, np.int64))
    hp = _params()
    wl = G.Workload("edges", [G.Table("all", [np.tile(near, 40)], [], [0], [0])] +
                    [G.Table(f"one {k}", [np.arange(k - 4, k + 5)], [], [0], [0], [("unique", k - 4, k + 5)])
                     for k in (p, -p, 2 * p, 1 << 31)], [0], [0], 16, w, 1, 1)
    dw = P.DeviceWorkload(wl)
    dw.hash_u64 = hp
    dw.hash_dev.copy_(torch.from_numpy(hp.reshape(-1).view(np.int64)))
    dw.build_batched(K.cmp_build_cfg.make(**cfg))
    torch.cuda.synchronize()
    dw.check_status()
    for t, dt in zip(wl.tables, dw.tables):
        ref, n = orc.build_sketch(t, hp, 16, w)
        assert np.array_equal(dt.counters.cpu().numpy(), ref), t.name
