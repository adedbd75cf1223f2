"""Simple cycles of four or more tables on their own kernel (product vectors of the distinct
values of one sketch, multi-limb integers): every row equal to the oracle's, for ties, zeros,
both signs, INT32_MIN, values of a few bits to beyond int128, edges listed in any order and
direction; rows whose bound needs more limbs than the kernel has keep the generic path.
Larger widths against the generic evaluation."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from test_gpu_wide import _fill, _one_row_tables, _oracle, _run

pytestmark = pytest.mark.gpu

FILLS = {
    "ties": lambda rng: (lambda s: rng.integers(-2, 3, s)),
    "zeros": lambda rng: (lambda s: rng.integers(-9, 10, s) * (rng.random(s) < 0.1)),
    "small": lambda rng: (lambda s: np.rint(rng.standard_t(2, s) * 20).clip(-2**20, 2**20)),
    "mid": lambda rng: (lambda s: rng.integers(-2**20, 2**20, s)),
    "big": lambda rng: (lambda s: rng.choice(np.array([-2**31, 2**31 - 1, -2**31 + 1, 7, -7, 0]), s)),
    "constant": lambda rng: (lambda s: np.full(s, -3)),
}


def _cycle(n, rng):
    """A cycle over tables 0..n-1 in a random order, its edges shuffled, ends swapped at random."""
    order = rng.permutation(n)
    edges = [(int(order[i]), int(order[(i + 1) % n])) for i in range(n)]
    edges = [e if rng.random() < 0.5 else e[::-1] for e in edges]
    rng.shuffle(edges)
    return [u for u, _ in edges], [v for _, v in edges]


@pytest.mark.parametrize("n,w,chunk,fill", [(4, 64, 8, "small"), (4, 61, 7, "ties"), (5, 64, 8, "zeros"),
                                            (5, 57, 8, "constant"), (6, 64, 4, "mid"), (9, 64, 8, "mid"),
                                            (4, 64, 8, "big"), (8, 33, 4, "big"), (12, 64, 8, "big"),
                                            (13, 40, 5, "small")])
def test_cycle_rows_match_oracle(orc, n, w, chunk, fill):
    rng = np.random.default_rng(n * 1000 + w)
    eu, ev = _cycle(n, rng)
    dw = _one_row_tables(eu, ev, n, 3, w)
    _fill(dw, FILLS[fill](rng))
    masks = [(1 << n) - 1]
    refs = _oracle(orc, dw, masks)
    for flags in (0, K.CMP_EST_CACHE_MESSAGES):
        est, st = _run(dw, masks, flags=flags, cond_chunk=chunk)
        assert st == 0
        assert est.wide_values()[0] == refs[0].rows
        assert float(est.est[0]) == refs[0].est
    # without the exact tier: the same rows while they stay in int128, else NaN and the status
    est, st = _run(dw, masks, flags=K.CMP_EST_NO_WIDE, cond_chunk=chunk)
    if all(-2**127 <= r < 2**127 for r in refs[0].rows) and fill in ("ties", "zeros", "small", "constant"):
        assert st == 0 and float(est.est[0]) == refs[0].est
    elif any(not -2**127 <= r < 2**127 for r in refs[0].rows):
        assert st == K.CMP_EOVERFLOW and np.isnan(float(est.est[0]))


@pytest.mark.parametrize("n,w", [(4, 449), (5, 1023), (4, 1024), (7, 1024), (4, 2049), (4, 4095), (4, 4097)])
def test_cycle_rows_match_generic_path(n, w):
    rng = np.random.default_rng(w)
    eu, ev = _cycle(n, rng)
    dw = _one_row_tables(eu, ev, n, 2, w)
    _fill(dw, FILLS["small"](rng))
    masks = [(1 << n) - 1]
    a, st_a = _run(dw, masks)
    b, st_b = _run(dw, masks, flags=K.CMP_EST_GENERIC_ONLY)
    assert st_a == st_b == 0 and a.wide_values() == b.wide_values()
    assert torch.equal(a.est, b.est)
