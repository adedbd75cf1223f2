"""The star lattice on residues: every tile shape (2 to 12 free leaf bits, blocks beyond), ragged
chunks of 16 sorted positions, one to five primes and the int128 evaluation beyond them, zeros,
signs and INT32_MIN, entries beyond int128.  Rows against the generic evaluation (both exact, the
exact tier on), the smaller families against the oracle too."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from test_gpu_wide import _fill, _one_row_tables, _oracle, _run

pytestmark = pytest.mark.gpu


def _magnitudes(rng, bits):
    def fn(shape):
        if bits == 31:
            return rng.choice(np.array([-2**31, 2**31 - 1, 1, -1, 0, 12345]), shape)
        a = rng.integers(-2**bits, 2**bits + 1, shape)
        return a * (rng.random(shape) < 0.9)
    return fn


@pytest.mark.parametrize("leaves,w,bits", [(3, 1, 31), (3, 17, 2), (4, 16, 7), (5, 33, 12), (6, 40, 20), (7, 113, 3),
                                           (7, 16, 31), (8, 129, 1), (9, 15, 9), (10, 64, 5), (11, 31, 2),
                                           (12, 17, 1), (13, 16, 3), (14, 20, 1)])
def test_lattice_rows_match_generic_and_oracle(orc, leaves, w, bits):
    rng = np.random.default_rng(100 * leaves + w)
    n = leaves + 1
    eu, ev = [0] * leaves, list(range(1, n))
    dw = _one_row_tables(eu, ev, n, 2, w)
    _fill(dw, _magnitudes(rng, bits))
    masks = G.connected_subplans(n, eu, ev)
    lat, st1 = _run(dw, masks, flags=K.CMP_EST_STAR_LATTICE)
    gen, st2 = _run(dw, masks)
    assert K.cmp_estimate_plan_stats(lat.plan_host.ctypes.data).n_star == 1
    assert st1 == st2 == 0
    assert torch.equal(lat.est, gen.est)
    assert torch.equal(lat.wide_rows, gen.wide_rows)
    if leaves <= 8:
        qs = np.random.default_rng(1).choice(len(masks), min(len(masks), 40), replace=False)
        rows = lat.wide_values()
        for q, ref in zip(qs, _oracle(orc, dw, [masks[q] for q in qs])):
            assert rows[q] == ref.rows and float(lat.est[q]) == ref.est
