"""The star lattice on both sides of the choice between residues and int128 for units of few entries:
leaves, widths and magnitudes next to where it changes.  Rows against the generic evaluation."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from test_gpu_wide import _fill, _one_row_tables, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [1, 4, 9, 16])
@pytest.mark.parametrize("w", [64, 129, 257, 512, 1024])
@pytest.mark.parametrize("leaves", [2, 3, 4, 5, 6, 8])
def test_rows_match_the_generic_path(leaves, w, bits):
    rng = np.random.default_rng(leaves * 10_000 + w + bits)
    n = leaves + 1
    eu, ev = [0] * leaves, list(range(1, n))
    dw = _one_row_tables(eu, ev, n, 3, w)
    _fill(dw, lambda s: rng.integers(-2**bits, 2**bits + 1, s))
    masks = G.connected_subplans(n, eu, ev)
    lat, st1 = _run(dw, masks, flags=K.CMP_EST_STAR_LATTICE)
    gen, st2 = _run(dw, masks)
    assert st1 == st2 == 0
    assert torch.equal(lat.est, gen.est) and torch.equal(lat.wide_rows, gen.wide_rows)
