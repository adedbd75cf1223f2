"""Presort of narrow rows, whose sort holds one, two, four or eight keys a thread, on both sides of
each width and with more rows than CTAs: ordered by magnitude, then bucket.  Integers: exact."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [3, 9001])
@pytest.mark.parametrize("w", [1, 2, 16, 31, 32, 33, 63, 64, 65, 127, 128, 129, 200, 256, 257])
def test_narrow_rows(w, rows):
    rng = np.random.default_rng(w)
    C = rng.integers(-w, w + 1, (rows, w)).astype(np.int32)
    C[1] = rng.choice([-2**31, 2**31 - 1, 0, -1], w)
    Cd = torch.from_numpy(C).cuda()
    a, p = torch.empty_like(Cd), torch.empty_like(Cd)
    K.cmp_presort(Cd.data_ptr(), rows, w, a.data_ptr(), p.data_ptr(), 0, 0, K.stream_handle())
    torch.cuda.synchronize()
    mag = np.abs(C.astype(np.int64))
    order = np.argsort(mag, axis=1, kind="stable")
    assert np.array_equal(p.cpu().numpy(), order)
    assert np.array_equal(a.cpu().numpy().view(np.uint32), np.take_along_axis(mag, order, 1))
