"""Presort at the edges of its block sort (8 or 16 keys per thread, padding to a power of two of
at least 256) and of its chunks: every row ordered by magnitude, then bucket, for ties, all
equal rows, already sorted and reversed rows and the extreme counters.  Integers: exact."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [1, 2, 7, 31, 33, 255, 256, 257, 1000, 1023, 4096, 4097, 8192, 8193, 16384, 16385, 40_000])
def test_rows_ordered_by_magnitude_then_bucket(w):
    rng = np.random.default_rng(w)
    I = np.iinfo(np.int32)
    rows = [rng.integers(-5, 6, w), rng.integers(I.min, I.max, w), np.zeros(w), np.arange(w), np.arange(w)[::-1],
            rng.choice([I.min, I.max, 0, -1], w), np.full(w, I.min)]
    C = np.stack(rows).astype(np.int32)
    Cd = torch.from_numpy(C).cuda()
    a = torch.empty_like(Cd)
    p = torch.empty_like(Cd)
    nb = K.cmp_presort_ws_bytes(len(C), w)
    ws = torch.empty(max(nb, 16), dtype=torch.uint8, device="cuda")
    K.cmp_presort(Cd.data_ptr(), len(C), w, a.data_ptr(), p.data_ptr(), ws.data_ptr(), nb, K.stream_handle())
    torch.cuda.synchronize()
    mag = np.abs(C.astype(np.int64))
    order = np.argsort(mag, axis=1, kind="stable")
    assert np.array_equal(p.cpu().numpy(), order)
    assert np.array_equal(a.cpu().numpy().view(np.uint32), np.take_along_axis(mag, order, 1))
