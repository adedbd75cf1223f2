"""Training step at the edges of its tiles: sample chunks of 128, hidden blocks of 16, column
blocks of 8 per group of hidden units.  Gradient and loss against the oracle (64-bit sums of
the same bfloat16 weights)."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import pipeline as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nin,nh,skip", [(1, 1, 1, -1), (127, 3, 16, 1), (128, 13, 64, 5), (129, 66, 17, 32),
                                           (1000, 33, 33, -1), (5000, 7, 48, 0)])
def test_training_step_at_tile_edges(orc, n, nin, nh, skip):
    rng = np.random.default_rng(n + nin)
    comb = P.Combiner(nin, nh, seed=2, skip=skip)
    xh = rng.normal(0.0, 0.3, (n, nin)).astype(np.float32)
    th = rng.uniform(0.0, 1.0, n).astype(np.float32)
    p0 = comb.params.cpu().numpy().copy()
    comb.train_step(torch.from_numpy(xh).cuda(), torch.from_numpy(th).cuda(), lr=1e-3, huber_delta=0.1)
    torch.cuda.synchronize()
    loss, g = orc.mlp_loss_grad(nin, nh, p0, xh, th, skip=skip, huber_delta=0.1)
    # fp32 sums of at most 5000 terms in chunks of 128: relative to the largest component
    np.testing.assert_allclose(comb.grad.cpu().numpy(), g, rtol=1e-4, atol=2e-6 * np.abs(g).max())
    assert abs(float(comb.loss.item()) - loss) <= 1e-5 * abs(loss) + 1e-7
    assert float(comb.m.abs().sum()) > 0 and torch.isfinite(comb.params).all()
