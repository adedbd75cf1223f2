"""Join-order enumeration of batches of more graphs than SMs, which takes two launches: searches
that end in the first, that are left open there and go on alone and in rounds, on both sides of
the batch's size, with budgets that end before, at and after the change, missing estimates, no
limit on the plans, graphs of 64 tables beside small ones, and a workspace at any address.
Plans, costs and counters are the oracle's."""
import numpy as np
import pytest
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import pipeline as P
from test_gpu_enumerate import _connected, _graph, _oracle, _run

pytestmark = pytest.mark.gpu


def _shape(kind, n):
    if kind == "star":
        return n, [0] * (n - 1), list(range(1, n))
    eu, ev = list(range(n - 1)), list(range(1, n))
    return (n, eu + [0], ev + [n - 1]) if kind == "cycle" else (n, eu, ev)


def _batch(rng, n_graphs, long_every, missing=()):
    """Small graphs, and among them every long_every-th one whose search takes thousands of extensions."""
    small = [("chain", 5), ("star", 5), ("cycle", 4), ("chain", 2), ("chain", 1)]
    graphs, subs, est_host, ref_in = [], [], [], []
    for gi in range(n_graphs):
        kind, n = ("chain", 13) if gi % long_every == 0 else small[gi % len(small)]
        n, eu, ev = _shape(kind, n)
        est = {m: (float(rng.integers(0, 3)) if gi % 2 else float(rng.lognormal(3, 3))) for m in _connected(n, eu, ev)}
        if n == 13:
            est[(1 << n) - 1] = 1e6  # the last join decides little: long searches
        if gi in missing:
            est.pop(next(iter(est)))
        card = [int(x) for x in rng.integers(0, 1000, n)]
        graphs.append(_graph(n, eu, ev, card))
        subs += [(gi, m) for m in sorted(est)]
        est_host += [est[m] for m in sorted(est)]
        ref_in.append((n, eu, ev, est, card))
    return graphs, subs, est_host, ref_in


@pytest.mark.parametrize("max_plans", [1, 10, -1])
@pytest.mark.parametrize("n_graphs", [152, 153, 311])
def test_batches_match_oracle(n_graphs, max_plans):
    rng = np.random.default_rng(n_graphs + max_plans)
    graphs, subs, est_host, ref_in = _batch(rng, n_graphs, 50 if max_plans > 0 else 10**6)
    ref = [_oracle(*r, max_plans) for r in ref_in]
    if max_plans > 0:
        assert max(r[2][1] for r in ref) > 800  # several rounds
    got, st = _run(graphs, subs, est_host, max_plans)
    assert st == 0
    for g, r in zip(got, ref):
        assert g == r


@pytest.mark.parametrize("budget", [1, 95, 96, 97, 192, 193, 250, 288, 289, 1000])
def test_budgets_around_the_change(budget):
    rng = np.random.default_rng(5)
    graphs, subs, est_host, ref_in = _batch(rng, 160, 40)
    ref = [_oracle(*r, 1) for r in ref_in]
    got, st = _run(graphs, subs, est_host, 1, max_nodes=budget)
    assert st == K.CMP_ETIMEOUT
    for g, r in zip(got, ref):
        assert g[2][1] == min(budget, r[2][1]) and g[2][0] <= r[2][0] and g[2][2] <= r[2][2]
        assert g == r if budget >= r[2][1] else g[1] >= r[1]


def test_missing_estimates_and_graphs_of_64_tables():
    rng = np.random.default_rng(6)
    graphs, subs, est_host, ref_in = _batch(rng, 155, 50, missing=(1,))
    n, eu, ev = _shape("chain", 64)
    masks = [((1 << m) - 1) << i for m in range(2, n + 1) for i in range(n - m + 1)]
    graphs.append(_graph(n, eu, ev, [1] * n))
    subs += [(155, m) for m in masks]
    est_host += [float(bin(m).count("1") * 100) for m in masks]
    got, st = _run(graphs, subs, est_host, 1, max_nodes=5000)
    assert st in (K.CMP_EUNSUPPORTED, K.CMP_ETIMEOUT)
    for g, r in list(zip(got, ref_in))[2:]:
        o = _oracle(*r, 1)
        assert g == o if o[2][1] <= 5000 else g[2][1] == 5000
    assert got[155] == _oracle(n, eu, ev, {m: float(bin(m).count("1") * 100) for m in masks}, [1] * n, 1)


def test_workspace_at_any_address():
    rng = np.random.default_rng(7)
    graphs, subs, est_host, ref_in = _batch(rng, 153, 60)
    en = P.Enumerator(graphs, [g for g, _ in subs], [m for _, m in subs], cfg=K.cmp_enum_cfg.make(max_plans=2))
    est = torch.tensor(est_host, dtype=torch.float64, device="cuda")
    need = en.ws.numel()
    store = torch.full((need + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    ref = [_oracle(*r, 2) for r in ref_in]
    for shift in (0, 1, 8, 13):
        store.fill_(0xA5)
        en.ws = store[shift:shift + need]
        en.run(est)
        torch.cuda.synchronize()
        assert en.plans() == ref
        assert bool((store[:shift] == 0xA5).all()) and bool((store[shift + need:] == 0xA5).all())
    en.ws = store[:need - 1]
    with pytest.raises(K.CompassError):
        en.run(est)
