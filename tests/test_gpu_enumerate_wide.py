"""Join-order enumeration where its tables leave the small case: graphs of more than 32 tables
(two candidates per lane), a prefix with more than 32 candidates, sub-plan tables at and
beyond the staged size, and search budgets that end inside a pruned frame."""
import numpy as np
import pytest

from oracle import enumerate as E
from paper_2102_02440_gb300 import compass as K
from test_gpu_enumerate import _connected, _graph, _oracle, _run

pytestmark = pytest.mark.gpu


def _chain_masks(n):
    return [((1 << m) - 1) << i for m in range(2, n + 1) for i in range(n - m + 1)]


@pytest.mark.parametrize("n,max_plans", [(33, 1), (64, 1), (12, 3)])
def test_long_chains(n, max_plans):
    rng = np.random.default_rng(n)
    eu, ev = list(range(n - 1)), list(range(1, n))
    # estimates growing with the prefix keep the search near its first plan
    est = {m: float(bin(m).count("1") * 100 + rng.integers(0, 3)) for m in _chain_masks(n)}
    card = [int(x) for x in rng.integers(1, 1000, n)]
    budget = 5000 if n > 12 else 0   # 0: no limit
    got, st = _run([_graph(n, eu, ev, card)], [(0, m) for m in est], list(est.values()), max_plans, max_nodes=budget)
    if n == 12:
        assert st == 0 and got[0] == _oracle(n, eu, ev, est, card, max_plans)
    else:
        assert st == K.CMP_ETIMEOUT and got[0][2][1] == budget and len(got[0][0]) == n


@pytest.mark.parametrize("leaves", [11, 12])   # 4096 and 8192 slots: staged, not staged
def test_stars_around_the_staged_size(leaves):
    rng = np.random.default_rng(leaves)
    n = leaves + 1
    eu, ev = [0] * leaves, list(range(1, n))
    est = {1 | (v << 1): float(rng.lognormal(4, 2)) if v % 7 else 5.0 for v in range(1, 1 << leaves)}
    card = [int(x) for x in rng.integers(1, 1000, n)]
    got, st = _run([_graph(n, eu, ev, card)], [(0, m) for m in est], list(est.values()), 2)
    assert st == 0 and got[0] == _oracle(n, eu, ev, est, card, 2)


def test_many_candidates_and_every_budget():
    """A star of 40 leaves whose two-table sub-plans alone are known: the root's frame has 40
    candidates, every longer prefix is missing (+inf)."""
    n = 41
    eu, ev = [0] * 40, list(range(1, n))
    est = {1 | (1 << v): float(v % 5) for v in range(1, n)}
    got, st = _run([_graph(n, eu, ev, [1] * n)], [(0, m) for m in est], list(est.values()), 1, max_nodes=300)
    assert st == K.CMP_EUNSUPPORTED and got[0][2][1] == 300 and got[0][2][2] == 0
    # budgets ending before, inside and after a pruned frame of a small star
    eu, ev = [0] * 5, list(range(1, 6))
    masks = _connected(6, eu, ev)
    est = {m: float(10 ** (bin(m).count("1") - 2) + m % 3) for m in masks}
    full = _oracle(6, eu, ev, est, [3] * 6, -1)
    g = _graph(6, eu, ev, [3] * 6)
    for budget in list(range(1, 30)) + [full[2][1], full[2][1] + 1]:
        got, st = _run([g], [(0, m) for m in masks], [est[m] for m in masks], -1, max_nodes=budget)
        if budget < full[2][1]:
            assert st == K.CMP_ETIMEOUT and got[0][2][1] == budget
        else:
            assert st == 0 and got[0] == full


@pytest.mark.parametrize("max_plans", [1, 2, 10])
@pytest.mark.parametrize("shape", ["chain", "cycle", "star", "tree"])
def test_long_searches_match_oracle(shape, max_plans):
    """Searches of thousands of extensions (parallel rounds), with ties and several completed
    plans per source, and their exact stops at a search budget."""
    rng = np.random.default_rng(len(shape) + max_plans)
    graphs, subs, est_host, ref = [], [], [], []
    for gi in range(6):
        n = {"chain": 13, "cycle": 11, "star": 8, "tree": 9}[shape]
        if shape == "star":
            eu, ev = [0] * (n - 1), list(range(1, n))
        elif shape == "tree":
            eu, ev = [int(rng.integers(0, t)) for t in range(1, n)], list(range(1, n))
        else:
            eu, ev = list(range(n - 1)), list(range(1, n))
            if shape == "cycle":
                eu, ev = eu + [0], ev + [n - 1]
        full = (1 << n) - 1
        est = {m: (float(rng.integers(0, 3)) if gi % 2 else float(rng.lognormal(3, 3)))
               for m in _connected(n, eu, ev)}
        est[full] = 1e6 if gi % 3 else 0.0   # the last join decides little: long searches
        card = [int(x) for x in rng.integers(0, 1000, n)]
        graphs.append(_graph(n, eu, ev, card))
        for m in sorted(est):
            subs.append((gi, m))
            est_host.append(est[m])
        ref.append(_oracle(n, eu, ev, est, card, max_plans))
    got, st = _run(graphs, subs, est_host, max_plans)
    assert st == 0
    for g, r in zip(got, ref):
        assert g == r
    assert max(r[2][1] for r in ref) > 200
    # budgets that end anywhere: exactly that many extensions, a prefix of the full search
    most = max(r[2][1] for r in ref)
    for budget in [int(b) for b in np.linspace(150, most - 1, 7)]:
        got, st = _run(graphs, subs, est_host, max_plans, max_nodes=budget)
        assert st == K.CMP_ETIMEOUT
        for g, r in zip(got, ref):
            assert g[2][1] == min(budget, r[2][1]) and g[2][0] <= r[2][0] and g[2][2] <= r[2][2]
            assert g == r if budget >= r[2][1] else g[1] >= r[1]
