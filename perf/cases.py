"""The work a user of this framework has it do, as cases that can be timed and compared.

Kinds of case (the entry point, and what it stands for in use):
  two_way      one query over two tables: batched build, presort, estimate.  The smallest
               call, an optimiser's single join; launches and latency count.
  five_table   one query over the 5-table cyclic graph (the paper's running example): build,
               presort, the estimate of all 19 sub-plans, combiner, join-order enumeration.
               option rate < 1: sketches over a Bernoulli row sample (no combiner trained on it).
  per_table    the same tables built by one cmp_sketch_build call each (an engine that has no
               plan for the query yet): the per-tuple path.
  scale        one query over a large fact table with int64 keys and wide sketches and two
               dimension tables, d = 15, w = 65536: build, presort, estimate, enumeration.
  graphs       a batch of chain / star / cycle graphs handled together: one batched build,
               one plan over every connected sub-plan, the enumeration of every graph.
               Many rows: the build counts.  Few rows and many sub-plans: the estimate counts.
  pairs        the learned combiner on a batch of two-table joins: build, estimates,
               features, network, combined estimate.
  train        one full-batch training step of the combiner.
  partition    partitioned (k-dimensional) sketches of a chain of three tables: build and
               contraction.

Sizes come from this repository's configurations (datagen.py, bench.py, the training script).
What a case fixes (row counts, predicates, Zipf exponents, graph shapes) does not depend on
the seed; the columns do.
"""
import math

import numpy as np
import torch

from paper_2102_02440_gb300 import compass as K
from paper_2102_02440_gb300 import datagen as G
from paper_2102_02440_gb300 import pipeline as P

DEV = "cuda"


def listed():
    return [
        # an optimiser's smallest question: one join of a 1e5- and a 1e6-row table
        {"name": "two_way", "kind": "two_way", "n_r": 100_000, "n_s": 1_000_000, "domain": 100_000, "s": 1.0,
         "d": 5, "w": 1024, "cut": 300},
        # the paper's running example at full size, through to the chosen join order
        {"name": "five_table", "kind": "five_table", "scale": 1.0, "d": 11, "w": 4096, "sel": 20, "rate": 1.0},
        # the same query answered from a 10% row sample
        {"name": "five_table_sampled", "kind": "five_table", "scale": 1.0, "d": 11, "w": 4096, "sel": 20, "rate": 0.1},
        # an engine that builds table by table, without a plan
        {"name": "per_table", "kind": "per_table", "scale": 0.125, "d": 11, "w": 4096, "sel": 20},
        # a data warehouse's fact table: the largest query, and an ordinary one of its shape
        {"name": "scale_1e9", "kind": "scale", "n_fact": 1_000_000_000, "n_d1": 100_000_000, "n_d2": 1_000_000,
         "d": 15, "w": 65536},
        {"name": "scale_1e7", "kind": "scale", "n_fact": 10_000_019, "n_d1": 1_000_003, "n_d2": 100_003,
         "d": 15, "w": 65536},
        # many queries at once: the rows dominate
        {"name": "graphs_build", "kind": "graphs", "n_chain": 4, "n_star": 4, "n_cycle": 4, "t_lo": 4, "t_hi": 9,
         "rows_lo": 10_000, "rows_hi": 10_000_000, "layout": 1, "d": 11, "w": 1024},
        # the sub-plans of long chains and cycles over small tables: the estimate dominates
        {"name": "graphs_paths", "kind": "graphs", "n_chain": 6, "n_star": 0, "n_cycle": 4, "t_lo": 4, "t_hi": 17,
         "rows_lo": 10_000, "rows_hi": 300_000, "layout": 2, "d": 11, "w": 1024},
        # star joins with many dimensions: tens of thousands of sub-plans
        {"name": "graphs_stars", "kind": "graphs", "n_chain": 0, "n_star": 3, "n_cycle": 0, "t_lo": 10, "t_hi": 15,
         "rows_lo": 10_000, "rows_hi": 100_000, "layout": 3, "d": 11, "w": 1024},
        # the combiner serving a batch of joins, and learning from the training set's 80% split
        {"name": "pairs", "kind": "pairs", "n_pairs": 48, "rows_lo": 10_000, "rows_hi": 10_000_000, "layout": 4,
         "d": 11, "w": 4096},
        {"name": "train", "kind": "train", "n": 80_000, "d": 11, "nh": 64},
        # the unbiased estimator of a 3-table chain, as wide as the merged sketches
        {"name": "partition", "kind": "partition", "scale": 1.0, "d": 11, "w0": 4096, "w1": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["two_way", "five_table", "per_table", "scale", "graphs", "graphs", "pairs", "train", "partition"])
    if kind == "two_way":
        return {"kind": kind, "n_r": _log(rng, 1e4, 1e6), "n_s": _log(rng, 1e5, 1e7), "domain": _log(rng, 1e4, 1e6),
                "s": round(rng.uniform(0.5, 1.5), 3), "d": rng.choice([3, 5, 7, 11]),
                "w": rng.choice([512, 1000, 1023, 1024, 2048, 4096]), "cut": rng.randint(10, 1000)}
    if kind == "five_table":
        return {"kind": kind, "scale": round(math.exp(rng.uniform(math.log(0.02), 0.0)), 4), "d": 11,
                "w": rng.choice([1023, 2048, 4096]), "sel": rng.randint(1, 50), "rate": rng.choice([1.0, 1.0, 0.3, 0.01])}
    if kind == "per_table":
        return {"kind": kind, "scale": round(math.exp(rng.uniform(math.log(0.01), math.log(0.125))), 4),
                "d": rng.choice([5, 11]), "w": rng.choice([1023, 1024, 4096]), "sel": rng.randint(1, 50)}
    if kind == "scale":
        n = _log(rng, 1e6, 5e8)
        return {"kind": kind, "n_fact": n, "n_d1": max(n // rng.randint(5, 20), 1000), "n_d2": _log(rng, 1e4, 1e6),
                "d": rng.choice([11, 15]), "w": rng.choice([16384, 32768, 65536])}
    if kind == "graphs":
        stars = rng.randint(0, 3)
        return {"kind": kind, "n_chain": rng.randint(0, 5) + (stars == 0), "n_star": stars, "n_cycle": rng.randint(0, 3),
                "t_lo": 4, "t_hi": rng.randint(5, 14), "rows_lo": 10_000, "rows_hi": _log(rng, 1e5, 5e6),
                "layout": rng.randint(10, 10**6), "d": 11, "w": rng.choice([1023, 1024])}
    if kind == "pairs":
        return {"kind": kind, "n_pairs": rng.randint(3, 48), "rows_lo": 10_000, "rows_hi": _log(rng, 1e5, 1e7),
                "layout": rng.randint(10, 10**6), "d": 11, "w": rng.choice([1000, 4096])}
    if kind == "train":
        return {"kind": kind, "n": _log(rng, 1e3, 8e4), "d": rng.choice([5, 11, 15]), "nh": rng.choice([16, 48, 64])}
    return {"kind": kind, "scale": round(math.exp(rng.uniform(math.log(0.05), 0.0)), 4), "d": rng.choice([5, 11]),
            "w0": rng.choice([64, 100, 256, 1024, 4096]), "w1": rng.choice([64, 255, 1024, 4096])}


# ------------------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _two_way(c, seed):
    gen, tabs = _gen(seed), []
    for name, n in (("R", c["n_r"]), ("S", c["n_s"])):
        key = G.zipf_keys_device(gen, n, c["domain"], c["s"], torch.int32)
        p = torch.randint(0, 1000, (n,), generator=gen, device=DEV, dtype=torch.int32)
        tabs.append(G.Table(name, [key, p], [G.Pred(1, G.RANGE, G.INT64_MIN, c["cut"])], [0], [0]))
    return G.Workload("two_way", tabs, [0], [1], c["d"], c["w"], 0xC0FFEE, seed)


def _shapes(c):
    """The graphs of a batch without their columns, the same for every seed: (edges, tables),
    a table = (rows, Zipf exponent per key column, None or ("eq",) or ("range", cut))."""
    r = np.random.default_rng(c["layout"])
    out = []
    for kind in ["chain"] * c["n_chain"] + ["star"] * c["n_star"] + ["cycle"] * c["n_cycle"]:
        n = int(r.integers(c["t_lo"], c["t_hi"] + 1))
        if kind == "star":
            edges = [(0, i) for i in range(1, n)]
        else:
            edges = [(i, i + 1) for i in range(n - 1)] + ([(0, n - 1)] if kind == "cycle" else [])
        tabs = []
        for t in range(n):
            rows = int(np.exp(r.uniform(np.log(c["rows_lo"]), np.log(c["rows_hi"]))))
            s = [float(r.uniform(0.5, 1.5)) for e in edges if t in e]
            u, v, cut = r.random(), r.random(), int(1000 * r.uniform(0.01, 0.5))
            tabs.append((rows, s, None if u >= 0.5 else (("eq",) if v < 0.5 else ("range", cut))))
        out.append((kind, edges, tabs))
    return out


def _graphs(c, seed):
    """datagen.graph_batch_device's recipe over the shapes of the case."""
    gen, domain, out = _gen(seed), 100_000, []
    for gi, (kind, edges, shapes) in enumerate(_shapes(c)):
        tabs = []
        for t, (rows, s, pred) in enumerate(shapes):
            on = [e for e, uv in enumerate(edges) if t in uv]
            cols = [G.zipf_keys_device(gen, rows, domain, x, torch.int32) for x in s]
            meta, preds = [("domain", 0, domain)] * len(cols), []
            if pred is not None and pred[0] == "eq":
                codes = G.zipf_keys_device(gen, rows, 1000, 1.0, torch.int32)
                preds = [G.Pred(len(cols), G.EQ, int(codes[0].item()))]
                cols, meta = cols + [codes], meta + [None]
            elif pred is not None:
                preds = [G.Pred(len(cols), G.RANGE, 0, pred[1])]
                cols = cols + [torch.randint(0, 1000, (rows,), generator=gen, device=DEV, dtype=torch.int32)]
                meta = meta + [None]
            tabs.append(G.Table(f"G{gi}T{t}", cols, preds, list(range(len(s))), on, meta))
        out.append(G.Workload(f"{kind}{len(tabs)}", tabs, [u for u, _ in edges], [v for _, v in edges], c["d"], c["w"],
                              0xC0FFEE + gi, seed))
    return out


def _connected(kind, n):
    """Every connected sub-plan of a chain, star (root 0) or cycle of n tables."""
    if kind == "star":
        return sorted([1 << i for i in range(1, n)] + [2 * v + 1 for v in range(1 << (n - 1))])
    wrap = n if kind == "cycle" else 0
    return sorted({sum(1 << ((i + k) % n) for k in range(m)) for i in range(n) for m in range(1, n + 1)
                   if i + m <= n or (wrap and m < n)})


def _n_sub(kind, n):
    return len(_connected(kind, n))


def _pair_shapes(c):
    """(rows R, rows S, domain, s R, s S) of every pair, the same for every seed."""
    r = np.random.default_rng(c["layout"])
    lo, hi = np.log(c["rows_lo"]), np.log(c["rows_hi"])
    return [(int(np.exp(r.uniform(lo, hi))), int(np.exp(r.uniform(lo, hi))), int(np.exp(r.uniform(np.log(1e3), np.log(1e6)))),
             float(r.uniform(0.5, 1.5)), float(r.uniform(0.5, 1.5))) for _ in range(c["n_pairs"])]


def _pair_keys(c, seed):
    """Every table's keys back to back in one tensor, as the training set's are."""
    gen, parts = _gen(seed), []
    for n_r, n_s, dom, s_r, s_s in _pair_shapes(c):
        parts += [G.zipf_keys_device(gen, n_r, dom, s_r, torch.int32), G.zipf_keys_device(gen, n_s, dom, s_s, torch.int32)]
    return torch.cat(parts), np.concatenate([[0], np.cumsum([p.numel() for p in parts])])


def _train_set(c, seed):
    """Features as cmp_mlp_features lays them out (sorted row estimates around their median,
    two self-join sizes, logarithms over 32) and targets around the median."""
    gen, n, d = _gen(seed), c["n"], c["d"]
    med = torch.rand((n, 1), generator=gen, device=DEV) * 0.9
    dev = torch.randn((n, d), generator=gen, device=DEV).sort(dim=1).values * torch.rand((n, 1), generator=gen, device=DEV) * 0.1
    x = dev - dev[:, d // 2:d // 2 + 1]
    x[:, d // 2:d // 2 + 1] = med
    f2 = med / 2 + torch.rand((n, 2), generator=gen, device=DEV) * 0.4
    y = (med[:, 0] + 0.02 * torch.randn((n,), generator=gen, device=DEV)).clamp(min=0)
    return torch.cat([x, f2], 1).contiguous(), y


def _trained(c):
    """The trained combiner where the repository ships one (d = 11, 64 hidden), else a fresh one."""
    if c["nh"] == 64:
        return P.Combiner.for_sketches(c["d"], 4096, device=DEV)[0]
    return P.Combiner(c["d"] + 2, c["nh"], seed=1, device=DEV, skip=c["d"] // 2)


# ----------------------------------------------------------------------- prepare and run

def _combiner_state(s, wl, masks):
    """What bench.py keeps for the combiner: the network, each two-table sub-plan's sketches."""
    dw = s["dw"]
    s["comb"], src = P.Combiner.for_sketches(wl.d, wl.w, device=DEV)
    trained = not str(src.get("weights", "")).startswith("untrained")
    s["below"] = float(src.get("use_median_at", 1.0))
    first = np.cumsum([0] + [t.k for t in dw.tables])
    idx = np.full((len(masks), 2), -1, np.int32)
    for q, m in enumerate(masks):
        for e in range(wl.n_edges):
            if m == (1 << wl.edge_u[e]) | (1 << wl.edge_v[e]):
                idx[q] = [first[t] + si for t, si in (wl.sketch_of(e, 0), wl.sketch_of(e, 1))]
    s["idx"] = torch.from_numpy(idx).to(DEV)
    s["eligible"] = torch.from_numpy(np.array([trained and bin(m).count("1") == 2 for m in masks], np.uint8)).to(DEV)
    n, k = len(masks), dw.counters_all.shape[0]
    s["f2"] = torch.zeros(k, dtype=torch.float64, device=DEV)
    s["feat"] = torch.zeros((n, wl.d + 2), dtype=torch.float32, device=DEV)
    s["y"] = torch.zeros(n, dtype=torch.float32, device=DEV)
    s["combined"] = torch.zeros(n, dtype=torch.float64, device=DEV)


def _combine(s):
    dw, est, st = s["dw"], s["est"], K.stream_handle()
    n, d = est.est.numel(), dw.d
    K.cmp_sketch_f2(dw.counters_all.data_ptr(), s["f2"].numel(), d, dw.w, s["f2"].data_ptr(), st)
    K.cmp_mlp_features_indexed(est.row_est.data_ptr(), n, d, s["f2"].data_ptr(), s["idx"].data_ptr(),
                               s["feat"].data_ptr(), st)
    K.cmp_mlp_infer(s["comb"].params.data_ptr(), d + 2, s["comb"].nh, s["comb"].skip, s["feat"].data_ptr(), n,
                    s["y"].data_ptr(), st)
    K.cmp_mlp_combine_ex(est.est.data_ptr(), s["y"].data_ptr(), s["eligible"].data_ptr(), n, s["below"],
                         s["combined"].data_ptr(), st)
    return s["combined"]


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind in ("two_way", "five_table", "per_table", "scale"):
        if kind == "two_way":
            wl = _two_way(c, seed)
        elif kind == "scale":
            wl = G.scale_workload_device(c["n_fact"], c["n_d1"], c["n_d2"], d=c["d"], w=c["w"], seed=seed)
        else:
            wl = G.five_table_device(scale=c["scale"], d=c["d"], w=c["w"], d1_sel_pct=c["sel"], data_seed=seed)
        rates = [c["rate"]] * len(wl.tables) if c.get("rate", 1.0) < 1.0 else None
        s["dw"] = dw = P.DeviceWorkload(wl, sample_rates=rates)
        if kind == "per_table":
            return s
        masks = G.connected_subplans(len(wl.tables), wl.edge_u, wl.edge_v)
        s["est"] = P.DeviceEstimator(dw, masks)
        dw.encode_batched()
        if kind != "two_way":
            s["enum"] = P.Enumerator(s["est"].graphs, np.zeros(len(masks), np.int32), masks)
        if kind == "five_table" and rates is None:
            _combiner_state(s, wl, masks)
    elif kind == "graphs":
        s["gb"] = gb = P.GraphBatch(_graphs(c, seed))
        sg, sm = [], []
        for gi, (k, _, tabs) in enumerate(_shapes(c)):
            m = _connected(k, len(tabs))
            sg += [gi] * len(m)
            sm += m
        gb.dw.encode_batched()
        s["plan"] = gb.plan(sg, sm, K.cmp_estimate_cfg.make(threads=256, ctas_per_sm=4, cond_chunk=16,
                                                            flags=K.CMP_EST_CACHE_MESSAGES | K.CMP_EST_STAR_LATTICE))
        s["enum"] = P.Enumerator(gb.graph_structs(), sg, sm, cfg=K.cmp_enum_cfg.make(max_plans=1))
    elif kind == "pairs":
        keys, off = _pair_keys(c, seed)
        s["pb"] = P.PairBatch(None, c["d"], c["w"], 0xC0FFEE + 3, device_keys=keys, offsets=off)
        s["pb"].prepare_estimate()
        s["pb"].dw.encode_batched()
        s["comb"] = P.Combiner.for_sketches(11, 4096, device=DEV)[0]
    elif kind == "train":
        s["x"], s["t"] = _train_set(c, seed)
        s["comb"] = _trained(c)
    else:
        wl = G.five_table_device(scale=c["scale"], d=c["d"], w=4096, data_seed=seed)
        s["pj"] = P.PartitionedJoin(wl, [3, 1, 2], [0, 1], [c["w0"], c["w1"]])
    return s


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "per_table":
        s["dw"].build()
        return {"counters": s["dw"].counters_all, "survivors": s["dw"].survivors}
    if kind in ("two_way", "five_table", "scale"):
        dw, est = s["dw"], s["est"]
        dw.build_batched()
        est.presort()
        est.estimate()
        out = {"counters": dw.counters_all, "survivors": dw.survivors, "est": est.est, "row_est": est.row_est}
        best = est.est
        if "comb" in s:
            best = out["combined"] = _combine(s)
        if "enum" in s:
            s["enum"].run(best)
            out.update(order=s["enum"].order, cost=s["enum"].cost, stats=s["enum"].stats)
        return out
    if kind == "graphs":
        gb = s["gb"]
        gb.build_batched()
        gb.presort()
        s["plan"].run(row_est=False)
        s["enum"].run(s["plan"].est)
        return {"counters": gb.dw.counters_all, "survivors": gb.dw.survivors, "est": s["plan"].est,
                "order": s["enum"].order, "cost": s["enum"].cost, "stats": s["enum"].stats}
    if kind == "pairs":
        pb = s["pb"]
        pb.build()
        pb.estimate()
        feat = pb.features()
        y = s["comb"].infer(feat)
        return {"counters": pb.counters, "est": pb.est, "row_est": pb.row_est, "feat": feat, "y": y,
                "combined": s["comb"].combine(pb.est, y)}
    if kind == "train":
        c = s["comb"]
        c.train_step(s["x"], s["t"], lr=3e-4, huber_delta=0.001)
        return {"loss": c.loss, "grad": c.grad, "params": c.params, "m": c.m, "v": c.v}
    s["pj"].build()
    s["pj"].estimate()
    return {"tensors": s["pj"].tensors, "survivors": s["pj"].survivors, "est": s["pj"].est, "row_est": s["pj"].row_est}


# ---------------------------------------------------------------------------------- work

def work(case):
    """Bytes: every referenced column read once, every output written once.  Flops: two per
    weight and sample of the network (forward, and twice that backward); the sketches and
    their contraction are integer work and count none."""
    c, kind = case, case["kind"]
    if kind == "train":
        np_ = c["nh"] * (c["d"] + 4) + 1
        return {"bytes": 4.0 * c["n"] * (c["d"] + 3) + 4.0 * np_ * 7, "flops": 6.0 * c["n"] * np_}
    if kind == "two_way":
        return {"bytes": 8.0 * (c["n_r"] + c["n_s"]) + 8.0 * c["d"] * c["w"], "flops": 0.0}
    if kind in ("five_table", "per_table"):
        return {"bytes": c["scale"] * 8.0 * 47_134_000 + 40.0 * c["d"] * c["w"], "flops": 0.0}
    if kind == "scale":
        return {"bytes": 24.0 * c["n_fact"] + 8.0 * (c["n_d1"] + c["n_d2"]) + 16.0 * c["d"] * c["w"], "flops": 0.0}
    if kind == "graphs":
        b = 0.0
        for k, _, tabs in _shapes(c):
            b += 8.0 * _n_sub(k, len(tabs))
            for rows, s, pred in tabs:
                b += 4.0 * rows * (len(s) + (pred is not None)) + 4.0 * len(s) * c["d"] * c["w"]
        return {"bytes": b, "flops": 0.0}
    if kind == "pairs":
        rows = sum(a + b for a, b, _, _, _ in _pair_shapes(c))
        return {"bytes": 4.0 * rows + 8.0 * c["n_pairs"] * c["d"] * c["w"], "flops": 2.0 * c["n_pairs"] * 64 * 15}
    return {"bytes": c["scale"] * 8.0 * 7_134_000 + 4.0 * c["d"] * (c["w0"] * c["w1"] + c["w0"] + c["w1"]),
            "flops": 0.0}


# --------------------------------------------------------------------------------- exact

P61 = (1 << 61) - 1


def _splitmix(seed, n_edges, d):
    """The hash parameters [edge][row] = (a, b, c0, c1, c2, c3) from their definition."""
    s, out, mask = seed, [], (1 << 64) - 1
    for _ in range(n_edges):
        rows = []
        for _ in range(d):
            f = []
            for _ in range(6):
                s = (s + 0x9E3779B97F4A7C15) & mask
                z = s
                z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
                z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
                v = (z ^ (z >> 31)) >> 3
                f.append(0 if v == P61 else v)
            f[0] = f[0] or 1
            rows.append(f)
        out.append(rows)
    return out


def _mul_small(y, x):
    """y x mod 2^61 - 1 for residues y (int64 tensor) and x < 2^20 (int64 tensor)."""
    lo, hi = (y & ((1 << 31) - 1)) * x, (y >> 31) * x            # y x = lo + hi 2^31, hi < 2^50
    v = (lo & P61) + (hi >> 30) + ((hi & ((1 << 30) - 1)) << 31)  # 2^61 = 1
    return v % P61


def _sketch_rows(keys, domain, params, w):
    """[d][w] int64 Fast-AGMS counters of keys in [0, domain), domain <= 2^20."""
    cnt = torch.bincount(keys.to(torch.int64), minlength=domain)
    x = torch.arange(domain, device=keys.device, dtype=torch.int64)
    rows = []
    for a, b, c0, c1, c2, c3 in params:
        h = (_mul_small(torch.full_like(x, a), x) + b) % P61 % w
        v = torch.full_like(x, c3)
        for k in (c2, c1, c0):
            v = (_mul_small(v, x) + k) % P61
        rows.append(torch.zeros(w, dtype=torch.int64, device=x.device).scatter_add_(0, h, cnt * (1 - 2 * (v & 1))))
    return torch.stack(rows)


def _mlp64(p, nin, nh, skip, x):
    """Forward pass in 64 bits over the network's bfloat16 weights: (y, hidden, weights)."""
    q = p.to(torch.bfloat16).to(torch.float64)
    w1, b1 = q[:nh * nin].view(nh, nin), q[nh * nin:nh * nin + nh]
    w2, b2 = q[nh * nin + nh:nh * nin + 2 * nh], q[-1]
    z = (x @ w1.T + b1).clamp(min=0)
    base = x[:, skip].clamp(min=0) if skip >= 0 else 0.0
    return base + z @ w2 + b2, z, w2


def _exact_two_way(c, seed):
    wl = _two_way(c, seed)
    par = _splitmix(wl.hash_seed, 1, c["d"])[0]
    sk, n = [], []
    for t in wl.tables:
        k = t.cols[0][t.cols[1] < c["cut"]]
        n.append(float(k.numel()))
        sk.append(_sketch_rows(k, c["domain"], par, c["w"]))
    e = (sk[0] * sk[1]).sum(1).sort().values
    return {"counters": None, "survivors": None, "est": torch.tensor(n + [float(e[c["d"] // 2])], dtype=torch.float64),
            "row_est": None}


def _exact_pairs(c, seed):
    keys, off = _pair_keys(c, seed)
    d, shapes = c["d"], _pair_shapes(c)
    par = _splitmix(0xC0FFEE + 3, len(shapes), d)
    est, feat = [], []
    for i, (_, _, dom, _, _) in enumerate(shapes):
        a, b = (_sketch_rows(keys[int(off[2 * i + k]):int(off[2 * i + k + 1])], dom, par[i], c["w"]) for k in (0, 1))
        e = (a * b).sum(1).sort().values
        est.append(float(e[d // 2]))
        e = e.to(torch.float64)
        v = torch.sign(e) * torch.log1p(e.abs()) / 32
        f = v - v[d // 2]
        f[d // 2] = v[d // 2]
        f2 = torch.stack([(z * z).sum(1).sort().values[d // 2] for z in (a, b)]).to(torch.float64)
        feat.append(torch.cat([f, torch.log1p(f2) / 32]))
    est, feat = torch.tensor(est, dtype=torch.float64, device=keys.device), torch.stack(feat)
    comb = P.Combiner.for_sketches(11, 4096, device=DEV)[0]
    y = _mlp64(comb.params, d + 2, comb.nh, comb.skip, feat)[0]
    return {"counters": None, "est": est, "row_est": None, "feat": feat, "y": y,
            "combined": torch.where(est >= 1, est, torch.expm1(32 * y).clamp(min=0))}


def _exact_train(c, seed):
    x, t = (v.to(torch.float64) for v in _train_set(c, seed))
    comb = _trained(c)
    nin, nh, n, delta, lr = c["d"] + 2, c["nh"], c["n"], float(np.float32(0.001)), float(np.float32(3e-4))
    y, z, w2 = _mlp64(comb.params, nin, nh, comb.skip, x)
    e = y - t
    a = e.abs()
    dy = torch.where(a <= delta, e, torch.sign(e) * delta) / n
    loss = torch.where(a <= delta, 0.5 * e * e, delta * (a - 0.5 * delta)).sum() / n
    dz = torch.where(z > 0, dy[:, None] * w2, torch.zeros_like(z))
    g = torch.cat([(dz.T @ x).reshape(-1), dz.sum(0), dy @ z, dy.sum()[None]])
    m, v = 0.9 * comb.m.double() + 0.1 * g, 0.999 * comb.v.double() + 0.001 * g * g
    k = comb.step + 1
    p = comb.params.double() - lr * (m / (1 - 0.9**k)) / ((v / (1 - 0.999**k)).sqrt() + 1e-8)
    return {"loss": loss[None], "grad": g, "params": p, "m": m, "v": v}


def exact(case, seed):
    """What run() returns, in 64 bits by plain torch, for the cases whose outputs such a
    computation reaches in seconds: two-table estimates, the network and its training step.
    The others' estimates are exact integers rounded once, beside whole numbers."""
    kind = case["kind"]
    if kind == "two_way":
        return _exact_two_way(case, seed)
    if kind == "pairs":
        return _exact_pairs(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    return None
