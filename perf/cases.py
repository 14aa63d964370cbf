"""Performance cases: the calls a user of the scoring library makes, over the sizes they are made at.

A case names an operation and its inputs' sizes; its graph is a seeded LFR-style
graph (mean degree 20, mixing `mu`, power-law degrees and community sizes, node
ids shuffled) and its partitions are the planted one with a share `moved` of
the nodes reassigned, the stand-in for a detected partition.

Operations:
  score     qm.score on one resident graph: every metric without ground truth
  compare   qm.compare: every index of a found partition against the truth
  evaluate  qm.evaluate_batched: candidates of one graph, both families at once
  graphs    qm.score_graphs_batched: one partition on each of several graphs
  detect    qm.label_propagation: a detected partition of the graph
  cover     qm.score_cover and qm.compare_covers: overlapping communities

`exact` states the same metrics in plain torch, in int64 and float64.
"""
import math

import numpy as np
import torch

from paper_1507_05492_gb300 import gen, qm

_MEAN_ARCS = 19.1  # stored arcs per node of the generated graphs (mean degree 20 less dropped repeats)


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one small graph, one partition: the latency of a call (the paper's smallest graphs)
        {"name": "score-10k", "op": "score", "n": 10_000, "mu": 0.3, "moved": 0.0, "reorder": False,
         "weighted": False, "communities": False},
        {"name": "compare-10k", "op": "compare", "n": 10_000, "moved": 0.1},
        # a mid-size graph kept resident, a rough partition, each community's values asked for
        {"name": "score-1m-communities", "op": "score", "n": 1_000_003, "mu": 0.3, "moved": 0.2, "reorder": True,
         "weighted": False, "communities": True},
        # many resident graphs of uneven sizes, one partition each (a serving batch)
        {"name": "graphs-32", "op": "graphs", "count": 32, "n_min": 1_000, "n_max": 100_000, "mu": 0.3,
         "moved": 0.2},
        # a large graph kept resident, a detected partition that is off for a fifth of the nodes
        {"name": "score-10m-moved", "op": "score", "n": 10_000_000, "mu": 0.3, "moved": 0.2, "reorder": True,
         "weighted": False, "communities": False},
        # weighted edges (interaction counts, similarities)
        {"name": "score-10m-weighted", "op": "score", "n": 10_000_000, "mu": 0.3, "moved": 0.0, "reorder": True,
         "weighted": True, "communities": False},
        # the largest graph of the paper's range, renumbered at load and as given
        {"name": "score-100m", "op": "score", "n": 100_000_000, "mu": 0.3, "moved": 0.0, "reorder": True,
         "weighted": False, "communities": False},
        {"name": "score-100m-given", "op": "score", "n": 100_000_000, "mu": 0.3, "moved": 0.0, "reorder": False,
         "weighted": False, "communities": False},
        # a detected partition of the largest graph against the truth
        {"name": "compare-100m", "op": "compare", "n": 100_000_000, "moved": 0.2},
        # model selection: many candidate partitions of one graph, all metrics of each
        {"name": "evaluate-256", "op": "evaluate", "n": 100_000, "count": 256, "mu": 0.3},
        # detection on the device, the step before scoring
        {"name": "detect-10m", "op": "detect", "n": 10_000_000, "mu": 0.3, "reorder": True, "rounds": 10},
        # overlapping communities: a cover scored and compared with the true cover
        {"name": "cover-1m", "op": "cover", "n": 1_000_000, "mu": 0.3, "moved": 0.1, "extra": 0.2,
         "reorder": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["score", "score", "score", "compare", "compare", "evaluate", "graphs", "detect", "cover"])
    mu = rng.choice([0.1, 0.2, 0.3, 0.4, 0.5])
    moved = rng.choice([0.0, round(rng.uniform(0.01, 0.5), 3)])
    if op == "score":
        weighted = rng.random() < 0.2
        # as given, rough partitions cost most: their sizes end where the largest listed cases' cost does
        n = _log_int(rng, 3_000, 30_000_000 if weighted else 50_000_000)
        return {"op": op, "n": n, "mu": mu, "moved": min(moved, 0.2) if n > 20_000_000 else moved,
                "reorder": rng.random() < 0.6, "weighted": weighted, "communities": rng.random() < 0.25}
    if op == "compare":
        return {"op": op, "n": _log_int(rng, 3_000, 100_000_000), "moved": max(moved, 0.01)}
    if op == "evaluate":
        n = _log_int(rng, 5_000, 300_000)
        return {"op": op, "n": n, "count": _log_int(rng, 8, max(9, min(256, 20_000_000 // n))), "mu": mu}
    if op == "graphs":
        hi = _log_int(rng, 10_000, 300_000)
        return {"op": op, "count": _log_int(rng, 2, 64), "n_min": _log_int(rng, 500, 5_000), "n_max": hi, "mu": mu,
                "moved": moved}
    if op == "detect":
        return {"op": op, "n": _log_int(rng, 10_000, 20_000_000), "mu": mu, "reorder": rng.random() < 0.5,
                "rounds": rng.randint(3, 12)}
    return {"op": op, "n": _log_int(rng, 5_000, 1_000_000), "mu": mu, "moved": min(max(moved, 0.01), 0.3),
            "extra": round(rng.uniform(0.02, 0.3), 3), "reorder": rng.random() < 0.5}


# ------------------------------------------------------------------ inputs

def _lfr(n, mu, seed):
    """The generator's graph at the sizes its named workloads use: small graphs have small communities."""
    small = n <= 300_000
    p = gen.LfrParams(n=n, k_mean=20, k_max=50 if small else 100, s_min=20, s_max=100 if small else 1000, mu=mu,
                      seed=seed)
    return gen.lfr_graph(p, device="cuda")


def _id_bound(n):
    """Label ids of a run that keeps per-community arrays of one length for every graph of n nodes: a little above
    the planted count (n over the mean community size), the rest unused."""
    mean = 80 / math.log(5) if n <= 300_000 else 980 / math.log(50)
    return int(n / mean * 1.05) + 64


def _hash(x):
    """A 31-bit hash of an int64 tensor."""
    x = (x ^ (x >> 15)) * 0x2C1B3C6D & 0xFFFFFFFF
    x = (x ^ (x >> 12)) * 0x297A2D39 & 0xFFFFFFFF
    return (x ^ (x >> 15)) & 0x7FFFFFFF


def _weights(row_ptr, col, seed):
    """A float32 weight in [0.05, 5) per arc, the same on both arcs of an edge."""
    n = row_ptr.numel() - 1
    u = torch.repeat_interleave(torch.arange(n, dtype=torch.int32, device=col.device), row_ptr[1:] - row_ptr[:-1])
    h = _hash(torch.minimum(u, col).long() * 2654435761 % (1 << 31) + torch.maximum(u, col).long() * 40503 + seed)
    return (0.05 + h.double() / float(1 << 31) * 4.95).float()


def _cover(labels, row_ptr, col, share, seed):
    """(mptr, memb): every node in its community, a share of the nodes in a neighbour's too (when it differs)."""
    n = labels.numel()
    ids = torch.arange(n, device=labels.device)
    deg = row_ptr[1:] - row_ptr[:-1]
    far = labels[col[(row_ptr[:-1] + _hash(ids + seed * 7919) % deg.clamp(min=1)).clamp(max=col.numel() - 1)].long()]
    two = (_hash(ids * 3 + seed * 104729 + 1).double() / float(1 << 31) < share) & (deg > 0) & (far != labels)
    mptr = torch.zeros(n + 1, dtype=torch.int64, device=labels.device)
    mptr[1:] = torch.cumsum(1 + two.long(), 0)
    memb = torch.empty(int(mptr[-1]), dtype=torch.int32, device=labels.device)
    memb[mptr[:-1]] = torch.where(two, torch.minimum(labels, far), labels)
    memb[mptr[:-1][two] + 1] = torch.maximum(labels, far)[two]
    return mptr, memb


def _planted(n, seed):
    """(labels, K) of a planted partition alone: community sizes as the graphs have them, members at random."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    s_max = 100 if n <= 300_000 else 1000
    u = torch.rand(int(n / ((s_max - 20) / math.log(s_max / 20)) * 1.2) + 32, generator=g, device="cuda",
                   dtype=torch.float64)
    ends = torch.cumsum(torch.round(20 * torch.pow(s_max / 20, u)).long(), 0)
    K = int(torch.searchsorted(ends, n)) + 1
    by_slot = torch.searchsorted(ends[:K], torch.arange(n, device="cuda"), right=True).clamp(max=K - 1)
    return by_slot[torch.randperm(n, generator=g, device="cuda")].to(torch.int32), K


def _inputs(case, seed):
    """The arrays of a case, on the GPU."""
    op = case["op"]
    if op == "compare":
        truth, K = _planted(case["n"], seed)
        return {"truth": truth, "found": gen.perturb(truth, K, case["moved"], seed=seed + 1), "K": K}
    if op == "graphs":
        count, lo, hi = case["count"], case["n_min"], case["n_max"]
        out = []
        for i in range(count):
            n = int(round(lo * (hi / lo) ** (i / max(1, count - 1)))) | 1
            g = _lfr(n, case["mu"], seed * 101 + i)
            out.append({"row_ptr": g.row_ptr, "col": g.col, "K": g.K,
                        "labels": gen.perturb(g.labels, g.K, case["moved"], seed=seed + i)})
        return {"graphs": out}
    g = _lfr(case["n"], case["mu"], seed)
    d = {"row_ptr": g.row_ptr, "col": g.col, "K": g.K}
    if op == "score":
        d["labels"] = gen.perturb(g.labels, g.K, case["moved"], seed=seed + 1) if case["moved"] else g.labels
        if case["communities"]:
            d["K"] = max(g.K, _id_bound(case["n"]))
        d["weights"] = _weights(g.row_ptr, g.col, seed) if case["weighted"] else None
    elif op == "evaluate":
        d["truth"] = g.labels
        d["labels"], d["Ks"] = gen.candidate_batch(g.labels, case["count"], seed=seed * 1009 + 17,
                                                   k_range=(max(2, case["n"] // 200), case["n"] // 20))
    elif op == "cover":
        d["truth"] = _cover(g.labels, g.row_ptr, g.col, case["extra"], seed)
        d["found"] = _cover(gen.perturb(g.labels, g.K, case["moved"], seed=seed + 1), g.row_ptr, g.col,
                            case["extra"] / 2, seed + 2)
    return d


def prepare(case, seed):
    """Resident graphs and label arrays on the GPU."""
    op = case["op"]
    d = _inputs(case, seed)
    if op == "graphs":
        s = {"op": op, "graphs": [qm.Graph(g["row_ptr"], g["col"]) for g in d["graphs"]],
             "labels": [g["labels"] for g in d["graphs"]], "K": [g["K"] for g in d["graphs"]]}
    elif op == "compare":
        s = {"op": op, **d}
    else:
        s = {"op": op, "n": case["n"],
             "graph": qm.Graph(d.pop("row_ptr"), d.pop("col"), reorder=case.get("reorder", False),
                               weights=d.pop("weights", None)), **d}
        s["rounds"] = case.get("rounds", 0)
        s["communities"] = case.get("communities", False)
    torch.cuda.empty_cache()  # the generator's scratch: the library allocates beside torch
    return s


def _columns(rows):
    return {k: np.array([r[k] for r in rows]) for k in rows[0]}


def run(s):
    """One pass through the public calls."""
    op = s["op"]
    if op == "score":
        return qm.score(s["graph"], s["labels"], s["K"], per_community=s["communities"])
    if op == "compare":
        return qm.compare(s["truth"], s["found"], s["K"], s["K"])
    if op == "evaluate":
        q, c = qm.evaluate_batched(s["graph"], s["labels"], s["Ks"], s["truth"], s["K"])
        return {"quality": _columns(q), "compare": _columns(c)}
    if op == "graphs":
        return _columns(qm.score_graphs_batched(s["graphs"], s["labels"], s["K"]))
    if op == "detect":
        labels, k = qm.label_propagation(s["graph"], rounds=s["rounds"])
        return {"labels": labels, "K": k}
    return {"quality": qm.score_cover(s["graph"], s["found"], s["K"]),
            "compare": qm.compare_covers(s["truth"], s["K"], s["found"], s["K"], s["n"])}


def work(case):
    """Bytes of one pass: adjacency, row offsets, labels and outputs, each once.  The arithmetic is counting
    (integer adds), with a handful of FP64 operations per community or cell: no operation rate bounds it."""
    op = case["op"]
    n = case.get("n", 0)
    arcs = _MEAN_ARCS * n
    graph = 4 * arcs + 8 * (n + 1)
    if op == "score":
        out = 64 * _id_bound(n) if case["communities"] else 128
        b = graph + 4 * n + (4 * arcs if case["weighted"] else 0) + out
    elif op == "compare":
        b = 8 * n
    elif op == "evaluate":
        b = graph + 4 * n * (case["count"] + 1)
    elif op == "graphs":
        lo, hi, c = case["n_min"], case["n_max"], case["count"]
        total = sum(lo * (hi / lo) ** (i / max(1, c - 1)) for i in range(c))
        b = total * (4 * _MEAN_ARCS + 8 + 4)
    elif op == "detect":
        b = graph + 4 * n
    else:
        b = graph + 2 * (8 * (n + 1)) + 4 * n * (2 + 1.5 * case["extra"])
    return {"bytes": b, "flops": 0}


# ------------------------------------------------------------------ the metrics in plain torch, 64 bits

_PIECE = 1 << 23  # nodes of the arc list that are expanded at once


def _entropy(p):
    return float((p * torch.log(p)).sum())


def _quality(n, E, size, ein, eout, cut, key, cnt, wkey=None, W=None, win=None, wout=None):
    """Eqs. (8)-(9) and the six measures from the integer counts; wkey, W, win, wout: the weighted amounts."""
    K = size.numel()
    i, j = key // K, key % K
    s, a, b = size.double(), ein.double(), eout.double()
    amount = cnt.double() if wkey is None else wkey
    A, B, T = (a, b, float(E)) if wkey is None else (win, wout, W)
    pair = amount / (2 * T) * (cnt.double() / (s[i] * s[j]))
    split = torch.bincount(i, pair, minlength=K) + torch.bincount(j, pair, minlength=K)
    here = size > 0
    one = s.clamp(min=1)
    dens = torch.where(size > 1, 2 * a / (one * (one - 1)).clamp(min=1), torch.zeros_like(s))
    vol = (2 * A + B) / (2 * T)
    term = A / T * dens - (vol * dens) ** 2 - split
    cond = torch.where(2 * a + b > 0, b / (2 * a + b).clamp(min=1), torch.zeros_like(s))
    k = int(here.sum())

    def mean(x):
        return float(x[here].sum()) / k

    q = {"n_nodes": n, "n_edges": E, "n_communities_nonempty": k, "intra_edges_total": int(ein.sum()),
         "cut_edges_total": cut, "n_community_pairs": key.numel(), "pair_count_sq_sum": int((cnt * cnt).sum()),
         "modularity": float((A / T - vol ** 2)[here].sum()), "modularity_density": float(term[here].sum()),
         "mean_intra_edges": mean(a), "mean_intra_density": mean(dens), "mean_contraction": mean(2 * a / one),
         "mean_inter_edges": mean(b), "mean_expansion": mean(b / one), "mean_conductance": mean(cond)}
    zero = torch.zeros_like(s)
    per = {"size": size, "intra_edges": ein, "inter_edges": eout, "intra_density": dens,
           "contraction": torch.where(here, 2 * a / one, zero), "expansion": torch.where(here, b / one, zero),
           "conductance": cond, "qds_term": torch.where(here, term, zero)}
    return q, per


def _score(row_ptr, col, labels, K, weights=None):
    n = labels.numel()
    size = torch.bincount(labels, minlength=K)
    ein, eout = (torch.zeros(K, dtype=torch.int64, device="cuda") for _ in range(2))
    win, wout = (torch.zeros(K, dtype=torch.float64, device="cuda") for _ in range(2))
    keys, wts = [], []
    for lo in range(0, n, _PIECE):
        hi = min(n, lo + _PIECE)
        a, b = int(row_ptr[lo]), int(row_ptr[hi])
        ls = torch.repeat_interleave(labels[lo:hi], row_ptr[lo + 1:hi + 1] - row_ptr[lo:hi])
        ld = labels[col[a:b]]
        same = ls == ld
        ein += torch.bincount(ls[same], minlength=K)
        eout += torch.bincount(ls[~same], minlength=K)
        up = ls < ld
        keys.append(ls[up].long() * K + ld[up])
        if weights is not None:
            w = weights[a:b].double()
            win += torch.bincount(ls[same], w[same], minlength=K)
            wout += torch.bincount(ls[~same], w[~same], minlength=K)
            wts.append(w[up])
        del ls, ld, same, up
    ein //= 2
    keys = torch.cat(keys)
    if weights is None:
        key, cnt = torch.unique(keys, return_counts=True)
        return _quality(n, col.numel() // 2, size, ein, eout, int(eout.sum()) // 2, key, cnt)
    key, inv, cnt = torch.unique(keys, return_inverse=True, return_counts=True)
    return _quality(n, col.numel() // 2, size, ein, eout, int(eout.sum()) // 2, key, cnt,
                    torch.bincount(inv, torch.cat(wts), minlength=key.numel()), float(weights.double().sum()) / 2,
                    win / 2, wout)


def _indices(n, na, nb, key, cnt, a11, sa2, sb2):
    """Eqs. (1)-(7) from the cells (key = truth * kb + found) and the pair counts."""
    kb = nb.numel()
    i, j, x = key // kb, key % kb, cnt.double()
    sa, sb = na.double()[i], nb.double()[j]
    vi = -float((x * torch.log(x * x / (sa * sb))).sum()) / n
    num = float((x / n * torch.log(x * n / (sa * sb))).sum())
    den = _entropy(na[na > 0].double() / n) + _entropy(nb[nb > 0].double() / n)
    best = torch.zeros(na.numel(), dtype=torch.float64, device="cuda").scatter_reduce_(
        0, i, 2 * x / (sa + sb), "amax")
    rmax = torch.zeros_like(na).scatter_reduce_(0, i, cnt, "amax")
    cmax = torch.zeros_like(nb).scatter_reduce_(0, j, cnt, "amax")
    nvd = int(rmax.sum()) + int(cmax.sum())
    pairs = n * (n - 1) // 2
    a10, a01 = sa2 - a11, sb2 - a11
    a00 = pairs - a11 - a10 - a01
    M = sa2 * sb2 / pairs
    down = 0.5 * (sa2 + sb2) - M
    return {"n_nodes": n, "k_truth": int((na > 0).sum()), "k_found": int((nb > 0).sum()), "n_cells": key.numel(),
            "a11": a11, "a10": a10, "a01": a01, "a00": a00, "nvd_sum": nvd, "vi": vi,
            "nmi": -2 * num / den if den else 1.0, "f_measure": float((na * best).sum()) / n,
            "nvd": 1 - nvd / (2 * n), "ri": (a11 + a00) / pairs, "ari": (a11 - M) / down if down else 1.0,
            "ji": a11 / (a11 + a10 + a01) if a11 + a10 + a01 else 1.0}


def _choose2(x):
    return int((x * (x - 1) // 2).sum())


def _compare(truth, found, ka, kb):
    na, nb = torch.bincount(truth, minlength=ka), torch.bincount(found, minlength=kb)
    key, cnt = torch.unique(truth.long() * kb + found, return_counts=True)
    return _indices(truth.numel(), na, nb, key, cnt, _choose2(cnt), _choose2(na), _choose2(nb))


def _lists(cover):
    """The cover's lists (one or two ids per node) as [n, 2], -1 where there is no second."""
    mptr, memb = cover
    first = memb[mptr[:-1]].long()
    two = mptr[1:] - mptr[:-1] > 1
    second = torch.where(two, memb[(mptr[:-1] + 1).clamp(max=memb.numel() - 1)].long(), -1)
    return torch.stack([first, second], 1)


def _score_cover(row_ptr, col, cover, K):
    M = _lists(cover)
    n = M.shape[0]
    size = torch.bincount(M[M >= 0], minlength=K)
    A = torch.repeat_interleave(M, row_ptr[1:] - row_ptr[:-1], dim=0)
    B = M[col]
    in_b = (A[:, :, None] == B[:, None, :]).any(2) & (A >= 0)  # ids of the near end that the far end has too
    in_a = (B[:, :, None] == A[:, None, :]).any(2) & (B >= 0)
    ein = torch.bincount(A[in_b], minlength=K) // 2
    eout = torch.bincount(A[~in_b & (A >= 0)], minlength=K)
    keys = []
    for x in range(2):
        for y in range(2):
            ok = (A[:, x] >= 0) & (B[:, y] >= 0) & ~in_b[:, x] & ~in_a[:, y] & (A[:, x] < B[:, y])
            keys.append(A[ok, x] * K + B[ok, y])
    key, cnt = torch.unique(torch.cat(keys), return_counts=True)
    return _quality(n, col.numel() // 2, size, ein, eout, int(eout.sum()), key, cnt)[0]


def _groups(M, K):
    """Per node its ids and, where it has two, an id of that pair (-1 else): a pair of nodes shares
    [ids in common] - [pairs in common] of them, which is 1 when they share any and 0 when none."""
    both = M[:, 1] >= 0
    pair = torch.full_like(M[:, 0], -1)
    pair[both] = K + torch.unique(M[both, 0] * K + M[both, 1], return_inverse=True)[1]
    return torch.cat([M, pair[:, None]], 1)


def _together(columns):
    """Node pairs that are together, from (key per node, sign) columns: signed sums of C(count, 2)."""
    return sum(sign * _choose2(torch.unique(k, return_counts=True)[1]) for k, sign in columns)


def _compare_covers(truth, found, ka, kb, n):
    A, B = _lists(truth), _lists(found)
    na, nb = torch.bincount(A[A >= 0], minlength=ka), torch.bincount(B[B >= 0], minlength=kb)
    cells = torch.cat([(A[:, x] * kb + B[:, y])[(A[:, x] >= 0) & (B[:, y] >= 0)] for x in range(2) for y in range(2)])
    key, cnt = torch.unique(cells, return_counts=True)
    GA, GB = _groups(A, ka), _groups(B, kb)
    wide = int(GB.max()) + 1

    def ids(G):  # the two id columns together (one kind of key), the pair column apart
        return [(G[:, :2], 1), (G[:, 2:], -1)]

    def flat(G):
        return G[G >= 0]

    sa2 = _together([(flat(g), s) for g, s in ids(GA)])
    sb2 = _together([(flat(g), s) for g, s in ids(GB)])
    cross = []
    for ga, sx in ids(GA):
        for gb, sy in ids(GB):
            x, y = ga[:, :, None].expand(-1, -1, gb.shape[1]), gb[:, None, :].expand(-1, ga.shape[1], -1)
            ok = (x >= 0) & (y >= 0)
            cross.append((x[ok] * wide + y[ok], sx * sy))
    return _indices(n, na, nb, key, cnt, _together(cross), sa2, sb2)


def exact(case, seed):
    op = case["op"]
    if op == "detect":
        return None  # whole numbers only
    d = _inputs(case, seed)
    if op == "score":
        q, per = _score(d["row_ptr"], d["col"], d["labels"], d["K"], d["weights"])
        return {**q, "per_community": per} if case["communities"] else q
    if op == "compare":
        return _compare(d["truth"], d["found"], d["K"], d["K"])
    if op == "evaluate":
        rows = [(_score(d["row_ptr"], d["col"], lab, k)[0], _compare(d["truth"], lab, d["K"], k))
                for lab, k in zip(d["labels"], d["Ks"])]
        return {"quality": _columns([q for q, _ in rows]), "compare": _columns([c for _, c in rows])}
    if op == "graphs":
        return _columns([_score(g["row_ptr"], g["col"], g["labels"], g["K"])[0] for g in d["graphs"]])
    return {"quality": _score_cover(d["row_ptr"], d["col"], d["found"], d["K"]),
            "compare": _compare_covers(d["truth"], d["found"], d["K"], d["K"], case["n"])}
