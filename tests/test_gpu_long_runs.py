"""Runs beyond the block tables of phase B, which take one block of 1,024 threads
each with classes of keys sized by the distinct keys a run can have: many entries of few
keys, more keys than one pass holds (13,984), one giant community among small
ones, several long runs beside runs of every other class, and covers.  Counts
must equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

from helpers import check_quality, csr_from_edges, star

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


def check(qm, oracle_mod, rp, col, lab, K, what):
    graph = qm.Graph(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda())
    dev = torch.from_numpy(lab).cuda()
    o = oracle_mod.score(rp, col, lab, K)
    check_quality(qm.score(graph, dev, K), o, what)
    check_quality(qm.score(graph, dev, K, per_community=True), o, what + ", per community")
    mptr = torch.arange(lab.size + 1, dtype=torch.int64, device="cuda")
    c = qm.score_cover(graph, (mptr, dev), K)
    assert c.pop("cut_edges_total") == 2 * o["cut_edges_total"]  # a cover counts a boundary edge from both sides
    check_quality({**c, "cut_edges_total": o["cut_edges_total"]}, o, what + ", cover")
    graph.close()


@pytest.mark.parametrize("keys", [1, 7, 13_984, 13_985, 40_000, 300_000])
@pytest.mark.parametrize("spread", [1, 3])  # 3: ids between the used ones
def test_one_long_run(qm, oracle_mod, keys, spread):
    m = 300_000
    rp, col = star(m)
    lab = np.zeros(m + 1, np.int32)
    lab[1:] = (1 + np.arange(m) % keys) * spread
    check(qm, oracle_mod, rp, col, lab, keys * spread + 1, f"keys={keys} spread={spread}")


@pytest.mark.parametrize("K", [3, 40, 5000, (1 << 19) + 5])
def test_long_runs_beside_others(qm, oracle_mod, K):
    rng = np.random.default_rng(K)
    n = 60_000
    hubs = np.repeat(np.arange(12), 20_000)
    edges = np.concatenate([rng.integers(0, n, (300_000, 2)), np.stack([hubs, rng.integers(0, n, hubs.size)], 1)])
    rp, col = csr_from_edges(n, edges)
    lab = rng.integers(0, K, n).astype(np.int32)
    lab[:12] = np.arange(12) % K
    lab[rng.random(n) < 0.4] = K // 2  # one giant community
    check(qm, oracle_mod, rp, col, lab, K, f"K={K}")
