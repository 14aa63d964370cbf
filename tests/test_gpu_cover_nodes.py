"""Covers at the sizes from which they are scored in node order (2^20 arcs, or 2^12
arcs a label id): lists of several lengths and empty ones, the longest list at its bound
and beyond, chunks with more arcs than a chunk's table holds, hub rows, on the
graph as given and renumbered; and the two sides of each bound."""
import numpy as np
import pytest
import torch

from helpers import check_quality, csr_from_edges, random_graph, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


def check(qm, oracle_mod, rp, col, lengths, K, rng, what):
    mptr = np.zeros(lengths.size + 1, np.int64)
    mptr[1:] = np.cumsum(lengths)
    first = rng.integers(0, K, lengths.size)
    owner = np.repeat(np.arange(lengths.size), lengths)
    ids = (first[owner] + (np.arange(mptr[-1]) - mptr[owner]) * max(1, K // 17)) % K  # distinct within a list of <= 17
    memb = ids[np.lexsort((ids, owner))].astype(np.int32)
    o = oracle_mod.score_cover(rp, col, mptr, memb, K)
    dev = (torch.from_numpy(mptr).cuda(), torch.from_numpy(memb).cuda())
    for reorder in (False, True):
        graph = qm.Graph(*to_dev(rp, col), reorder=reorder)
        check_quality(qm.score_cover(graph, dev, K), o, f"{what} reorder={reorder}")
        graph.close()


@pytest.mark.parametrize("kind", ["ones", "up to two", "empty and three", "16 now and then", "17 now and then"])
@pytest.mark.parametrize("n,m,K", [(50_001, 560_000, 900), (6_007, 600_000, 300), (6_007, 600_000, 17)])
def test_lists_of_all_lengths(qm, oracle_mod, n, m, K, kind):
    rng = np.random.default_rng(n + len(kind))
    rp, col = random_graph(n, m, seed=n)
    assert len(col) > 1 << 20
    lengths = np.ones(n, np.int64)
    if kind == "up to two":
        lengths += rng.random(n) < 0.3
    elif kind == "empty and three":
        lengths = rng.integers(0, 4, n)
    elif "now" in kind:
        lengths[::n // 60] = int(kind[:2])
    check(qm, oracle_mod, rp, col, np.minimum(lengths, K), K, rng, f"{kind} n={n}")


@pytest.mark.parametrize("K", [1, 2, 19, 20])  # 81,920 arcs: 20 ids at 2^12 arcs each
def test_few_communities(qm, oracle_mod, K):
    rng = np.random.default_rng(K)
    rp, col = csr_from_edges(4096, np.stack([np.repeat(np.arange(4096), 10), np.tile(np.arange(1, 11), 4096)], 1)
                             @ np.array([[1, 1], [0, 1]]) % 4096)
    assert len(col) == 81_920
    for lengths in (np.ones(4096, np.int64), rng.integers(0, min(K, 3) + 1, 4096)):
        if lengths.sum():
            check(qm, oracle_mod, rp, col, lengths, K, rng, f"K={K}")


@pytest.mark.parametrize("m", [8_190, 8_192, 60_000])  # 8,192 arcs: the longest row a warp walks alone
def test_hub_rows(qm, oracle_mod, m):
    rng = np.random.default_rng(m)
    n = m + 3
    hubs = [np.stack([np.full(m, h), rng.permutation(n)[:m]], 1) for h in (0, n // 2, n - 1)]
    rp, col = csr_from_edges(n, np.concatenate(hubs + [rng.integers(0, n, (700_000, 2))]))
    assert len(col) > 1 << 20
    lengths = rng.integers(0, 3, n)
    lengths[[0, n // 2]] = [16, 0]
    check(qm, oracle_mod, rp, col, lengths, 300, rng, f"m={m}")
