"""Covers scored by packed runs in node order: chunks of nodes with more arcs
than a chunk's table holds, lists of several lengths and empty ones, runs whose
segments just fit and do not fit the scratch (those are scored by member
lists), few and many label ids; each against the oracle, on the graph as given
and renumbered, and comparisons whose communities share one found id."""
import numpy as np
import pytest
import torch

from helpers import check_compare, check_quality, random_graph, star, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


def cover(n, K, lengths, rng):
    """Every node in as many distinct communities as lengths says."""
    mptr = np.zeros(n + 1, np.int64)
    mptr[1:] = np.cumsum(lengths)
    memb = np.concatenate([np.sort(rng.choice(K, int(x), replace=False)) for x in lengths]).astype(np.int32)
    return mptr, memb


@pytest.mark.parametrize("n,m,K", [(33, 60, 5), (1000, 5000, 40), (1000, 5000, 5000), (3001, 150_000, 200)])
@pytest.mark.parametrize("kind", ["ones", "up to two", "empty and three", "long"])
def test_lists_of_all_lengths(qm, oracle_mod, n, m, K, kind):
    rng = np.random.default_rng(n + len(kind))
    rp, col = random_graph(n, m, seed=n)
    if kind == "ones":
        lengths = np.ones(n, np.int64)
    elif kind == "up to two":
        lengths = 1 + (rng.random(n) < 0.3)
    elif kind == "empty and three":
        lengths = rng.integers(0, 4, n)
    else:  # hubs of the graph in many communities: the segments outgrow the scratch
        lengths = np.ones(n, np.int64)
        lengths[np.argsort(np.diff(rp))[-max(1, n // 20):]] = min(K, 60)
    mptr, memb = cover(n, K, lengths, rng)
    o = oracle_mod.score_cover(rp, col, mptr, memb, K)
    dev = (torch.from_numpy(mptr).cuda(), torch.from_numpy(memb).cuda())
    for reorder in (False, True):
        graph = qm.Graph(*to_dev(rp, col), reorder=reorder)
        check_quality(qm.score_cover(graph, dev, K), o, f"{kind} n={n} reorder={reorder}")
    found = cover(n, 7, np.minimum(lengths, 3), rng)
    check_compare(qm.compare_covers(dev, K, tuple(torch.from_numpy(x).cuda() for x in found), 7, n),
                  oracle_mod.compare_cover(mptr, memb, K, found[0], found[1], 7), f"{kind} n={n} compare")


def test_hub_with_a_long_list(qm, oracle_mod):
    """A star whose hub is in 3,000 communities: the leaves' segments hold the
    hub's list each."""
    rng = np.random.default_rng(5)
    rp, col = star(2000)
    lengths = np.ones(2001, np.int64)
    lengths[0] = 3000
    mptr, memb = cover(2001, 4000, lengths, rng)
    graph = qm.Graph(*to_dev(rp, col))
    dev = (torch.from_numpy(mptr).cuda(), torch.from_numpy(memb).cuda())
    check_quality(qm.score_cover(graph, dev, 4000), oracle_mod.score_cover(rp, col, mptr, memb, 4000), "hub")
    big = (1 << 20) + 5  # ids for which only the member lists are used
    check_quality(qm.score_cover(graph, dev, big), oracle_mod.score_cover(rp, col, mptr, memb, big), "many ids")
