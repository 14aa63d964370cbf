"""Covers around the list length up to which they are scored in node order (16): the
longest list just at it and just beyond, on nodes apart and on neighbours."""
import numpy as np
import pytest
import torch

from helpers import check_compare, check_quality, csr_from_edges, random_graph, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


@pytest.mark.parametrize("longest", [15, 16, 17, 300])
@pytest.mark.parametrize("where", ["first", "last", "every 100th", "neighbours"])
def test_longest_list(qm, oracle_mod, longest, where):
    n, K = 5003, 700
    rp, col = random_graph(n, 40_000, seed=longest)
    rng = np.random.default_rng(longest)
    lengths = rng.integers(0, 3, n)
    at = {"first": [0], "last": [n - 1], "every 100th": range(0, n, 100),
          "neighbours": np.unique(np.append(col[rp[7]:rp[8]], 7))}[where]
    lengths[list(at)] = longest
    mptr = np.zeros(n + 1, np.int64)
    mptr[1:] = np.cumsum(lengths)
    memb = np.concatenate([np.sort(rng.choice(K, int(x), replace=False)) for x in lengths]).astype(np.int32)
    o = oracle_mod.score_cover(rp, col, mptr, memb, K)
    dev = (torch.from_numpy(mptr).cuda(), torch.from_numpy(memb).cuda())
    for reorder in (False, True):
        graph = qm.Graph(*to_dev(rp, col), reorder=reorder)
        check_quality(qm.score_cover(graph, dev, K), o, f"{where} reorder={reorder}")
        graph.close()


# members of one community that are in others too: their pairs are enumerated as a
# rectangle; beyond 2,048 of them the whole member list is
@pytest.mark.parametrize("L", [1, 2, 3, 32, 33, 255, 256, 257, 1000, 2048, 2049])
def test_pairs_of_overlapping_members(qm, oracle_mod, L):
    n = 2600
    rng = np.random.default_rng(L)

    def side(shared):
        lists = [[2 + int(rng.integers(0, 40))] for _ in range(n)]
        for u in rng.choice(n, shared, replace=False):  # in community 0 and its own, some in 1 too
            lists[u] = [0] + ([1] if rng.random() < 0.5 else []) + lists[u]
        mptr = np.zeros(n + 1, np.int64)
        mptr[1:] = np.cumsum([len(x) for x in lists])
        return mptr, np.concatenate(lists).astype(np.int32)

    a, b = side(L), side(max(1, L // 2))
    o = oracle_mod.compare_cover(a[0], a[1], 42, b[0], b[1], 42)
    dev = [tuple(torch.from_numpy(x).cuda() for x in s) for s in (a, b)]
    check_compare(qm.compare_covers(dev[0], 42, dev[1], 42, n), o, f"L={L}")


@pytest.mark.parametrize("m", [8191, 8192, 8193, 60_000])  # 8,192 arcs: the longest row a warp walks alone
def test_hub_rows(qm, oracle_mod, m):
    rng = np.random.default_rng(m)
    n = m + 3
    edges = [np.stack([np.full(m, h), rng.permutation(n)[:m]], 1) for h in (0, n // 2, n - 1)]
    # hubs of m arcs or a few more (the other hubs'), and some other edges
    rp, col = csr_from_edges(n, np.concatenate(edges + [rng.integers(0, n, (2 * n, 2))]))
    K = 300
    lengths = rng.integers(0, 3, n)
    lengths[[0, n // 2]] = [5, 0]
    mptr = np.zeros(n + 1, np.int64)
    mptr[1:] = np.cumsum(lengths)
    memb = np.concatenate([np.sort(rng.choice(K, int(x), replace=False)) for x in lengths]).astype(np.int32)
    o = oracle_mod.score_cover(rp, col, mptr, memb, K)
    dev = (torch.from_numpy(mptr).cuda(), torch.from_numpy(memb).cuda())
    for reorder in (False, True):
        graph = qm.Graph(*to_dev(rp, col), reorder=reorder)
        check_quality(qm.score_cover(graph, dev, K), o, f"m={m} reorder={reorder}")
        graph.close()


# 32,768 memberships of both covers: the most whose logarithms are formed per cell
@pytest.mark.parametrize("n", [16_384, 16_385])
def test_comparisons_with_and_without_tables(qm, oracle_mod, n):
    rng = np.random.default_rng(n)
    a, b = rng.integers(0, 90, n).astype(np.int32), rng.integers(0, 70, n).astype(np.int32)
    mptr = np.arange(n + 1, dtype=np.int64)
    o = oracle_mod.compare_cover(mptr, a, 90, mptr, b, 70)
    dev = [(torch.from_numpy(mptr).cuda(), torch.from_numpy(x).cuda()) for x in (a, b)]
    c = qm.compare_covers(dev[0], 90, dev[1], 70, n)
    check_compare(c, o, f"n={n}")
    assert c == qm.compare(dev[0][1], dev[1][1], 90, 70)  # a cover of one community a node: the partition's bits
