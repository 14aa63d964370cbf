"""Weighted scoring with more label ids than the one-word tables leave 12 bits of
repeats for: runs at the longest that a word still takes, beyond it, and many
short ones, against the oracle."""
import numpy as np
import pytest
import torch

from helpers import random_graph, star, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


def check(qm, oracle_mod, rp, col, lab, K, seed):
    n = len(rp) - 1
    src = np.repeat(np.arange(n), np.diff(rp))
    key = np.minimum(src, col) * np.int64(n) + np.maximum(src, col)
    w = np.exp2(np.random.default_rng(seed).uniform(-20, 19.9, 4096))[key * 2654435761 % 4093].astype(np.float32)
    graph = qm.Graph(*to_dev(rp, col), weights=torch.from_numpy(w).cuda(), validate=True)
    o = oracle_mod.score_weighted(rp, col, w.astype(np.float64), lab, K)
    u = oracle_mod.score(rp, col, lab, K)
    q = qm.score(graph, torch.from_numpy(lab).cuda(), K)
    for name, cond in (("modularity", "cond_modularity"), ("modularity_density", "cond_modularity_density")):
        assert abs(q[name] - o[name]) <= 1e-12 * max(abs(o[name]), abs(o[cond])), (name, q[name], o[name])
    assert q["n_community_pairs"] == u["n_community_pairs"] and q["pair_count_sq_sum"] == u["pair_count_sq_sum"]
    graph.close()


# 2^20 ids: 11 bits for the repeats, runs of up to 2,047 entries; 2^22: 511; 2^24: 127
@pytest.mark.parametrize("K,most", [(1 << 20, 2047), (1 << 22, 511), ((1 << 22) - 1, 1023), (1 << 24, 127)])
def test_runs_around_the_longest(qm, oracle_mod, K, most):
    for m in (most - 1, most, most + 1):
        rp, col = star(m)
        for keys in (1, 2, m):
            lab = np.zeros(m + 1, np.int32)
            lab[1:] = K - 1 - np.arange(m) % keys
            check(qm, oracle_mod, rp, col, lab, K, m)


@pytest.mark.parametrize("K", [1 << 20, 5_000_000])
def test_short_runs(qm, oracle_mod, K):
    n = 30_000
    rp, col = random_graph(n, 100_000, seed=1)
    rng = np.random.default_rng(K)
    lab = np.sort(rng.choice(K, n // 2, replace=False)).astype(np.int32)[rng.integers(0, n // 2, n)]
    check(qm, oracle_mod, rp, col, lab, K, 3)
    lab[rng.random(n) < 0.3] = lab[0]  # and one long run
    check(qm, oracle_mod, rp, col, lab, K, 4)
