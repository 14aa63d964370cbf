"""Phase B with one-word counting tables: runs at the edges of its classes
(single warps, blocks of four warps, staged blocks, the unstaged table, hash
classes), with every key once, every key twice or more and a handful of keys,
with label-id counts at which a word's repeat field narrows, and with ids too
many for the one-word tables.  A star's hub community borders one community a
leaf, so its run has exactly as many entries as leaves; counts must equal the
oracle's bit for bit, the metrics within the parity tolerance, and the
per-community call (which counts every label) must agree."""
import numpy as np
import pytest
import torch

from helpers import check_quality, star

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


# 768 entries: the largest run of a warp; 3,072: of four warps; 6,144: of a
# staged block; 12,288: of the unstaged table
@pytest.mark.parametrize("m", [1, 31, 33, 127, 129, 767, 768, 769, 3071, 3072, 3073, 6144, 6145, 12288, 12289, 20000])
def test_hub_run_lengths(qm, oracle_mod, m):
    rp, col = star(m)
    graph = qm.Graph(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda())
    for keys in sorted({1, min(m, 3), max(1, m // 2), m}):
        lab = np.zeros(m + 1, np.int32)
        lab[1:] = 1 + np.arange(m) % keys
        o = oracle_mod.score(rp, col, lab, keys + 1)
        check_quality(qm.score(graph, torch.from_numpy(lab).cuda(), keys + 1), o, f"m={m} keys={keys}")
        q = qm.score(graph, torch.from_numpy(lab).cuda(), keys + 1, per_community=True)
        check_quality(q, o, f"m={m} keys={keys}, per community")


# 2^18, 2^19: 14, 13 and 12 bits are left for the repeats of a key; 2^20: other tables
@pytest.mark.parametrize("K", [(1 << 18) - 1, 1 << 18, 1 << 19, (1 << 20) - 1, 1 << 20])
@pytest.mark.parametrize("m", [700, 4095, 4096, 9000])
def test_many_label_ids(qm, oracle_mod, K, m):
    rp, col = star(m)
    graph = qm.Graph(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda())
    rng = np.random.default_rng(m)
    for keys in (1, 50, m):
        ids = 1 + np.sort(rng.choice(K - 1, keys, replace=False)).astype(np.int32)
        ids[-1] = K - 1
        lab = np.zeros(m + 1, np.int32)
        lab[1:] = ids[np.arange(m) % keys]
        check_quality(qm.score(graph, torch.from_numpy(lab).cuda(), K), oracle_mod.score(rp, col, lab, K),
                      f"K={K} m={m} keys={keys}")


@pytest.mark.parametrize("m", [1, 33, 96, 97, 768, 769, 3072, 3073, 12288, 12289])
def test_weighted_hub_run_lengths(qm, oracle_mod, m):
    """The weighted count's classes, with weights over the whole accepted range
    (products beyond 64 bits among them)."""
    rp, col = star(m)
    rng = np.random.default_rng(m)
    leaf = np.exp2(rng.uniform(-20, 19.9, m)).astype(np.float32)
    leaf[rng.random(m) < 0.1] = 0.0
    leaf[0] = 1.0
    w = np.concatenate([leaf, leaf])  # the hub's row, then one arc a leaf
    graph = qm.Graph(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), weights=w, validate=True)
    for keys in sorted({1, min(m, 3), max(1, m // 2), m}):
        lab = np.zeros(m + 1, np.int32)
        lab[1:] = 1 + np.arange(m) % keys
        o = oracle_mod.score_weighted(rp, col, w.astype(np.float64), lab, keys + 1)
        q = qm.score(graph, torch.from_numpy(lab).cuda(), keys + 1)
        for name, cond in (("modularity", "cond_modularity"), ("modularity_density", "cond_modularity_density")):
            assert abs(q[name] - o[name]) <= 1e-12 * max(abs(o[name]), abs(o[cond])), (m, keys, name)
        u = oracle_mod.score(rp, col, lab, keys + 1)
        assert q["n_community_pairs"] == u["n_community_pairs"] and q["pair_count_sq_sum"] == u["pair_count_sq_sum"]
