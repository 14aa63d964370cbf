"""Few communities whose labels do not follow the stored order: members and arcs
counted in shared memory by the passes that permute the labels, around the
number of ids up to which they are, through the one gather and through the two
bucket passes."""
import numpy as np
import pytest
import torch

from helpers import check_quality, random_graph, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


# 2,048 ids: the most that are counted in shared memory
@pytest.mark.parametrize("K", [1, 2, 33, 2047, 2048, 2049])
@pytest.mark.parametrize("bits", [None, (8, 8), (12, 11)])  # windows and tiles of the bucket passes
def test_counts_beside_the_permutation(qm, oracle_mod, K, bits):
    n = 20_011
    rp, col = random_graph(n, 60_000, seed=K)
    try:
        if bits:
            qm.debug_set_perm_buckets(*bits, 0)
        graph = qm.Graph(*to_dev(rp, col), reorder=True)
    finally:
        qm.debug_set_perm_buckets(-1, -1, -1)
    rng = np.random.default_rng(K)
    for lab in (rng.integers(0, K, n), np.arange(n) * K // n, np.where(rng.random(n) < 0.9, 0, K - 1)):
        lab = lab.astype(np.int32)
        o = oracle_mod.score(rp, col, lab, K)
        dev = torch.from_numpy(lab).cuda()
        check_quality(qm.score(graph, dev, K), o, f"K={K}")
        q = qm.score(graph, dev, K, per_community=True)
        assert np.array_equal(q["per_community"]["size"].cpu().numpy(), np.bincount(lab, minlength=K))
    bad = torch.from_numpy(lab).cuda()
    bad[n - 1] = K
    with pytest.raises(qm.QmError) as e:
        qm.score(graph, bad, K)
    assert e.value.status == qm.QM_EINVAL
    graph.close()


# 256 ids: the most whose weights a block adds up in shared memory; 600,000 edges: long rows
@pytest.mark.parametrize("K", [2, 9, 255, 256, 257])
@pytest.mark.parametrize("n,m", [(20_011, 60_000), (6_007, 600_000)])
@pytest.mark.parametrize("reorder", [False, True])
def test_weights_of_few_communities(qm, oracle_mod, K, n, m, reorder):
    rp, col = random_graph(n, m, seed=K)
    src = np.repeat(np.arange(n), np.diff(rp))
    key = np.minimum(src, col) * np.int64(n) + np.maximum(src, col)
    rng = np.random.default_rng(K)
    # over the whole accepted range, so that sums carry from word to word
    w = np.exp2(rng.uniform(-20, 19.99, n * 3))[key % (3 * n)].astype(np.float32)
    graph = qm.Graph(*to_dev(rp, col), weights=torch.from_numpy(w).cuda(), reorder=reorder, validate=True)
    for lab in (rng.integers(0, K, n), np.arange(n) * K // n, np.arange(n) // 12 % K):
        lab = lab.astype(np.int32)
        o = oracle_mod.score_weighted(rp, col, w.astype(np.float64), lab, K)
        q = qm.score(graph, torch.from_numpy(lab).cuda(), K)
        for name, cond in (("modularity", "cond_modularity"), ("modularity_density", "cond_modularity_density")):
            assert abs(q[name] - o[name]) <= 1e-12 * max(abs(o[name]), abs(o[cond])), (name, q[name], o[name])
    graph.close()
