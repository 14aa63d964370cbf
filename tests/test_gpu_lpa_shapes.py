"""Label propagation at the sizes at which a warp takes 4, 8, 16 and 32 nodes (the
last with rounds that decide most nodes by votes over packed slots): isolated
nodes, sampled rows (degree above 32), ragged last warps; labels and their count
equal the oracle's."""
import numpy as np
import pytest

from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 2_049, 300_007, 700_001, 1_300_021])
@pytest.mark.parametrize("clusters", [1, 40])  # of no structure, and of clusters of 40 nodes
def test_sizes_of_every_shape(oracle_mod, n, clusters):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm
    rng = np.random.default_rng(n + clusters)
    m = 4 * n
    a = rng.integers(0, n, m)
    b = a // clusters * clusters + rng.integers(0, clusters, m) if clusters > 1 else rng.integers(0, n, m)
    far = rng.random(m) < 0.2
    b = np.where(far, rng.integers(0, n, m), np.minimum(b, n - 1))
    hubs = np.stack([np.repeat(np.arange(0, n, max(1, n // 50)), 60), rng.integers(0, n, 60 * len(range(0, n, max(1, n // 50))))], 1)
    edges = np.concatenate([np.stack([a, b], 1), hubs])
    edges = edges[(edges[:, 0] % 97 != 13) & (edges[:, 1] % 97 != 13)]  # some nodes stay alone
    key = np.unique(np.minimum(*edges.T) * n + np.maximum(*edges.T))
    lo, hi = key // n, key % n
    lo, hi = lo[lo != hi], hi[lo != hi]
    src, dst = np.concatenate([lo, hi]), np.concatenate([hi, lo])
    order = np.argsort(src * n + dst)
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(src, minlength=n))
    col = dst[order].astype(np.int32)
    for rounds in (1, 4, 7):
        ref, k_ref = oracle_mod.label_propagation(rp, col, rounds)
        for reorder in (False, True):
            lab, k = qm.label_propagation(qm.Graph(*to_dev(rp, col), reorder=reorder), rounds)
            assert k == k_ref and np.array_equal(lab.cpu().numpy(), ref), (rounds, reorder)
