"""Buckets of contingency cells that overflow their table again and again: few
found communities and mostly distinct truth labels, so that every bucket is split
into several hash classes and its warps meet the overflow at different places."""
import numpy as np
import pytest
import torch

from helpers import check_compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


# 3 found: buckets of 700,000 nodes; 300: some buckets just above and below the table's 18,432 keys
@pytest.mark.parametrize("kb", [3, 110, 300])
@pytest.mark.parametrize("share", [1, 4])
def test_split_buckets(qm, oracle_mod, kb, share):
    n = (1 << 21) + 12_345
    rng = np.random.default_rng(kb + share)
    a = (rng.permutation(n) // share).astype(np.int32)
    b = rng.integers(0, kb, n).astype(np.int32)
    ka = n // share + 1
    o = oracle_mod.compare(a, b, ka, kb)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    first = qm.compare(da, db, ka, kb)
    check_compare(first, o, f"kb={kb} share={share}")
    for _ in range(5):
        assert qm.compare(da, db, ka, kb) == first


# buckets of 24,700 nodes whose cells stay below the table's limit while half
# full, pass it at the end, or come first and then no more
@pytest.mark.parametrize("share", [0.5, 0.72, 0.76, 0.8, 0.95])
@pytest.mark.parametrize("first", [False, True])
def test_cells_around_the_limit(qm, oracle_mod, share, first):
    n, kb = (1 << 21) + 999, 85  # 24,700 nodes a bucket of one found label
    rng = np.random.default_rng(int(share * 100))
    a = np.where(rng.random(n) < share, rng.permutation(n), 0)
    b = np.repeat(rng.permutation(kb), n // kb + 1)[:n]
    if first:  # within every found community the distinct truths first
        order = np.lexsort((a == 0, b))
        a, b = a[order], b[order]
    else:
        order = rng.permutation(n)
        a, b = a[order], b[order]
    a, b = a.astype(np.int32), b.astype(np.int32)
    c = qm.compare(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), n, kb)
    check_compare(c, oracle_mod.compare(a, b, n, kb), f"share={share}")
