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
