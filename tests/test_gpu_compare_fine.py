"""Comparisons of two labellings in very small communities around the sizes at which
they leave the one-kernel path (10,000 nodes, communities of 8/3 nodes on
average on both sides): counts bit-exact against the oracle, and the batched
path's bits."""
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


@pytest.mark.parametrize("n", [10_000, 10_001, 16_128])
@pytest.mark.parametrize("k", ["n", "3n/8", "3n/8 - 1"])
def test_fine_labellings(qm, oracle_mod, n, k):
    rng = np.random.default_rng(n)
    kb = {"n": n, "3n/8": -(-3 * n // 8), "3n/8 - 1": -(-3 * n // 8) - 1}[k]
    a = rng.integers(0, n, n).astype(np.int32)
    b = (rng.permutation(n) % kb).astype(np.int32)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    c = qm.compare(da, db, n, kb)
    check_compare(c, oracle_mod.compare(a, b, n, kb), f"n={n} kb={kb}")
    assert qm.compare_batched(da, db[None], n, kb)[0] == c
