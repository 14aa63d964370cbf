"""Contingency cells by buckets of found communities (comparisons of more than
2^21 nodes): planted and moved labels, one community on either side, most nodes
in one community, few communities with so many truth labels that a bucket's
cells are counted in several hash classes, label counts around the buckets'
bounds, and labels out of range on either side.  Counts bit-exact against the
oracle, indices within the parity tolerance.  Then small comparisons around the
classes of cells whose terms are formed apart (one node, small products)."""
import numpy as np
import pytest
import torch

from helpers import check_compare

pytestmark = pytest.mark.gpu

N = (1 << 21) + 4099  # a ragged last tile


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


def labels(kind, rng):
    ident = np.arange(N)
    if kind == "moved":
        a = rng.integers(0, 9000, N)
        b = np.where(rng.random(N) < 0.2, rng.integers(0, 9000, N), a)
        return a, b, 9000, 9000
    if kind == "same":
        a = rng.integers(0, 257, N)
        return a, a, 257, 257
    if kind == "one truth":
        return np.zeros(N, np.int64), rng.integers(0, 5000, N), 1, 5000
    if kind == "one found":
        return rng.integers(0, 5000, N), np.zeros(N, np.int64), 5000, 1
    if kind == "skewed":
        b = np.where(rng.random(N) < 0.6, 77, rng.integers(0, 4000, N))
        return rng.integers(0, 50, N), b, 50, 4000
    if kind == "many truths":  # 40 buckets of 52,000 nodes, nearly all cells distinct
        return rng.permutation(ident) // 2, rng.integers(0, 40, N), N // 2 + 1, 40
    if kind == "wide":         # 1024 found labels a bucket, and one more bit than the buckets take
        return rng.integers(0, 1000, N), rng.integers(0, 1 << 18, N), 1000, 1 << 18
    return rng.integers(0, 1000, N), rng.integers(0, (1 << 18) + 1, N), 1000, (1 << 18) + 1


@pytest.mark.parametrize("kind", ["moved", "same", "one truth", "one found", "skewed", "many truths", "wide", "wider"])
def test_large_comparisons(qm, oracle_mod, kind):
    a, b, ka, kb = labels(kind, np.random.default_rng(len(kind)))
    a, b = a.astype(np.int32), b.astype(np.int32)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    o = oracle_mod.compare(a, b, ka, kb)
    c = qm.compare(da, db, ka, kb)
    if min(ka, kb) == 1:
        # NMI is zero and so is every term of the oracle's numerator, which leaves
        # the rule (relative to the sum of |terms|) nothing to be relative to; here
        # a term is a difference of two logarithms below 16, each rounded once:
        # 2^-49 a term at most, weighted by n / N
        assert abs(c["nmi"]) <= 2.0 ** -49 / o["nmi_den_abs"]
        c["nmi"] = o["nmi"]
    check_compare(c, o, kind)
    if kind == "moved":
        for side in (0, 1):
            for bad in (-1, ka):
                x = [da.clone(), db.clone()]
                x[side][N - 5] = bad
                with pytest.raises(qm.QmError) as e:
                    qm.compare(x[0], x[1], ka, kb)
                assert e.value.status == qm.QM_EINVAL
        check_compare(qm.compare(da, db, ka, kb), o, "after refused calls")


@pytest.mark.parametrize("n,ka,kb", [(2, 1, 2), (5, 2, 3), (33, 30, 30), (1000, 900, 3), (20_000, 2, 20_000)])
def test_cells_of_one_node(qm, oracle_mod, n, ka, kb):
    rng = np.random.default_rng(n)
    a, b = rng.integers(0, ka, n).astype(np.int32), rng.integers(0, kb, n).astype(np.int32)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    c = qm.compare(da, db, ka, kb)
    check_compare(c, oracle_mod.compare(a, b, ka, kb), f"n={n}")
    assert qm.compare_batched(da, db[None], ka, kb)[0] == c


# 16,128 nodes: the largest comparison of the one-kernel path
@pytest.mark.parametrize("n", [2, 31, 513, 16_127, 16_128, 16_129])
@pytest.mark.parametrize("kind", ["few", "one found", "distinct", "many ids"])
def test_small_comparisons(qm, oracle_mod, n, kind):
    rng = np.random.default_rng(n)
    ka, kb = {"few": (20, 30), "one found": (9, 1), "distinct": (n, n), "many ids": (1 << 16, (1 << 15) - 1)}[kind]
    a, b = rng.integers(0, ka, n).astype(np.int32), rng.integers(0, kb, n).astype(np.int32)
    if kind == "distinct":
        a, b = rng.permutation(n).astype(np.int32), rng.permutation(n).astype(np.int32)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    c, o = qm.compare(da, db, ka, kb), oracle_mod.compare(a, b, ka, kb)
    assert qm.compare(a, b, ka, kb) == c                            # host labels
    assert qm.compare_batched(da, db[None], ka, kb)[0] == c         # the other path's bits
    if min(c["k_truth"], c["k_found"]) > 1:
        check_compare(c, o, f"{kind} n={n}")
    for bad in (-1, kb):
        x = db.clone()
        x[n - 1] = bad
        with pytest.raises(qm.QmError) as e:
            qm.compare(da, x, ka, kb)
        assert e.value.status == qm.QM_EINVAL
