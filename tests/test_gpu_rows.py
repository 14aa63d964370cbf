"""Phase A in stored node order: chunks of 32 nodes with one, few and many
stretches of one label, more arcs than a mixed chunk's table holds, ragged last
chunks and blocks, isolated nodes, few and many label ids (volumes counted in
shared memory and in global memory), and the block encoding with one, two and
more labels a block and with too many of the latter.  Every result must equal
the one-kernel pipeline's bit for bit and match the oracle."""
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


def patterns(n, rng):
    i = np.arange(n)
    yield "one label", np.zeros(n, np.int64), 1
    for run in (1, 3, 9, 16, 40):
        yield f"stretches of {run}", i // run, n // run + 1
    yield "two labels in turn", i % 2, 2
    yield "random few", rng.integers(0, 7, n), 7
    yield "random many", rng.integers(0, 7000, n), 7000  # beyond the ids counted in shared memory
    lab = i // 50
    lab[rng.integers(0, n, max(1, n // 60))] = 0         # stretches with strays
    yield "stretches with strays", lab, n // 50 + 1


@pytest.mark.parametrize("n,m", [(2, 1), (33, 60), (47, 100), (1000, 4000), (5003, 200_000)])
def test_label_patterns(qm, oracle_mod, n, m):
    rng = np.random.default_rng(n)
    rp, col = random_graph(n, m, seed=n)
    if len(col) == 0:
        rp, col = np.array([0, 1, 2], np.int64), np.array([1, 0], np.int32)
    rp = np.concatenate([rp, np.full(37, rp[-1])])  # isolated nodes at the end
    plain = qm.Graph(*to_dev(rp, col))
    reord = qm.Graph(*to_dev(rp, col), reorder=True)
    for name, lab, K in patterns(n + 37, rng):
        lab = torch.from_numpy(lab.astype(np.int32)).cuda()
        o = oracle_mod.score(rp, col, lab.cpu().numpy(), K)
        qm.set_tuning(plain, K, 512, 96 * 1024, 48, 0)
        ref = qm.score(plain, lab, K)
        check_quality(ref, o, f"n={n} {name}")
        for graph in (plain, reord):
            for algo in (1, 4):
                qm.set_tuning(graph, K, 512, 96 * 1024, 48, algo)
                assert qm.score(graph, lab, K) == ref, (n, name, algo)
                q = qm.score(graph, lab, K, per_community=True)
                assert int(q.pop("per_community")["size"].sum()) == n + 37 and q == ref, (n, name, algo)


@pytest.mark.parametrize("n", [4096, 4103])
def test_block_encoding_of_a_renumbered_graph(qm, oracle_mod, n):
    """The renumbering of a random graph moves few nodes together, so labels laid
    out along the caller's order reach the stored order in many mixes."""
    rng = np.random.default_rng(n)
    rp, col = random_graph(n, 6 * n, seed=n + 1)
    reord = qm.Graph(*to_dev(rp, col), reorder=True)
    plain = qm.Graph(*to_dev(rp, col))
    cases = [np.arange(n) // 64, np.arange(n) // 20, np.arange(n) // 6, np.arange(n)]
    # a sixth of the blocks may hold three labels or more: just below and above
    for share in (0.12, 0.25):
        lab = np.zeros(n, np.int64)
        for b in np.nonzero(rng.random(n // 16) < share)[0]:
            lab[16 * b:16 * b + 16] = 1 + rng.integers(0, 50, 16)
        cases.append(lab)
    for lab in cases:
        K = int(lab.max()) + 1
        lab = torch.from_numpy(lab.astype(np.int32)).cuda()
        qm.set_tuning(plain, K, 512, 96 * 1024, 48, 0)
        ref = qm.score(plain, lab, K)
        check_quality(ref, oracle_mod.score(rp, col, lab.cpu().numpy(), K), f"K={K}")
        qm.set_tuning(reord, K, 512, 96 * 1024, 48, 4)
        assert qm.score(reord, lab, K) == ref, K
