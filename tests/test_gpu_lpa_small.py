"""Label propagation on graphs around a warp's 32 consecutive nodes: isolated
nodes among them, ties between the own label, half and less of the neighbours,
sampled rows (degree above 32); labels and their count equal the oracle's."""
import numpy as np
import pytest

from helpers import csr_from_edges, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 100])
def test_small_random_graphs_round_by_round(oracle_mod, n):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm
    rng = np.random.default_rng(n)
    edges = rng.integers(0, n + 1, (6 * n + 2, 2)).tolist() + [[n, n + 1]]
    if n > 32:
        edges += [[0, v] for v in range(1, n)]
    rp, col = csr_from_edges(n + 3, edges)
    for rounds in (1, 2, 3, 5):
        ref, k_ref = oracle_mod.label_propagation(rp, col, rounds)
        for reorder in (False, True):
            lab, k = qm.label_propagation(qm.Graph(*to_dev(rp, col), reorder=reorder), rounds)
            assert k == k_ref and np.array_equal(lab.cpu().numpy(), ref), (n, rounds, reorder)
