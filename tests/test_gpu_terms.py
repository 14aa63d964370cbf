"""The terms of the communities and the results from them, at the edges of the
rules that spread them: numbers of ids where the terms' blocks take twice the
threads (multiples of 32 times the SMs), and numbers of candidates where a
cluster per candidate gets fewer blocks.  Every result must match the oracle and
be the same bits on the plain and the batched path."""
import numpy as np
import pytest
import torch

from helpers import check_compare, check_quality, random_graph, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


@pytest.mark.parametrize("mult", [32, 64, 128, 256])
@pytest.mark.parametrize("step", [0, 1])
def test_terms_block_sizes(qm, oracle_mod, mult, step):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    K = mult * sms + step
    n = K + 100
    rng = np.random.default_rng(K)
    rp, col = random_graph(n, 3 * n, seed=K)
    lab = (rng.permutation(n) % K).astype(np.int32)
    q = qm.score(qm.Graph(*to_dev(rp, col)), torch.from_numpy(lab).cuda(), K)
    check_quality(q, oracle_mod.score(rp, col, lab, K), f"K={K}")


@pytest.mark.parametrize("count", [1, 2, 75, 76, 77, 151, 153, 303, 305, 607, 609])
def test_candidates_per_cluster(qm, oracle_mod, count):
    n, k = 700, 300
    rng = np.random.default_rng(count)
    rp, col = random_graph(n, 4 * n, seed=3)
    truth = torch.from_numpy(rng.integers(0, 40, n).astype(np.int32)).cuda()
    L = torch.from_numpy(rng.integers(0, k, (count, n)).astype(np.int32)).cuda()
    graph = qm.Graph(*to_dev(rp, col))
    oq, oc = qm.evaluate_batched(graph, L, [k] * count, truth, 40)
    assert oq == qm.score_batched(graph, L, [k] * count)
    for p in {0, count // 2, count - 1}:
        assert oq[p] == qm.score(graph, L[p], k)
        assert oc[p] == qm.compare(truth, L[p], 40, k)
        check_quality(oq[p], oracle_mod.score(rp, col, L[p].cpu().numpy(), k), f"p={p}")
        check_compare(oc[p], oracle_mod.compare(truth.cpu().numpy(), L[p].cpu().numpy(), 40, k), f"p={p}")


@pytest.mark.parametrize("k", [1, 2, 31, 33, 64, 129, 300])
def test_candidate_counters_around_the_run_length(qm, oracle_mod, k):
    """Runs with as many entries as counters above the community's id, fewer and
    more: counters read in order, or through the run's entries again."""
    n = 600
    rng = np.random.default_rng(k)
    rp, col = random_graph(n, 9 * n, seed=5)
    L = torch.from_numpy(rng.integers(0, k, (5, n)).astype(np.int32)).cuda()
    graph = qm.Graph(*to_dev(rp, col))
    for p, q in enumerate(qm.score_batched(graph, L, [k] * 5)):
        assert q == qm.score(graph, L[p], k)
        check_quality(q, oracle_mod.score(rp, col, L[p].cpu().numpy(), k), f"p={p}")


@pytest.mark.parametrize("K", [1, 31, 32, 33, 255, 257, 1100])
@pytest.mark.parametrize("reorder", [False, True])
def test_half_edge_members(qm, oracle_mod, K, reorder):
    """Members of each community placed together by warps of 32 ids, empty ones
    among them (algorithm 7), on graphs as given and renumbered."""
    n = 1000
    rng = np.random.default_rng(K)
    rp, col = random_graph(n, 5 * n, seed=K + 1)
    lab = (rng.integers(0, (K + 1) // 2, n) * 2 % K).astype(np.int32)  # about every other id is empty
    graph, d = qm.Graph(*to_dev(rp, col), reorder=reorder), torch.from_numpy(lab).cuda()
    ref = qm.score(graph, d, K)
    check_quality(ref, oracle_mod.score(rp, col, lab, K), f"K={K}")
    qm.set_tuning(graph, K, 512, 96 * 1024, 48, 7)
    assert qm.score(graph, d, K) == ref
    q = qm.score(graph, d, K, per_community=True)
    assert int(q.pop("per_community")["size"].sum()) == n and q == ref
