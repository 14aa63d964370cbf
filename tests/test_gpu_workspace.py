"""The scratch of a scoring call: the plain pipeline reserves no member array and no arc
offsets, and what qm_workspace_bytes reports covers every algorithm of the graph
that gathers directly."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_no_member_array_for_the_walk_by_rows():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import gen, qm
    g = gen.lfr_graph(gen.LfrParams(n=4_000_000, k_mean=4, k_max=10, s_min=20, s_max=1000, mu=0.3, seed=2), device="cuda")
    graph = qm.Graph(g.row_ptr, g.col)
    need = qm.workspace_bytes(graph, g.K)
    results, taken = [], []
    for algo in (1, 7, 5):
        sh = qm.get_tuning(graph, g.K)
        qm.set_tuning(graph, g.K, sh["threads"], sh["smem_bytes"], sh["big_community"], algo)
        qm.release_cache()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        results.append(qm.score(graph, g.labels, g.K))
        taken.append(before - torch.cuda.mem_get_info()[0])
    assert results[0] == results[1] == results[2]
    slack = 16 << 20  # the allocator's granularity, pinned blocks and module memory
    assert all(t <= need + slack for t in taken), (taken, need)
    # the half-edge call alone keeps the members, 4 bytes a node
    assert taken[1] - taken[0] >= 4 * g.labels.numel() - slack, taken
    graph.close()
