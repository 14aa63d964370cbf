"""Weighted sums of communities of millions of nodes.  Nodes of one parity are
linked among themselves only (u to u +- 2, 4, ..) and the labels are the parity,
so the two communities alternate along the node order, every node's weights are
added to its community's sum apart, and Q_w follows from the weights' exact sums:
    Q_w = sum_c W_c / W - (W_c / W)^2
with fractional weights, whose fixed-point values fill every bit of a sum's low
word.  Then a hub whose row sums to more than 2^81 in a lane."""
from fractions import Fraction

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


def fixed_sum(x):
    """Exact sum of float32 weights as an integer multiple of 2^-43."""
    v = (x.double() * 2.0 ** 43).long()
    return (int((v >> 24).sum()) << 24) + int((v & 0xFFFFFF).sum())


# degree 6: a warp's 32 nodes are walked together; 80: their rows exceed what it
# tabulates, and each stretch of a label is walked apart
@pytest.mark.parametrize("n,half", [(12_000_000, 3), (10_000_000, 40)])
def test_alternating_communities(qm, n, half):
    gen = torch.Generator(device="cuda").manual_seed(half)
    deg = 2 * half
    u = torch.arange(n, dtype=torch.int32, device="cuda")
    edge = torch.rand(half, n, generator=gen, device="cuda") * 4.95 + 0.05  # edge[d - 1][u]: weight of (u, u + 2d)
    col = torch.empty(n, deg, dtype=torch.int32, device="cuda")
    wt = torch.empty(n, deg, dtype=torch.float32, device="cuda")
    for d in range(1, half + 1):
        col[:, half - d] = (u - 2 * d) % n
        wt[:, half - d] = edge[d - 1].roll(2 * d)
        col[:, half + d - 1] = (u + 2 * d) % n
        wt[:, half + d - 1] = edge[d - 1]
    for part in (slice(0, deg), slice(n - deg, n)):  # the rows that wrap around
        order = col[part].argsort(dim=1)
        col[part], wt[part] = col[part].gather(1, order), wt[part].gather(1, order)
    row_ptr = torch.arange(n + 1, dtype=torch.int64, device="cuda") * deg
    graph = qm.Graph(row_ptr, col.view(-1), weights=wt.view(-1))
    W = [sum(fixed_sum(edge[d][p::2]) for d in range(half)) for p in (0, 1)]
    share = [Fraction(x, sum(W)) for x in W]
    dens = Fraction(deg, n // 2 - 1)  # 2 E_in / (s (s - 1))
    for K in (2, 7):
        q = qm.score(graph, (u % 2).contiguous(), K)
        Q = sum(x - x * x for x in share)
        Qds = sum(x * dens - (x * dens) ** 2 for x in share)
        assert abs(q["modularity"] - float(Q)) <= 1e-12 * 2
        assert abs(q["modularity_density"] - float(Qds)) <= 1e-12 * 2 * float(dens)
        assert q["cut_edges_total"] == 0 and q["intra_edges_total"] == n * half
    parts = [qm.score_part(graph, (u % 2).contiguous(), 2, r, 2) for r in range(2)]  # a shard per community
    q = qm.finalize_part(qm.combine_parts(parts))
    assert abs(q["modularity"] - float(Q)) <= 1e-12 * 2
    graph.close()


def test_heavy_hub(qm):
    """A star of 10^7 leaves with the largest weights, one leaf in a community of its own:
    W_0 / W = (m - 1) / m, and vol_0 = (2 m - 1) w, vol_1 = w of 2 W = 2 m w."""
    m = 10_000_000
    leaf = torch.arange(1, m + 1, dtype=torch.int32, device="cuda")
    row_ptr = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"),
                         m + torch.arange(m + 1, dtype=torch.int64, device="cuda")])
    weights = torch.full((2 * m,), 1048575.9375, device="cuda")
    labels = torch.zeros(m + 1, dtype=torch.int32, device="cuda")
    labels[m] = 1
    graph = qm.Graph(row_ptr, torch.cat([leaf, torch.zeros_like(leaf)]), weights=weights)
    q = qm.score(graph, labels, 2)
    Q = Fraction(m - 1, m) - Fraction(2 * m - 1, 2 * m) ** 2 - Fraction(1, 2 * m) ** 2
    assert q["intra_edges_total"] == m - 1
    # (m - 1) / m, (2 m - 1) / (2 m) and its square are rounded once each
    assert abs(q["modularity"] - float(Q)) <= 1e-12 * 2
    graph.close()


# 2^24 nodes: the most whose labels a weighted call gathers as given; 2^21 ids: the
# most that are packed beyond that
@pytest.mark.parametrize("n", [1 << 24, (1 << 24) + 1, 17_500_000])
@pytest.mark.parametrize("K", [200_000, (1 << 21) + 1])
def test_ring_of_blocks(qm, n, K):
    """A ring (u to u +- 1) with blocks of consecutive nodes as communities, ids in
    a scattered order: every W_c^in and W_c^out is a sum of few weights."""
    gen = torch.Generator(device="cuda").manual_seed(K)
    u = torch.arange(n, dtype=torch.int64, device="cuda")
    edge = torch.rand(n, generator=gen, device="cuda") * 4.95 + 0.05  # edge[u]: weight of (u, u + 1)
    block = u * min(K, 150_000) // n
    labels = (block * 7919 % K).to(torch.int32)
    col = torch.stack([(u - 1) % n, (u + 1) % n], 1).int()
    wt = torch.stack([edge.roll(1), edge], 1)
    for row in (0, n - 1):
        col[row], wt[row] = col[row].flip(0), wt[row].flip(0)
    graph = qm.Graph(torch.arange(n + 1, dtype=torch.int64, device="cuda") * 2, col.view(-1), weights=wt.view(-1))
    v = (edge.double() * 2.0 ** 43).long()  # at most 118 edges a block: sums below 2^53
    last = block != block.roll(-1)          # edges between blocks
    B = int(block[-1]) + 1
    w_in = torch.zeros(B, dtype=torch.int64, device="cuda").index_add_(0, block[~last], v[~last])
    w_out = torch.zeros(B, dtype=torch.int64, device="cuda")
    w_out.index_add_(0, block[last], v[last]).index_add_(0, block.roll(-1)[last], v[last])
    W = fixed_sum(edge)
    fin, vol = w_in.double() / float(W), (2 * w_in + w_out).double() / float(2 * W)
    q = qm.score(graph, labels, K)
    assert abs(q["modularity"] - float((fin - vol * vol).sum())) <= 1e-12 * 2
    assert q["cut_edges_total"] == int(last.sum())
    graph.close()
