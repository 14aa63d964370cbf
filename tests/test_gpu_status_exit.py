"""Kernels that may set the status word they read at their start: a block that
starts while earlier blocks set it must leave whole, or not at all.  Comparisons
whose truth labels are bad in every tile run beside other comparisons and
scoring calls that keep the SMs busy, so that their blocks start at different
times; every bad call must be refused, every good one give the result it gives
alone.  Likewise expired staging waits, which the blocks of a counting kernel
report while others start."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm as q
    return q


def test_refused_comparisons_beside_others(qm):
    n, K = (1 << 23) + 77, 20_000
    gen = torch.Generator(device="cuda").manual_seed(5)
    truth = torch.randint(0, K, (n,), generator=gen, device="cuda", dtype=torch.int32)
    found = torch.where(torch.rand(n, generator=gen, device="cuda") < 0.3,
                        torch.randint(0, K, (n,), generator=gen, device="cuda", dtype=torch.int32), truth)
    bad = truth.clone()
    bad[::40_000] = K
    torch.cuda.synchronize()
    want = qm.compare(truth, found, K, K)
    errors = []

    def work(t, refused):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(8):
                    if not refused:
                        assert qm.compare(truth, found, K, K) == want
                        continue
                    with pytest.raises(qm.QmError) as e:
                        qm.compare(bad, found, K, K)
                    assert e.value.status == qm.QM_EINVAL
        except BaseException as e:  # noqa: BLE001 - reported by the test
            errors.append((t, e))

    threads = [threading.Thread(target=work, args=(t, t % 2 == 0)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert qm.compare(truth, found, K, K) == want


def test_expired_waits_repeated(qm):
    from paper_1507_05492_gb300 import gen
    g = gen.lfr_graph(gen.LfrParams(n=400_000, k_max=100, s_min=500, s_max=3000, mu=0.5, seed=3), device="cuda")
    graph = qm.Graph(g.row_ptr, g.col, reorder=True)
    want = qm.score(graph, g.labels, g.K, per_community=True)
    try:
        qm.debug_set_stage_wait(0)
        for _ in range(30):
            with pytest.raises(qm.QmError) as e:
                qm.score(graph, g.labels, g.K, per_community=True)
            assert e.value.status == qm.QM_ETIMEOUT
    finally:
        qm.debug_set_stage_wait(-1)
    got = qm.score(graph, g.labels, g.K, per_community=True)
    per_got, per_want = got.pop("per_community"), want.pop("per_community")
    assert got == want
    for k, v in per_want.items():
        assert torch.equal(per_got[k], v), k
    graph.close()
