"""The largest comparison the library takes, 2^31 - 1 nodes: the walk over the last
bucket's nodes steps past 2^31.  Both labellings are blocks of consecutive nodes,
so the counts have closed forms."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_most_nodes():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1507_05492_gb300 import qm
    n = (1 << 31) - 1
    if torch.cuda.get_device_properties(0).total_memory < 120 * (1 << 30):
        pytest.skip("needs 75 GB of device memory")
    found = torch.arange(n, dtype=torch.int32, device="cuda")
    truth = found >> 19
    found >>= 20
    c = qm.compare(truth, found, 4096, 2048)

    def pairs(block):
        full, rest = divmod(n, block)
        return full * (block * (block - 1) // 2) + rest * (rest - 1) // 2

    sa, sb = pairs(1 << 19), pairs(1 << 20)
    assert (c["n_nodes"], c["k_truth"], c["k_found"], c["n_cells"]) == (n, 4096, 2048, 4096)
    assert (c["a11"], c["a10"], c["a01"]) == (sa, 0, sb - sa)  # truth refines found
    assert c["a00"] == n * (n - 1) // 2 - sb
    # every truth community lies in one found community; of each found one the larger half counts
    assert c["nvd_sum"] == n + 2048 * (1 << 19)
    del truth, found
    torch.cuda.empty_cache()
    qm.release_cache()
