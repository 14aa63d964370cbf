"""The node count from which untuned calls gather each edge once is stated in the
header and defined in one constant."""
import os
import re

from paper_1507_05492_gb300 import build


def test_the_header_states_the_constant():
    text = open(os.path.join(build.CSRC, "qm_internal.h")).read()
    m = re.search(r"constexpr long long HALF_MIN_NODES = (\d+)LL << (\d+);", text)
    header = open(os.path.join(build.ROOT, "include", "qm.h")).read()
    assert f"QM_REORDER above {m[1]} * 2^{m[2]} nodes" in re.sub(r"\s*\n \*\s*", " ", header)
    assert int(m[1]) << int(m[2]) <= 48_000_000  # gathers of both ends lose there where few edges are cut
