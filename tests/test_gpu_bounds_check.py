"""The diagnostic build (-DQM_BOUNDS_CHECK): an entry of a packed run whose label
fails its check is recorded and takes no part in the count, in the full steps of
a run as well as in its last one."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def checked(tmp_path_factory):
    from paper_1507_05492_gb300 import build
    out = str(tmp_path_factory.mktemp("checked") / "libchecked.so")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([build.nvcc(), *build.FLAGS, "-DQM_BOUNDS_CHECK", "-shared", "-I", build.CSRC, "-I",
                    os.path.join(build.ROOT, "include"), os.path.join(here, "checked_run.cu"), "-o", out], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("mode", [1, 2])  # labels above the community's only; all labels, with its own penalty
@pytest.mark.parametrize("at", [0, 37, 199])
@pytest.mark.parametrize("bad", [-7, 50, 1 << 30])
def test_bad_label_is_left_out(checked, mode, at, bad):
    K, m = 50, 200
    rng = np.random.default_rng(at)
    labels = rng.integers(1, K, m).astype(np.int32)
    good = np.delete(labels, at)
    labels[at] = bad
    dev = torch.from_numpy(labels).cuda()
    recip = torch.ones(2 * K, dtype=torch.int64, device="cuda")
    inter = torch.zeros(K, dtype=torch.int32, device="cuda")
    rec = torch.zeros(8 * K, dtype=torch.int64, device="cuda")
    dbg = (ctypes.c_ulonglong * 8)()
    torch.cuda.synchronize()
    vp = ctypes.c_void_p
    rc = checked.checked_run(mode, vp(dev.data_ptr()), m, K, vp(recip.data_ptr()), vp(inter.data_ptr()),
                             vp(rec.data_ptr()), dbg)
    assert rc == 0
    assert list(dbg)[:4] == [6, bad % (1 << 64), K, 1]  # site, index, bound, failures
    counts = np.bincount(good, minlength=K)
    words = rec.view(K, 8)[0].cpu().numpy()
    assert words[2] == (counts > 0).sum() and words[3] == (counts * counts).sum()  # keys, squares of their counts
