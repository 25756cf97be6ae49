"""A device budget holds as many suffixes in one slice after a build by the merge
plan as before any build."""
import numpy as np
import pytest

from paper_1401_7457_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MERGE = 64


def on_gpu(codes, lens):
    from paper_1401_7457_gb300 import binding
    return torch.from_numpy(binding.pack_codes(codes).view(np.int32)).cuda(), torch.from_numpy(lens.view(np.int32)).cuda()


def test_merge_workspace_is_given_back_to_a_sort():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    merged = on_gpu(*synth.uniform_reads(250, 4000, 1))
    codes, lens = synth.mixed_length_reads(40_000, 20, 100, 3)
    most = []
    for merge_first in (False, True):
        lo, hi = 1_000, 40_000  # reads whose build has one slice, and more than one
        while hi - lo > 10:
            n = (lo + hi) // 2
            with binding.Context(device=0, budget_bytes=32 << 20, plan_flags=MERGE) as c:
                if merge_first:
                    c.build(*merged)
                    assert c.stats()["merge_launches"] == 4001
                c.reset_stats()
                c.build(*on_gpu(codes[:int(lens[:n].sum())], lens[:n]))
                if c.stats()["slices"] == 1:
                    lo = n
                else:
                    hi = n
        assert hi < 40_000
        most.append(lo)
    assert most[1] >= most[0], most
