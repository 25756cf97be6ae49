"""Group finish by one warp: groups of every size around the edges of its
windows of 32 rows (odd and even ones: with keys of 10 and more words each pair
is compared once), larger ones, ties throughout, and the key widths of reads of
20 to 520 bases: the oracle's whole suffix order."""
import numpy as np
import pytest

from gpu_helpers import assert_same, gpu_bwt, oracle_of

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SIZES = [1, 2, 3, 4, 5, 16, 17, 31, 32, 33, 34, 63, 64, 65]


def grouped(length, seed, copies):
    """Reads that share their first 16 bases with `size` others and differ in
    one later base each (or, `copies`, in none)."""
    rng = np.random.default_rng(seed)
    rows = []
    for size in SIZES:
        head = rng.integers(0, 4, size=length)
        for _ in range(size):
            r = head.copy()
            if not copies and length > 16:
                r[rng.integers(16, length)] = rng.integers(0, 4)
            rows.append(r)
    rows = np.array(rows, dtype=np.uint8)[rng.permutation(len(rows))]
    return rows.reshape(-1), np.full(rows.shape[0], length, dtype=np.uint32)


@pytest.mark.parametrize("copies", [False, True])
@pytest.mark.parametrize("length", [20, 60, 100, 130, 170, 200, 260, 330, 390, 520])
def test_group_windows(length, copies):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = grouped(length, length, copies)
    with binding.Context(device=0, algorithm=binding.Context.ALGO_GROUPS) as c:
        got = gpu_bwt(c, codes, lens, want_sa=True)
    assert_same(got, oracle_of(codes, lens), sa=True)
