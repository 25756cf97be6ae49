"""Parts listed by the listing kernel with the store in L2, their suffix lengths
counted by its counting walk: read lengths around its edges (one base, its two
halves of 128 threads, 256 digit slots, and one past them, which lists by digit
passes), read counts that leave ragged tiles; merged, the oracle's result."""
import numpy as np
import pytest

from gpu_helpers import oracle_of
from paper_1401_7457_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,length", [(5, 1), (4097, 2), (1001, 16), (333, 127), (1, 128), (777, 128), (259, 255), (131, 256)])
@pytest.mark.parametrize("flags", [0, 1 | 8])
def test_parts_listed(n, length, flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = synth.uniform_reads(n, length, n + length)
    ref = oracle_of(codes, lens)
    N = n * (length + 1)
    words = torch.from_numpy(binding.pack_codes(codes).view(np.int32)).cuda()
    d_lens = torch.from_numpy(lens.view(np.int32)).cuda()
    bwt, dollar, counts = np.zeros((N + 15) // 16, dtype=np.uint32), np.full(n, -1, dtype=np.int64).view(np.uint64), 0
    with binding.Context(device=0, plan_flags=flags) as c:
        bounds, rows = binding.split_parts(c.bucket_counts(words, d_lens), 3)
        for p in range(3):
            if bounds[p] == bounds[p + 1]:
                continue
            row0, k = int(rows[p]), int(rows[p + 1] - rows[p])
            w, dpos, cnt = c.build_part(words, d_lens, int(bounds[p]), int(bounds[p + 1]), row0, k)
            if k:
                binding.merge_part(bwt, w.cpu().numpy()[:binding.part_words(row0, k)], row0, k)
            dollar = np.minimum(dollar, dpos.cpu().numpy().view(np.uint64))
            counts = counts + cnt.cpu().numpy()
    assert binding.unpack_ascii(bwt, dollar, N) == ref["bwt"]
    assert np.array_equal(dollar, ref["dollar_pos"]) and np.array_equal(counts.astype(np.uint64), ref["counts"])
