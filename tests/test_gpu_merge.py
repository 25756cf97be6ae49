"""The merge plan (one suffix length per step) against the oracle: read lengths
around its 16-base refills, read counts around the edges of its parts, tiles
and groups of tiles, all three tile sizes, 32- and 64-bit rows, reads whose
suffixes fall into one class or tie throughout, parts of a build, and the
switch from the group plan by size."""
import numpy as np
import pytest

from gpu_helpers import assert_same, gpu_bwt, oracle_of
from paper_1401_7457_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MERGE, ID64 = 64, 1


def reads(kind, n, length):
    rng = np.random.default_rng(n * 1000 + length)
    if kind == "random":
        return synth.uniform_reads(n, length, n + length)
    if kind == "genome":
        g = synth.random_genome(max(2 * length, n * length // 30), n + length)
        return synth.sample_reads(g, n, length, n + length + 1, 0.01)
    if kind == "same":
        one = rng.integers(0, 4, size=length).astype(np.uint8)
        return np.tile(one, n), np.full(n, length, dtype=np.uint32)
    return np.full(n * length, "ACGT".index(kind), dtype=np.uint8), np.full(n, length, dtype=np.uint32)


CASES = [("random", 1, 1), ("random", 1, 4096), ("random", 3, 15), ("random", 31, 16), ("random", 33, 17),
         ("genome", 257, 33), ("random", 5000, 1), ("random", 8191, 7), ("random", 8192, 31), ("random", 8193, 2),
         ("genome", 3000, 400), ("genome", 1200, 600), ("same", 2000, 50), ("A", 3000, 40), ("T", 1025, 64),
         ("genome", 20_000, 150), ("genome", 70_000, 100), ("random", 400_000, 20)]


@pytest.mark.parametrize("flags", [MERGE, MERGE | ID64])
@pytest.mark.parametrize("kind,n,length", CASES)
def test_merge_plan(kind, n, length, flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = reads(kind, n, length)
    with binding.Context(device=0, plan_flags=flags) as c:
        got = gpu_bwt(c, codes, lens, where="host" if n % 2 else "device")
        assert c.stats()["merge_launches"] == length + 1
    assert_same(got, oracle_of(codes, lens))


def test_merge_plan_after_other_sizes():
    """One context, builds of sizes up and down (the workspace of a larger
    build is reused), a sort between them: each is the oracle's."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    with binding.Context(device=0, plan_flags=MERGE) as c:
        for kind, n, length, sa in [("genome", 30_000, 100, False), ("random", 100, 33, False),
                                    ("genome", 5_000, 76, True), ("random", 9_000, 250, False),
                                    ("genome", 30_000, 100, False)]:
            codes, lens = reads(kind, n, length)
            before = c.stats()["merge_launches"]
            got = gpu_bwt(c, codes, lens, want_sa=sa)
            assert (c.stats()["merge_launches"] > before) == (not sa)
            assert_same(got, oracle_of(codes, lens), sa=sa)


@pytest.mark.parametrize("kind,n,length", [("genome", 9_000, 100), ("random", 20_001, 35), ("A", 2_000, 20)])
def test_merge_plan_parts(kind, n, length):
    """Parts built by the merge plan (their rows, $ rows and counts alone)
    merge to the oracle's result."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = reads(kind, n, length)
    ref = oracle_of(codes, lens)
    N = n * (length + 1)
    words = torch.from_numpy(binding.pack_codes(codes).view(np.int32)).cuda()
    d_lens = torch.from_numpy(lens.view(np.int32)).cuda()
    bwt, dollar, counts = np.zeros((N + 15) // 16, dtype=np.uint32), np.full(n, -1, dtype=np.int64).view(np.uint64), 0
    with binding.Context(device=0, plan_flags=MERGE) as c:
        bounds, rows = binding.split_parts(c.bucket_counts(words, d_lens), 5)
        for p in range(5):
            if bounds[p] == bounds[p + 1]:
                continue
            row0, k = int(rows[p]), int(rows[p + 1] - rows[p])
            w, dpos, cnt = c.build_part(words, d_lens, int(bounds[p]), int(bounds[p + 1]), row0, k)
            if k:
                binding.merge_part(bwt, w.cpu().numpy()[:binding.part_words(row0, k)], row0, k)
            dollar = np.minimum(dollar, dpos.cpu().numpy().view(np.uint64))
            counts = counts + cnt.cpu().numpy()
        assert c.stats()["merge_launches"] > 0
    assert binding.unpack_ascii(bwt, dollar, N) == ref["bwt"]
    assert np.array_equal(dollar, ref["dollar_pos"]) and np.array_equal(counts.astype(np.uint64), ref["counts"])


@pytest.mark.parametrize("n,length,merged", [(20_000, 100, False), (300_000, 36, True), (3_000, 700, False), (20_000, 700, True)])
def test_merge_plan_is_taken_by_size(n, length, merged):
    """The automatic plan: the oracle's result on either side of the rule."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = reads("genome", n, length)
    with binding.Context(device=0) as c:
        got = gpu_bwt(c, codes, lens)
        assert (c.stats()["merge_launches"] > 0) == merged
    assert_same(got, oracle_of(codes, lens))
