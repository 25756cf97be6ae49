"""Edges of bucket-range parts: ranges that hold no suffix."""
import numpy as np
import pytest

from paper_1401_7457_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def device(a):
    return torch.from_numpy(a.view(np.int32)).cuda()


@pytest.mark.parametrize("given", [True, False])
@pytest.mark.parametrize("where", ["device", "host"])
@pytest.mark.parametrize("length", [1, 10, 20, 100, 300])
def test_empty_part(length, where, given):
    """A range without suffixes whose first row is inside a word: that word is
    written as 0, the counts as 0 and every $ row as ~0, whatever the buffers
    (the caller's and the context's) held before; no plan runs for it."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = synth.uniform_reads(1001, length, length)
    words = binding.pack_codes(codes)
    if where == "device":
        words, lens = device(words), device(lens)
    with binding.Context(device=0) as c:
        c.build(words, lens)
        counts = c.bucket_counts(words, lens)
        before = np.concatenate([[0], np.cumsum(counts.astype(np.int64))])
        lo = int(np.nonzero((counts == 0) & (before[:-1] % 16 != 0))[0][0])
        row0 = int(before[lo])
        out = np.full(1, 0xFFFFFFFF, dtype=np.uint32), np.full(1001, 7, dtype=np.uint64), np.full(5, 7, dtype=np.uint64)
        if where == "device":
            out = device(out[0]), torch.full((1001,), 7, device="cuda"), torch.full((5,), 7, device="cuda")
        c.reset_stats()
        c.build_part(words, lens, lo, lo + 1, row0, 0, *out, bucket_counts=counts if given else None)
        if where == "device":
            out = [t.cpu().numpy() for t in out]
        assert int(out[0][0]) == 0
        assert (out[1].view(np.uint64) == np.uint64(0xFFFFFFFFFFFFFFFF)).all() and not out[2].any()
        assert c.stats()["merge_launches"] == 0 and c.stats()["sort_pass_launches"] == 0


@pytest.mark.parametrize("flags", [0, 64])
def test_empty_part_counts_as_no_slice(flags):
    """Nothing is sorted or merged for an empty part: its time is no plan's."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = synth.uniform_reads(1001, 50, 3)
    words, lens = device(binding.pack_codes(codes)), device(lens)
    with binding.Context(device=0, plan_flags=flags, timing=True) as c:
        counts = c.bucket_counts(words, lens)
        lo = int(np.nonzero(counts == 0)[0][0])
        c.reset_stats()
        c.build_part(words, lens, lo, lo + 1, int(counts[:lo].sum()), 0, bucket_counts=counts)
        st = c.stats()
        assert st["builds"] == 1 and st["slices"] == 0 and st["build_ms"] > 0
        assert st["merge_ms"] == 0 and st["merge_launches"] == 0


@pytest.mark.parametrize("flags", [0, 1, 64])
def test_counts_that_wrap_are_rejected(flags):
    """Counts that sum to N only modulo 2^64 (a part whose rows would start
    before or end after B_R): EINVAL, by the host, whatever the plan."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    codes, lens = synth.uniform_reads(3000, 12, 3)
    words, lens = device(binding.pack_codes(codes)), device(lens)
    N = 3000 * 13
    with binding.Context(device=0, plan_flags=flags) as c:
        for first, lo, row0, rows in ((2**64 - 1600, 1, 2**64 - 1600, 1600), (2**64 - 1600, 0, 0, 2**64 - 1600)):
            counts = np.zeros(binding.BUCKETS, dtype=np.uint64)
            counts[0], counts[1], counts[2] = first, 1600, N
            out = torch.zeros(N, dtype=torch.int32, device="cuda")
            with pytest.raises((binding.CxbwtError, ValueError)) as e:
                c.build_part(words, lens, lo, lo + 1, row0, rows, out, bucket_counts=counts)
            assert isinstance(e.value, ValueError) or e.value.status == -1
        assert c.stats()["builds"] == 0
        ok = c.bucket_counts(words, lens)
        c.build_part(words, lens, 0, binding.BUCKETS, 0, N, bucket_counts=ok)


@pytest.mark.parametrize("length,flags", [(12, 64), (100, 64), (127, 64), (128, 65), (255, 64), (256, 64), (300, 64), (528, 64)])
def test_counts_of_other_reads_are_noticed_by_the_merge_plan(length, flags):
    """Counts of other reads with the same sum, over a range that holds more or
    fewer suffixes than they say: an error, as when the part is sorted; the
    right counts of the same ranges are taken."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    n = 3000 * 100 // (length + 1) + 31
    a, la = synth.uniform_reads(n, length, 1)
    b, _ = synth.uniform_reads(n, length, 2)
    lens, a, b = device(la), device(binding.pack_codes(a)), device(binding.pack_codes(b))
    with binding.Context(device=0, plan_flags=flags) as c:
        of_a, of_b = c.bucket_counts(a, lens), c.bucket_counts(b, lens)
        diff = np.cumsum(of_a.astype(np.int64) - of_b.astype(np.int64))
        for hi in (int(np.argmax(diff[:-1])) + 1, int(np.argmin(diff[:-1])) + 1):
            assert diff[hi - 1] != 0
            for lo, h in ((0, hi), (hi, binding.BUCKETS)):
                before = c.stats()["merge_launches"]
                with pytest.raises(binding.CxbwtError) as e:
                    c.build_part(a, lens, lo, h, int(of_b[:lo].sum()), int(of_b[lo:h].sum()), bucket_counts=of_b)
                assert e.value.status == -7
                c.build_part(a, lens, lo, h, int(of_a[:lo].sum()), int(of_a[lo:h].sum()), bucket_counts=of_a)
                assert c.stats()["merge_launches"] > before
