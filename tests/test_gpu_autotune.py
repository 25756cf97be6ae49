"""Builds of a tuned context are built as the tuner reports, and tuning is no loss
against an untuned context."""
import numpy as np
import pytest

from gpu_helpers import assert_same, gpu_bwt, oracle_of
from paper_1401_7457_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def on_gpu(codes, lens):
    from paper_1401_7457_gb300 import binding
    return torch.from_numpy(binding.pack_codes(codes).view(np.int32)).cuda(), torch.from_numpy(lens.view(np.int32)).cuda()


def outputs(n, suffixes):
    return (torch.zeros((suffixes + 15) // 16, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int64, device="cuda"),
            torch.zeros(5, dtype=torch.int64, device="cuda"))


@pytest.mark.parametrize("n,length", [(1_500, 100), (4_000, 100), (12_000, 20), (200_000, 30), (300_000, 36), (20_000, 600)])
def test_a_tuned_build_is_the_reported_one(n, length):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    words, lens = on_gpu(*synth.uniform_reads(n, length, 5))
    out, want = outputs(n, n * (length + 1)), outputs(n, n * (length + 1))
    with binding.Context(device=0) as c, binding.Context(device=0, algorithm=binding.Context.ALGO_LSD) as lsd:
        t = c.autotune(words, lens, out[0], out[1])
        c.reset_stats()
        c.build(words, lens, *out)
        lsd.build(words, lens, *want)
        torch.cuda.synchronize()
        st = c.stats()
    if t["algorithm"] == binding.Context.ALGO_MERGE:
        assert st["merge_launches"] == length + 1 and st["sort_pass_launches"] == 0
        assert t["tile_items"] == 0 and t["prefix_len"] == 0
    else:
        assert st["merge_launches"] == 0
        digits = (length + 3) // 4
        if t["algorithm"] == binding.Context.ALGO_GROUPS:
            digits = min(digits, t["prefix_len"] // 4)
        assert st["sort_pass_launches"] == digits
    assert all(torch.equal(a, b) for a, b in zip(out, want))


def test_tuning_small_builds_is_no_loss():
    """Times of 60 builds: a tuned context is at most a fifth slower than an
    untuned one (it was a third, with neither the small tiles nor l = 8 tried)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    words, lens = on_gpu(*synth.uniform_reads(1_500, 100, 7))
    out = outputs(1_500, 1_500 * 101)
    stream = torch.cuda.current_stream()

    def best(c):
        ms = []
        for _ in range(60):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            c.build(words, lens, *out, stream=stream)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms)

    with binding.Context(device=0) as c, binding.Context(device=0) as untuned:
        c.autotune(words, lens, out[0], out[1])
        assert best(c) <= 1.2 * best(untuned)


def test_other_builds_of_a_tuned_class():
    """The suffix list and parts of classes tuned to any plan."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    for n, length in ((1_500, 100), (120_000, 20), (300_000, 20)):
        codes, lens = synth.uniform_reads(n, length, 9)
        words, dl = on_gpu(codes, lens)
        N = n * (length + 1)
        ref = oracle_of(codes, lens)
        with binding.Context(device=0) as c:
            out = outputs(n, N)
            c.autotune(words, dl, out[0], out[1])
            assert_same(gpu_bwt(c, codes, lens, want_sa=True), ref, sa=True)
            counts = c.bucket_counts(words, dl)
            bounds, rows = binding.split_parts(counts, 2)
            bwt, got = np.zeros((N + 15) // 16, dtype=np.uint32), 0
            for p in range(2):
                w, _, cnt = c.build_part(words, dl, int(bounds[p]), int(bounds[p + 1]), int(rows[p]), int(rows[p + 1] - rows[p]),
                                         bucket_counts=counts)
                binding.merge_part(bwt, w.cpu().numpy(), int(rows[p]), int(rows[p + 1] - rows[p]))
                got = got + cnt.cpu().numpy()
            assert binding.unpack_ascii(bwt, ref["dollar_pos"], N) == ref["bwt"] and np.array_equal(got, ref["counts"].astype(np.int64))
