"""Which builds take the merge plan by themselves: on either side of the rule's
lines, every result the group plan's."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def reads(n, length):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + length)
    words = torch.randint(-2**31, 2**31, ((n * length + 15) // 16,), generator=g, device="cuda").to(torch.int32)
    if n * length % 16:  # the bits after the last base
        words[-1] &= -1 << (32 - 2 * (n * length % 16))
    return words, torch.full((n,), length, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("n,length,workers,k,merged", [
    (140_000, 50, 3, 3, True), (120_000, 50, 3, 3, False), (140_000, 50, 2, 3, False), (200_000, 50, 2, 3, True),
    (140_000, 50, 3, 1, False), (800_000, 12, 3, 3, True), (150_000, 15, 3, 3, False), (140_000, 330, 3, 3, False)])
def test_merge_plan_in_batches(n, length, workers, k, merged):
    """Builds that run at once take it from fewer reads on; the batch's counters
    include its steps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    words, lens = reads(n, length)
    N = n * (length + 1)
    outs = [(torch.zeros((N + 15) // 16, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int64, device="cuda"),
             torch.zeros(5, dtype=torch.int64, device="cuda")) for _ in range(k)]
    with binding.Context(device=0, batch_workers=workers) as c, \
            binding.Context(device=0, algorithm=binding.Context.ALGO_GROUPS) as sort:
        want = sort.build(words, lens)
        c.build_batch([(words, lens, *o) for o in outs])
        torch.cuda.synchronize()
        assert c.stats()["builds"] == k and c.stats()["merge_launches"] == (k * (length + 1) if merged else 0)
    for o in outs:
        for a, b in zip(o, want[:3]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("n,length,merged", [
    (100_000, 1, False), (1_000_000, 4, False), (1_000_000, 8, False), (4_194_304, 8, True), (50_000, 12, False),
    (1_048_576, 12, True), (100_000, 20, False), (393_215, 20, False), (393_216, 20, True), (150_000, 36, False),
    (262_143, 50, False), (262_144, 50, True), (200_000, 100, False), (262_144, 105, False), (250_000, 150, False),
    (393_216, 150, True), (250_000, 250, False), (250_000, 400, False), (786_432, 200, True)])
def test_merge_plan_by_reads_and_bases(n, length, merged):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    words, lens = reads(n, length)
    with binding.Context(device=0) as c, binding.Context(device=0, algorithm=binding.Context.ALGO_GROUPS) as sort:
        got, want = c.build(words, lens), sort.build(words, lens)
        assert (c.stats()["merge_launches"] > 0) == merged
        assert sort.stats()["merge_launches"] == 0
    for a, b in zip(got[:3], want[:3]):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n,length,share,merged", [
    (100_000, 8, 0.5, False), (10_000, 12, 0.9, False), (262_144, 40, 0.5, False), (262_144, 40, 0.97, True),
    (524_288, 40, 0.6, False), (524_288, 40, 0.9, True), (1_572_864, 40, 0.4, False), (1_572_864, 40, 0.6, True)])
def test_merge_plan_for_parts(n, length, share, merged):
    """Parts of a share of the rows; with the rest, the whole of the group plan's."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    words, lens = reads(n, length)
    N = n * (length + 1)
    with binding.Context(device=0) as c, binding.Context(device=0, algorithm=binding.Context.ALGO_GROUPS) as sort:
        counts = c.bucket_counts(words, lens)
        before = counts.cumsum()
        hi = int((before <= share * N).sum())
        rows = int(before[hi - 1])
        got = torch.zeros((N + 15) // 16 + 1, dtype=torch.int32, device="cuda")
        w, dollar, cnt = c.build_part(words, lens, 0, hi, 0, rows, bucket_counts=counts)
        assert (c.stats()["merge_launches"] > 0) == merged
        got[:w.numel()] |= w
        w, d, k = sort.build_part(words, lens, hi, binding.BUCKETS, rows, N - rows, bucket_counts=counts)
        got[rows // 16:rows // 16 + w.numel()] |= w
        want = sort.build(words, lens)
    assert torch.equal(got[:(N + 15) // 16], want[0])
    none = torch.full_like(d, -1)
    assert torch.equal(torch.where(dollar == none, d, dollar), want[1]) and torch.equal(cnt + k, want[2])


@pytest.mark.parametrize("n,length", [(20_164, 12), (20_166, 12), (65_536, 15), (65_537, 15), (80_000, 13), (70_000, 16),
                                      (17_476, 14), (17_477, 14), (80_000, 17)])
def test_group_plan_depth_by_size(n, length):
    """Either side of the lines between l = 8, 12 and 16, for reads of 12 to 17
    bases: the LSD plan's result, with and without a context."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    words, lens = reads(n, length)
    with binding.Context(device=0) as c, binding.Context(device=0, algorithm=binding.Context.ALGO_LSD) as lsd:
        got, want = c.build(words, lens), lsd.build(words, lens)
        assert c.stats()["merge_launches"] == 0
    out = [torch.zeros_like(t) for t in want[:3]]
    binding.build_noalloc(words, lens.cpu().numpy().view("uint32"), *out)
    torch.cuda.synchronize()
    for a, b, d in zip(got[:3], want[:3], out):
        assert torch.equal(a, b) and torch.equal(d, b)
