"""The merge plan above 2.1 billion rows, where a tile's counts are summed over
more groups of tiles than a CTA has threads: the group plan's result."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_merge_plan_above_two_billion_rows():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_7457_gb300 import binding
    n, length = 22_000_000, 100  # 2.222G rows: 265 groups of 256 tiles of 32,768 rows
    N = n * (length + 1)
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    words = torch.randint(-2**31, 2**31, (n * length // 16,), generator=g, device="cuda").to(torch.int32)
    lens = torch.full((n,), length, dtype=torch.int32, device="cuda")
    outs = []
    for algorithm in (0, binding.Context.ALGO_GROUPS):
        out = (torch.zeros((N + 15) // 16, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int64, device="cuda"),
               torch.zeros(5, dtype=torch.int64, device="cuda"))
        with binding.Context(device=0, algorithm=algorithm, budget_bytes=60 << 30) as c:
            c.build(words, lens, *out)
            assert c.stats()["merge_launches"] == (0 if algorithm else length + 1)
        outs.append(out)
    for a, b in zip(*outs):
        assert torch.equal(a, b)
