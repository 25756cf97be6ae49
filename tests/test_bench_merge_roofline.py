"""The benchmark's roofline names the kernel that ran: the merge step for builds
by the merge plan, the carried digit pass for sorted ones."""
import importlib

import pytest


def stats(**kw):
    st = dict.fromkeys(("sort_pass_ms", "group_ms", "emit_ms", "build_ms", "carried_pass_ms", "sort_pass_items", "slices",
                        "carried_pass_items", "carried_pass_launches", "merge_launches", "merge_ms"), 0)
    return {**st, **kw}


def test_roofline_of_merged_and_sorted_builds():
    bench = importlib.import_module("bench")
    n, length, steps = 1_000_000, 100, 5
    bases, N = n * length, n * (length + 1)
    r = bench.roofline_of(stats(merge_launches=101 * steps, merge_ms=2.5 * steps, build_ms=2.5 * steps, slices=steps),
                          steps, n, bases, 4, 6787.2, "measured")
    # L + 1 steps: half the rows on average, 2 bits read and written, and 24 bytes per read
    want = 101 * (0.25 * N + 24 * n)
    assert "k_merge_step" in r["kernel"] and r["launches_per_step"] == 101
    assert r["algorithmic_bytes_per_launch"] == pytest.approx(want / 101)
    assert r["achieved"] == pytest.approx(want / 2.5e-3 / 1e9) and r["frac"] == pytest.approx(r["achieved"] / 6787.2)
    assert r["avg_launch_ms"] == pytest.approx(2.5 / 101)

    r = bench.roofline_of(stats(carried_pass_launches=3 * steps, carried_pass_ms=1.5 * steps, carried_pass_items=3 * N * steps,
                                sort_pass_items=4 * N * steps, sort_pass_ms=2.0 * steps, build_ms=4.0 * steps, slices=steps),
                          steps, n, bases, 4, 6787.2, "measured")
    assert "k_onesweep" in r["kernel"] and r["launches_per_step"] == 3
    assert r["achieved"] == pytest.approx(16 * N / 0.5e-3 / 1e9)
