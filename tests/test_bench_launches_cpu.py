"""The benchmark's count of launches per step against launch lists of the
profiler (profiles/bench_graph_1m_launches.md: 480 launches in 8 steps; the
other calls 48 without the 8 of the connectivities or 56 with them, and in FP32
15, 43 + 8, 44 + 8 and 46 + 8)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("metric,precision,n,count", [
    ("euclidean", "bf16", 1_000_000, 60),
    ("euclidean", "bf16", 68_579, 56),
    ("cosine", "bf16", 400_009, 56),
    ("euclidean", "fp32", 10_000, 15),
    ("euclidean", "fp32", 24_000, 51),
    ("euclidean", "fp32", 100_003, 52),
    ("euclidean", "fp32", 1_000_000, 54),
])
def test_launches_per_step_agree_with_the_profiler(metric, precision, n, count):
    assert bench.launches_per_step(metric, precision, n) == count
