"""bench.py's bytes per site update name the kernels that a job runs."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("algo,polish,bulk_bytes,polish_bytes", [
    ("or", "same", 8 * 48 + 3 * 48, 112 + 384 + 48 + 192),      # links as loaded; K0 in 28 reals
    ("sr", "same", 16 * 48 + 2 * 48, 144 + 384 + 48 + 192),     # links rewritten; K0 in pairs
    ("sr", "or", 16 * 48 + 2 * 48, 112 + 384 + 48 + 192),       # rewritten, then the overrelaxed polish
])
def test_bytes_of_the_kernels_a_job_runs(algo, polish, bulk_bytes, polish_bytes):
    sys.path.insert(0, ROOT)
    import bench
    bulk, after = bench.ladder_kinds(algo, polish)
    assert bench.algorithmic_bytes_per_site(bulk) == bulk_bytes
    assert bench.algorithmic_bytes_per_site(after) == polish_bytes
