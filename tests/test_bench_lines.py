"""The bench's k-furthest and range lines from a step's counters: tiles and walks
each by their own arithmetic, phases and pair counts."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

ZERO = dict(point_pairs=0, seed_point_pairs=0, query_blocks=0, ns_seed=0, ns_traverse=0, ns_basecase=0, ns_fallback=0)


@pytest.mark.parametrize("is_range", [False, True])
def test_tiles(is_range):
    st = dict(ZERO, point_pairs=5e12, seed_point_pairs=1e12, query_blocks=100, ns_seed=1e6, ns_traverse=2e6, ns_basecase=1e9,
              ns_fallback=3e6)
    how = bench.kfn_range_line(is_range, 16, st, 152, 1100.0)
    assert how["dtype"] == "bf16" and "BF16" in how["precision"] and how["roofline"]["bound"] == "tensor"
    # the tile launch's own pairs over its own time
    assert how["roofline"]["achieved"] == pytest.approx(2 * 16 * 4e12 / 1e12)
    ph = how["phases_ms"]
    assert sum(ph.values()) == pytest.approx(1100.0)
    assert sorted(v for k, v in ph.items() if k != "build_and_rest") == pytest.approx([1.0, 2.0, 3.0, 1000.0])


@pytest.mark.parametrize("is_range,kernel", [(False, "k_kfn"), (True, "k_range")])
def test_walks(is_range, kernel):
    how = bench.kfn_range_line(is_range, 3, dict(ZERO, point_pairs=1e12, ns_basecase=2e9), 152, 2500.0)
    assert how["dtype"] == "f32" and "fp32" in how["precision"]
    assert how["roofline"]["bound"] == "alu" and how["roofline"]["kernel"].startswith(kernel)
    assert how["roofline"]["achieved"] == pytest.approx(3 * 3 * 1e12 / 2e12)
    assert sum(how["phases_ms"].values()) == pytest.approx(2500.0)
