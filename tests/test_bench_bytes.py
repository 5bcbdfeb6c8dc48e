"""The benchmark's algorithmic bytes of one hull, by the way its points took."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_two_pass_limit_is_the_librarys():
    text = open(os.path.join(ROOT, "paper_2209_12310_gb300", "csrc", "ch_internal.cuh")).read()
    shift = int(re.search(r"kTwoPassMax = 1 << (\d+);", text).group(1))
    assert bench.TWO_PASS_MAX == 1 << shift


def test_dense_data_after_the_extremes_is_read_twice():
    star = {"raw": 5_000, "records": 4_000, "two_pass": 1, "stage": 1, "star_vertices": 3_000}
    small = bench.algorithmic_bytes(1_000_000, star)
    assert small["main_filter"] == 8 * 1_000_000
    assert small["dense_filter"] == 8 * 1_000_000 + 12 * 5_000
    assert small["post"] == 12 * 5_000 + 12 * 4_000 and small["large"] == 12 * 4_000
    large = bench.algorithmic_bytes(100_000_000, star)
    assert "main_filter" not in large and large["dense_filter"] == 8 * 100_000_000 + 12 * 5_000
