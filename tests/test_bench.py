"""bench.py's account of the work of a build: by the cells it put out, not by
the events of another kernel."""
import inspect
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_needed_flops_of_known_cells():
    # a truncated octahedron: 14 faces, 24 vertices, 72 directed face edges
    one = 24 * 51 + 14 * 24 * 6 + 14 * 30 + 72 * 60
    assert bench.needed_flops([14]) == one
    # empty cells cost nothing; fewer site faces than a polytope has count as four
    assert bench.needed_flops([14, 0, 14]) == 2 * one
    assert bench.needed_flops([1]) == bench.needed_flops([4]) == 4 * 51 + 16 * 6 + 4 * 30 + 12 * 60
    assert bench.needed_flops(np.full(1000, 14, np.int32)) == 1000 * one
    assert bench.needed_flops([]) == 0


def test_achieved_rate_reads_no_event_counter():
    """The event counters come from a build with counters = 1, whose cells
    another kernel makes than the one that is timed."""
    src = inspect.getsource(bench.run_ours)
    used = [line for line in src.splitlines() if "flop" in line or "achieved" in line]
    assert used and not any("cnt[" in line for line in used)


def test_plain_fp32_form_has_its_own_knobs():
    """Those that the tuner leaves alone in the default modes are read by the
    kernel of plain FP32."""
    tuned = {"leaf_size": 16, "warm_start": 0, "warps_per_block": 2, "precision": 0, "timing": 1}
    cfg = bench.plain_fp32_config(tuned, "")
    assert cfg == {"leaf_size": 32, "warm_start": 2, "warps_per_block": 2, "precision": 1, "timing": 0}
    assert bench.plain_fp32_config(tuned, '{"leaf_size": 8}')["leaf_size"] == 8
    assert "plain_fp32_config(cfg" in inspect.getsource(bench.run_ours)
