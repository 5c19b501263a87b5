"""Bytes of a captured run of steps: what the first seven of eight steps leave out."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("steps,before,contrast,want", [
    (1, 0, True, 344.0), (7, 0, True, 344.0), (8, 0, True, 340.5), (8, 1, True, 344.0), (17, 3, True, 344 - 4 * 14 / 17),
    (20, 4, True, 344 - 4 * 14 / 20), (3000, 3, True, 344 - 4 * 7 * 374 / 3000), (8, 2, False, 332 - 16 * 7 / 8)])
def test_run_bytes_per_fluid_node(steps, before, contrast, want):
    """D3Q19 FP32: a step by itself moves 344 B per fluid node (332 without a
    contrast); seven of each eight captured steps leave out p (4 B), and u (12 B)
    without a contrast.  8 steps from an odd one: 1 alone, then 7 alone."""
    assert bench.run_bytes_per_fluid_node(344.0 if contrast else 332.0, steps, before, 3, 4, contrast) == pytest.approx(want)
