"""Interval bounds of a network whose weights are streamed: the last wave's smaller tiles give the bits of the full ones.

A batch is cut into whole waves of 32-row tiles and one wave of tiles with fewer rows (4, 8, .. 32, by what is left),
whose layers run with other thread tiles; each output is one thread's chain of directed roundings over the inputs in
order, whatever the tile, so that a box's bounds are equal bits in any batch.
"""
import numpy as np
import pytest
import torch

from paper_2412_09584_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# widths above 128 (1, 2 or 4 rows a thread), between 32 and 128 (1 or 2) and at most 32, odd ones among them
S, K, HIDDEN, H = 20, 3, [256, 250, 100, 64, 30], 2


@pytest.mark.parametrize("rows", [1, 5, 9, 16, 17, 24, 31, 33])
def test_rows_left_for_the_last_wave(gp, rows):
    p = W.make_problem(S, K, HIDDEN, H, 0.01, seed=4, weight_scale=0.5)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lo, hi, _ = W.random_boxes(K * H, 34 * sms + 1, seed=5, min_width=0.0, max_width=0.8)
    g = gp(p)
    full, n = g.ibp(lo, hi), rows * sms - 3
    for a, b in zip(full, g.ibp(lo[:n], hi[:n])):
        assert np.array_equal(a[:n], b)
