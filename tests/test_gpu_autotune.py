"""The autotuner times the warp-per-cell clipper's settings only where that
clipper has a share of the cells; elsewhere they stay as the caller set them."""
import numpy as np
import pytest

from paper_1707_05333_gb300 import workloads as WL
from tests import helpers as H

pytestmark = pytest.mark.gpu

CASES = {
    "small box: all cells": (lambda: WL.random_points(1000, seed=41), True),
    "grouped clipper, hardly any": (lambda: WL.random_points(9000, seed=42), False),
    "grouped clipper, crowded bins": (lambda: WL.clustered_points(9000, seed=43), True),
}


@pytest.mark.parametrize("case", list(CASES))
def test_warp_per_cell_settings(case):
    make, tuned = CASES[case]
    c, torch = H.gpu_context(clip_warps=5, clip_sort=1)
    best = c.mm_autotune(H.to_dev(torch, make().T), np.ones(3), reps=1)
    assert best["cand_cap"] in (32, 64) and best["bin_scale"] in (0.8, 1.0, 1.25, 1.5) and best["tessellate_ms"] > 0
    if tuned:
        assert best["clip_warps"] in (2, 4, 8)
    else:
        assert best["clip_warps"] == 5 and best["clip_sort"] == 1
    c.close()
