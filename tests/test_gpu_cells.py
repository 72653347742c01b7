"""The grouped clipper (several cells to a warp, 4096 cells and more) against
the warp-per-cell filtered clipper, which runs when the work counters are on:
the same mesh, bit for bit.  (The direct FP64 clipper forms its search limit in
FP64 and may meet candidates in other batches, which orders a cell's faces
differently; that pair is compared where the batches agree.)"""
import numpy as np
import pytest

from paper_1707_05333_gb300 import workloads as WL
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c, torch = H.gpu_context()
    yield c, torch
    c.close()


def bcc(m):
    s = 1.0 / m
    k = np.arange(m)
    g = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    return (np.concatenate([g, g + 0.5]) + 0.25) * s


def sheet(n):
    """A dense plane in a sparse box: cells of very different shapes, many
    faces, long searches, bins of very different counts."""
    p = WL.random_points(n, seed=31)
    q = p[: n // 3].copy()
    q[:, 2] = 0.5 + 0.002 * (q[:, 2] - 0.5)
    return np.concatenate([q, p[n // 3:]])


CASES = {
    # the rule's edge, and counts that fill the warps of four and of eight cells unevenly
    "random_4095": lambda: (WL.random_points(4095, seed=33), np.ones(3)),
    "random_4096": lambda: (WL.random_points(4096, seed=34), np.ones(3)),
    "random_4099": lambda: (WL.random_points(4099, seed=35), np.ones(3)),
    "random_7999": lambda: (WL.random_points(7999, seed=21), np.ones(3)),
    "random_8000": lambda: (WL.random_points(8000, seed=22), np.ones(3)),
    "random_8003": lambda: (WL.random_points(8003, seed=23), np.ones(3)),
    "random_20011": lambda: (WL.random_points(20011, seed=24), np.ones(3)),
    "jittered_21^3": lambda: (WL.smooth_wave(21).pos, np.ones(3)),
    # exact ties of the sort keys and of the plane tests
    "bcc_16": lambda: (bcc(16), np.ones(3)),
    # crowded bins and cells past the lists: handed to the warp-per-cell clipper
    "clustered_9000": lambda: (WL.clustered_points(9000, seed=25), np.ones(3)),
    "sheet_9000": lambda: (sheet(9000), np.ones(3)),
    # few bins across: images on every side
    "slab": lambda: (WL.random_points(9000, box=(4.0, 4.0, 0.1), seed=26), np.array([4.0, 4.0, 0.1])),
    "rod": lambda: (WL.random_points(8200, box=(30.0, 0.3, 0.3), seed=27), np.array([30.0, 0.3, 0.3])),
    # the ends of the box sizes
    "tiny_box": lambda: (WL.random_points(8100, box=(2.0**-38,) * 3, seed=28), np.full(3, 2.0**-38)),
    "huge_box": lambda: (WL.random_points(8100, box=(2.0**38,) * 3, seed=29), np.full(3, 2.0**38)),
}


@pytest.mark.parametrize("case", list(CASES))
def test_same_mesh_as_the_warp_per_cell_clipper(ctx, case):
    c, torch = ctx
    pos, box = CASES[case]()
    c.set_config(collect_stats=1)
    try:
        _, _, A = H.gpu_tessellate(c, torch, pos, box)
    finally:
        c.set_config(collect_stats=0)
    _, _, B = H.gpu_tessellate(c, torch, pos, box)
    for k in A:
        np.testing.assert_array_equal(A[k], B[k], err_msg=k)


@pytest.mark.parametrize("cand_cap", [32, 48])
def test_candidate_buffer_sizes(ctx, cand_cap):
    c, torch = ctx
    pos = WL.random_points(8009, seed=30)
    out = []
    for counted in (1, 0):
        c.set_config(collect_stats=counted, cand_cap=cand_cap)
        try:
            out.append(H.gpu_tessellate(c, torch, pos, np.ones(3))[2])
        finally:
            c.set_config(collect_stats=0, cand_cap=64)
    for k in out[0]:
        np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=k)


def test_coincident_generators_are_refused(ctx):
    c, torch = ctx
    from paper_1707_05333_gb300 import binding as BD
    pos = WL.random_points(8500, seed=32)
    pos[4321] = pos[17]
    with pytest.raises(BD.MMError, match="two generators at one position"):
        H.gpu_tessellate(c, torch, pos, np.ones(3))
