"""bench.py's figures of the clipper are those of the code that runs: flops of
a vertex solve as the source has them, and the kernel a box's cells take."""
import os
import re

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_1707_05333_gb300", "csrc")
COUNTS = {"fp64_plane_tests": 1000, "fp64_vertex_solves": 100, "fp64_fan_terms": 100}


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_flops_of_a_vertex_solve():
    body = source("mm_clip.cuh").split("void solve64(")[1].split("\n}\n")[0]
    flops = 2 * body.count("__fma_rn(") + body.count("__dmul_rn(") + body.count("rcp64(")
    assert bench.FLOPS_SOLVE == flops


def test_kernel_named_is_the_one_that_runs():
    least = int(re.search(r"CELLS_MIN = (\d+);", source("mm_internal.cuh")).group(1))
    assert bench.GROUPED_MIN == least
    for n, filt, kernel in ((least - 1, 1, "k_clip"), (least, 1, "k_cells"), (least, 0, "k_clip")):
        r = bench.clip_roofline(COUNTS, COUNTS, 1.0, n, filt)
        assert r["kernel"] == kernel
        # the filtered clipper's counters are k_clip's
        assert ("executed_fp64_equivalent" in r) == (kernel == "k_clip" and filt == 1)


def test_no_traffic_for_a_box_k_cells_does_not_take(monkeypatch):
    monkeypatch.setitem(bench.CLIP_TRAFFIC, "bytes_per_cell", 900.0)
    monkeypatch.setitem(bench.CLIP_TRAFFIC, "sha256_16", bench.clip_sources_digest())
    assert bench.clip_traffic(bench.GROUPED_MIN, 1) == pytest.approx(900 * bench.GROUPED_MIN)
    assert bench.clip_traffic(bench.GROUPED_MIN - 1, 1) is None


def test_traffic_digest_covers_what_the_clippers_include():
    names = {"mm_cells.cu", "mm_clip.cu"}
    while True:
        more = {inc for n in names for inc in re.findall(r'#include "(mm_\w+\.cuh)"', source(n))} - names
        if not more:
            break
        names |= more
    assert {os.path.basename(f) for f in bench.CLIP_TRAFFIC["sources"]} == names
