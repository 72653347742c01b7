"""Lattices in the grouped clipper: whole runs of candidates at one distance,
equal bit for bit or up to rounding, settled by rank within a run (a batch of
up to 32 candidates, and of up to 64); the mesh is the warp-per-cell
clipper's bit for bit."""
import numpy as np
import pytest

from paper_1707_05333_gb300 import binding
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c, torch = H.gpu_context()
    yield c, torch
    c.close()


def lattice(kind, m, jitter=0.0):
    k = np.arange(m)
    g = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3).astype(float)
    if kind == "bcc":
        g = np.concatenate([g, g + 0.5])
    elif kind == "fcc":
        g = np.concatenate([g, g + [0.5, 0.5, 0.0], g + [0.5, 0.0, 0.5], g + [0.0, 0.5, 0.5]])
    g += 0.25 + jitter * np.random.default_rng(1712).normal(size=g.shape)
    return g / m


@pytest.mark.parametrize("cand_cap", [32, 64])
@pytest.mark.parametrize("kind,m,jitter", [("cubic", 16, 0.0), ("cubic", 17, 0.0), ("bcc", 13, 0.0), ("bcc", 16, 0.0),
                                           ("fcc", 11, 0.0), ("fcc", 16, 0.0), ("cubic", 17, 1e-5), ("bcc", 13, 1e-7),
                                           ("cubic", 17, 1e-12)])
def test_same_mesh_as_the_warp_per_cell_clipper(ctx, kind, m, jitter, cand_cap):
    c, torch = ctx
    pos = lattice(kind, m, jitter)
    assert len(pos) >= 4096
    out = []
    for counted in (1, 0):
        c.set_config(collect_stats=counted, cand_cap=cand_cap)
        try:
            out.append(H.gpu_tessellate(c, torch, pos, np.ones(3))[2])
        except binding.MMError as e:  # lattices jittered by 1e-13..1e-10 can be refused as near-degenerate: by both
            out.append({"refused": e.status})
        finally:
            c.set_config(collect_stats=0, cand_cap=64)
    assert out[0].keys() == out[1].keys()
    for k in out[0]:
        np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=k)
