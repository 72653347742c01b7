"""Which clipper a tessellation takes, and what only the grouped one has: its
list of cells left to the warp-per-cell clipper, a warp's second geometry
pass, boxes that share a warp, bins of every width."""
import numpy as np
import pytest

from paper_1707_05333_gb300 import workloads as WL
from tests import helpers as H

pytestmark = pytest.mark.gpu

PLANES, VERTICES, PASS_VERTICES = 32, 56, 176  # the grouped clipper's lists, and vertices of one geometry pass


@pytest.fixture(scope="module")
def ctx():
    c, torch = H.gpu_context()
    yield c, torch
    c.close()


def both(ctx, pos, box, **cfg):
    """(mesh, launches) by the warp-per-cell clipper (counters on) and by the dispatch's choice."""
    c, torch = ctx
    keep = {k: getattr(c.mm_get_config(), k) for k in cfg}
    out = []
    try:
        for counted in (1, 0):
            c.set_config(collect_stats=counted, **cfg)
            l0 = c.mm_kernel_launches()
            G = H.gpu_tessellate(c, torch, pos, box)[2]
            out.append((G, c.mm_kernel_launches() - l0))
    finally:
        c.set_config(collect_stats=0, **keep)
    for k in out[0][0]:
        np.testing.assert_array_equal(out[0][0][k], out[1][0][k], err_msg=k)
    return out


@pytest.mark.parametrize("n,grouped", [(4095, False), (4096, True), (4097, True)])
def test_grouped_clipper_runs_from_its_least_size_on(ctx, n, grouped):
    (_, counted), (_, plain) = both(ctx, WL.random_points(n, seed=50), np.ones(3))
    assert plain - counted == (1 if grouped else 0)


def layered(m=32, md=64, d=0.7 / 32, lz=0.5):
    """A sparse layer between two dense sheets: its cells have 26 faces on
    average and follow one another in the bins."""
    rng = np.random.default_rng(1)

    def sheet(k, z, j):
        g = (np.arange(k) + 0.5) / k
        p = np.stack(np.meshgrid(g, g, indexing="xy"), -1).reshape(-1, 2)
        p = np.mod(p + j / k * rng.uniform(-1, 1, p.shape), 1.0)
        return np.concatenate([p, np.full((len(p), 1), z)], 1)

    return np.concatenate([sheet(m, 0.5 * lz, 0.2), sheet(md, 0.5 * lz - d, 0.3), sheet(md, 0.5 * lz + d, 0.3)])


def test_list_and_second_geometry_pass(ctx):
    pos, box = layered(), np.array([1.0, 1.0, 0.5])
    (G, _), _ = both(ctx, pos, box)
    n = len(pos)
    faces = np.diff(G["inc_off"])
    # a cell of more faces than the grouped clipper has plane slots has gone to the list
    assert (faces > PLANES).sum() >= 1
    # four cells in a row whose vertices exceed one pass (a simple cell of F faces has 2 F - 4)
    g = np.maximum(1, np.floor(box / np.cbrt(np.prod(box) / n)).astype(int))
    b = np.minimum(np.floor(pos * (g / box)).astype(int), g - 1)
    row = faces[np.lexsort((np.arange(n), b[:, 0] + g[0] * (b[:, 1] + g[1] * b[:, 2])))][: n // 4 * 4].reshape(-1, 4)
    assert ((2 * row.max(1) - 4 <= VERTICES - 2) & ((2 * row - 4).sum(1) > PASS_VERTICES)).sum() >= 10


@pytest.mark.parametrize("bin_scale", [0.5, 0.8, 1.25, 2.0, 3.0, 4.0])
def test_bins_of_every_width(ctx, bin_scale):
    """From bins that hold a generator in eight (searches past the grouped
    clipper's shells) to crowded ones (its cells all go to the list)."""
    both(ctx, WL.random_points(8101, seed=51), np.ones(3), bin_scale=bin_scale)


@pytest.mark.parametrize("precision,integrator", [(0, 0), (1, 0), (0, 1)])
def test_batch_of_the_grouped_clipper_equals_boxes_alone(precision, integrator):
    """Boxes of 5 to 4500 generators, whose ends fall inside warps, in one
    batch of 8421 (grouped clipper); alone all but one take the other one."""
    import torch
    from paper_1707_05333_gb300 import binding
    sizes = [1501, 7, 333, 4500, 5, 2049, 26]
    shapes = [(1.0, 1.0, 1.0), (0.5, 0.7, 1.3), (2.0, 1.0, 1.0), (1.0, 1.0, 1.0), (1.0, 1.0, 1.0), (1.0, 0.25, 2.0),
              (1.0, 1.0, 1.0)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    assert off[-1] >= 4096 and np.any(off[1:-1] % 4 != 0)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        kw = dict(stream=stream, limiter=1, regularize=1, precision=precision, integrator=integrator)
        one, ref = binding.Context(**kw), binding.Context(**kw)
        P, U = [], []
        for k, (n, box) in enumerate(zip(sizes, shapes)):
            rho, vel, pres = WL.random_state(n, seed=60 + k, v_sigma=0.2)
            pb = H.to_dev(torch, WL.random_points(n, box=box, seed=70 + k).T)
            mesh = ref.mm_tessellate(pb, box)
            U.append(ref.mm_prims_to_charges(mesh, H.to_dev(torch, rho), H.to_dev(torch, vel.T), H.to_dev(torch, pres)))
            P.append(pb)
        pos, Ua = torch.cat(P, 1).contiguous(), torch.cat(U, 1).contiguous()
        dt = torch.empty(len(sizes), dtype=torch.float64, device="cuda")
        for step in range(2):
            one.mm_step_batched(pos, Ua, off, np.array(shapes), dt_out=dt)
            one.mm_sync_status()
            for b, box in enumerate(shapes):
                d1 = torch.empty(1, dtype=torch.float64, device="cuda")
                ref.mm_step(P[b], U[b], box, dt_out=d1)
                sl = slice(int(off[b]), int(off[b + 1]))
                assert torch.equal(pos[:, sl], P[b]) and torch.equal(Ua[:, sl], U[b]), (b, step)
                assert float(dt[b].item()) == float(d1.item()), (b, step)
        one.close()
        ref.close()


@pytest.mark.parametrize("value", [np.nan, -1e-9, 1.0, 1.5])
def test_generators_outside_the_box_are_refused(ctx, value):
    """One generator that is not in the box, and a whole warp of them: the
    call is refused and the context stays usable."""
    from paper_1707_05333_gb300 import binding
    c, torch = ctx
    for bad in ([17], list(range(40, 72))):
        pos = WL.random_points(5003, seed=52)
        pos[bad, 1] = value
        with pytest.raises(binding.MMError, match="outside"):
            H.gpu_tessellate(c, torch, pos, np.ones(3))
    assert abs(H.gpu_tessellate(c, torch, WL.random_points(5003, seed=52), np.ones(3))[2]["cell_volume"].sum() - 1.0) < 1e-12
