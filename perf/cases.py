"""The work this library is used for, as timed cases.

A case is one call a user's program makes: a whole step of one box (`mm_step`),
of a batch of boxes (`mm_step_batched`) or of host arrays (`mm_step_host`), a
tessellation whose mesh is read out, or the step's stages called one by one.
The inputs are the synthetic test problems of `workloads.py` drawn on the
device (jittered lattices, uniform random generators), each from its own seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1707_05333_gb300 import binding

F8 = torch.float64

# fields a case may leave out
DEFAULTS = dict(precision=0, limiter=1, riemann=0, regularize=0, entropy=0, integrator=0, phase=0)


def listed():
    return [
        # the smallest run: one box of 16^3 generators, FP64, where launches and latency count
        dict(name="step_wave_16", kind="step", recipe="wave", nx=16, ny=16, nz=16),
        # the Sod tube in its long box, FP64 (gamma 1.4)
        dict(name="step_tube_128x16x16", kind="step", recipe="tube", nx=128, ny=16, nz=16),
        # the Gresho vortex in its thin box with every option of the FP64 scheme that
        # changes the arithmetic: Duffell-MacFadyen limiter, HLL, mesh regularisation
        dict(name="step_gresho_64x64x13", kind="step", recipe="gresho", nx=64, ny=64, nz=13, limiter=2, riemann=1,
             regularize=1),
        # the point blast in mixed precision
        dict(name="step_blast_64_mixed", kind="step", recipe="blast", nx=64, ny=64, nz=64, precision=1),
        # the energy/entropy switch (a sixth column), odd sizes, generators anywhere in their bins
        dict(name="step_entropy_97x51x33", kind="step", recipe="shear", nx=97, ny=51, nz=33, entropy=1, phase=1),
        # Heun integration: two tessellations and two flux stages a step
        dict(name="step_heun_72", kind="step", recipe="shear", nx=72, ny=72, nz=72, integrator=1, phase=1),
        # a shear layer in the middle of its run (generators anywhere in their bins), mixed precision
        dict(name="step_shear_131_mixed", kind="step", recipe="shear", nx=131, ny=131, nz=131, precision=1, phase=1),
        # the headline: the 256^3 shear layer in FP64
        dict(name="step_shear_256", kind="step", recipe="shear", nx=256, ny=256, nz=256),
        # the ensemble: 512 boxes of 2^10..2^16 random generators, one captured graph a step, mixed precision
        dict(name="batch_512_mixed", kind="batch", boxes=512, lo=10.0, hi=16.0, precision=1),
        # a tessellation used by itself: random generators, the whole mesh read out
        dict(name="tessellate_random_200003", kind="tessellate", n=200003, bx=1.0, by=1.0, bz=1.0),
        # a step on page-locked host arrays, copies included
        dict(name="host_shear_100", kind="host", recipe="shear", nx=100, ny=100, nz=100, phase=1),
        # a program that drives the stages itself and looks at the mesh and the gradients between them
        dict(name="stages_17x15x13", kind="stages", recipe="wave", nx=17, ny=15, nz=13, phase=1),
    ]


def draw(rng):
    """One more case of the same ranges: sides from 8 to 200 a box, 2 to 300
    boxes a batch, 500 to 2 million random generators."""
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "step", "batch", "tessellate", "host", "stages"])
    if kind == "batch":
        lo = rng.uniform(8.0, 11.0)
        return dict(kind=kind, boxes=side(2, 300), lo=lo, hi=lo + rng.uniform(0.5, 4.5),
                    precision=rng.choice([0, 1, 1]))
    if kind == "tessellate":
        return dict(kind=kind, n=side(500, 2_000_000), bx=1.0, by=rng.uniform(0.5, 2.0), bz=rng.uniform(0.5, 2.0))
    recipe = rng.choice(["wave", "tube", "shear", "gresho"] + ["blast"] * (kind != "host"))
    s = side(8, 32 if kind == "stages" else (110 if kind == "host" else 200))
    if recipe == "tube":
        nx, ny, nz = 4 * s, max(4, s // 2), max(4, s // 2 - 1)
    elif recipe == "gresho":
        nx, ny, nz = 2 * s, 2 * s, max(4, (2 * s) // 5)
    else:
        nx, ny, nz = s, max(4, s - rng.randrange(0, 4)), max(4, s + rng.randrange(0, 4))
    case = dict(kind=kind, recipe=recipe, nx=nx, ny=ny, nz=nz, phase=rng.randrange(2), limiter=rng.choice([1, 1, 1, 2, 3]),
                riemann=rng.choice([0, 0, 1]), regularize=rng.choice([0, 0, 1]))
    option = rng.choice(["plain", "plain", "mixed", "mixed", "entropy", "heun"])
    if option == "mixed":
        case["precision"] = 1
    elif option == "entropy" and kind != "stages":
        case["entropy"] = 1
    elif option == "heun" and kind != "stages" and _cells(case) <= 3_000_000:
        case["integrator"] = 1
    return case


def _opt(case, key):
    return case.get(key, DEFAULTS.get(key))


def _cells(case):
    if case["kind"] == "batch":
        return int(_batch_sizes(case).sum())
    if case["kind"] == "tessellate":
        return case["n"]
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Bytes and operations one pass cannot do without.

    Bytes: positions and charges read and written once (a tessellation:
    positions in, the mesh out; 8 faces a cell).  Operations: the FP64 work of
    the clipped cells (28 vertices of 41 operations, 84 face corners of 9, 16
    faces of 45), which every path does, and of the finite-volume update (two
    gradients of 16 faces a cell, 8 fluxes a cell of 236) where it runs in
    FP64."""
    n = _cells(case)
    mesh_flops = n * (28 * 41 + 84 * 9 + 16 * 45)
    mesh_bytes = n * (8 * (12 + 8 + 24 + 24) + 8 + 24 + 4 + 16 * 4)
    if case["kind"] == "tessellate":
        return {"bytes": 24 * n + mesh_bytes, "flops": mesh_flops}
    hydro = n * (2 * 16 * 40 + 8 * 236 + 16 * 10)
    tess = 2 if _opt(case, "integrator") else 1
    rows = 6 if _opt(case, "entropy") else 5
    b = 2 * n * (24 + 8 * rows)
    if case["kind"] == "stages":
        b += mesh_bytes + n * (24 + 120)
    return {"bytes": b, "flops": tess * (mesh_flops + hydro)}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _lattice(case, gen, dev):
    """Jittered lattice (+-0.1 spacing) in the recipe's box, (3, n), and the box."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h = {"tube": (8.0 / nx, 1.0 / ny, 1.0 / nz), "gresho": (1.0 / nx, 1.0 / ny, 0.2 / nz)}.get(
        case["recipe"], (1.0 / nx,) * 3)
    box = [nx * h[0], ny * h[1], nz * h[2]]
    pos = torch.empty((3, nx * ny * nz), dtype=F8, device=dev)
    ix = torch.arange(nx * ny * nz, device=dev)
    shift = torch.rand(3, dtype=F8, generator=gen, device=dev).tolist()
    for d, k in enumerate((ix % nx, (ix // nx) % ny, ix // (nx * ny))):
        x = k.to(F8) + 0.5 + (shift[d] if _opt(case, "phase") else 0.0)
        x += torch.rand(x.shape, dtype=F8, generator=gen, device=dev).mul_(0.2).sub_(0.1)
        x = torch.remainder(x * h[d], box[d])
        pos[d] = torch.where(x >= box[d], torch.zeros_like(x), x)
    return pos, box


def _fields(case, pos, box):
    """Density, velocity (3, n) and pressure of the recipe at the generators, and gamma."""
    x, y = pos[0], pos[1]
    one = torch.ones_like(x)
    vel = torch.zeros_like(pos)
    recipe = case["recipe"]
    if recipe == "wave":
        vel[:] = 0.01 * torch.sin(2.0 * math.pi * x / box[0])
        return one, vel, one.clone(), 5.0 / 3.0
    if recipe == "tube":
        left = x < 0.5 * box[0]
        return torch.where(left, 1.0, 0.125).to(F8), vel, torch.where(left, 1.0, 0.1).to(F8), 1.4
    if recipe == "blast":
        return one, vel, one * 1e-5, 5.0 / 3.0
    if recipe == "shear":
        inner = (y / box[1] - 0.5).abs() < 0.25
        vel[0] = torch.where(inner, 0.5, -0.5).to(F8)
        vel[1] = 0.01 * torch.sin(4.0 * math.pi * x / box[0])
        return torch.where(inner, 2.0, 1.0).to(F8), vel, one * 2.5, 5.0 / 3.0
    dx, dy = x - 0.5, y - 0.5
    r = torch.sqrt(dx * dx + dy * dy).clamp_min(1e-300)
    vphi = torch.where(r < 0.2, 5.0 * r, torch.where(r < 0.4, 2.0 - 5.0 * r, torch.zeros_like(r)))
    mid = 9.0 + 12.5 * r * r - 20.0 * r + 4.0 * torch.log(5.0 * r)
    pres = torch.where(r < 0.2, 5.0 + 12.5 * r * r, torch.where(r < 0.4, mid, one * (3.0 + 4.0 * math.log(2.0))))
    vel[0], vel[1] = -vphi * dy / r, vphi * dx / r
    return one, vel, pres, 5.0 / 3.0


def _deposit(case, pos, U):
    """The blast's thermal energy of 1 in the 8 generators nearest the centre."""
    if case["recipe"] == "blast":
        d2 = ((pos - 0.5) ** 2).sum(0)
        U[4, torch.topk(d2, 8, largest=False).indices] += 0.125


def _batch_sizes(case):
    rng = np.random.Generator(np.random.PCG64(int(case["boxes"] * 1000 + 10 * case["lo"] + case["hi"])))
    return np.rint(2.0 ** rng.uniform(case["lo"], case["hi"], size=case["boxes"])).astype(np.int64)


def _random_field(gen, dev, m=32):
    """Periodic Gaussian random field of unit variance with power spectrum k^-3."""
    k = torch.fft.fftfreq(m, device=dev, dtype=F8) * m
    kk = torch.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2)
    amp = torch.where(kk > 0, kk.clamp_min(1.0) ** -1.5, torch.zeros_like(kk))
    noise = torch.randn((m, m, m), dtype=F8, generator=gen, device=dev)
    f = torch.fft.ifftn(torch.fft.fftn(noise) * amp).real
    return (f - f.mean()) / f.std()


def _sample(field, pos):
    """Trilinear samples of a periodic field on the unit box at pos (3, n)."""
    m = field.shape[0]
    x = pos * m - 0.5
    i0 = torch.floor(x)
    f = x - i0
    i0 = i0.to(torch.int64)
    out = torch.zeros_like(pos[0])
    for c in range(8):
        w, idx = 1.0, []
        for d in range(3):
            b = (c >> d) & 1
            w = w * (f[d] if b else 1.0 - f[d])
            idx.append((i0[d] + b) % m)
        out += w * field[idx[0], idx[1], idx[2]]
    return out


def _mesh_buffers(n, dev):
    """Arrays a program keeps for the meshes of n cells it reads out: faces at a
    capacity (a periodic Voronoi mesh has about 8 a cell), zero past the mesh's own."""
    cap = 10 * n + 1024
    shapes = dict(face_i=(cap,), face_j=(cap,), face_shift=(cap,), face_area=(cap,), face_normal=(3, cap),
                  face_centroid=(3, cap), cell_volume=(n,), cell_centroid=(3, n), inc_off=(n + 1,), inc_face=(2 * cap,))
    ints = ("face_i", "face_j", "face_shift", "inc_off", "inc_face")
    return {k: torch.zeros(s, dtype=torch.int32 if k in ints else F8, device=dev) for k, s in shapes.items()}


def _read_mesh(mesh, kept):
    """The mesh's arrays in the program's own buffers."""
    for k, v in mesh.to_torch().items():
        kept[k][..., :v.shape[-1]].copy_(v)
    return dict(kept)


def _config(case, gamma):
    return dict(gamma=gamma, cfl=0.3, precision=_opt(case, "precision"), limiter=_opt(case, "limiter"),
                riemann=_opt(case, "riemann"), regularize=_opt(case, "regularize"), entropy=_opt(case, "entropy"),
                integrator=_opt(case, "integrator"))


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    st = {"kind": case["kind"]}
    if case["kind"] == "tessellate":
        box = [case["bx"], case["by"], case["bz"]]
        st["pos"] = torch.rand((3, case["n"]), dtype=F8, generator=gen, device=dev) * torch.tensor(
            box, dtype=F8, device=dev)[:, None]
        st["box"] = box
        st["mesh"] = _mesh_buffers(case["n"], dev)
        st["ctx"] = binding.Context()
        return st
    if case["kind"] == "batch":
        return _prepare_batch(case, gen, dev, st)
    pos, box = _lattice(case, gen, dev)
    rho, vel, pres, gamma = _fields(case, pos, box)
    ctx = binding.Context(**_config(case, gamma))
    mesh = ctx.mm_tessellate(pos, box)
    U = ctx.mm_prims_to_charges(mesh, rho, vel, pres)
    _deposit(case, pos, U)
    st.update(ctx=ctx, box=box, pos=pos, U=U, dt=torch.empty(1, dtype=F8, device=dev))
    if case["kind"] == "step":
        st.update(pos0=pos.clone(), U0=U.clone())
    if case["kind"] == "host":
        st["pos"] = pos.cpu().pin_memory()
        st["U"] = U.cpu().pin_memory()
        st["dt"] = torch.empty(1, dtype=F8).pin_memory()
    elif case["kind"] == "stages":
        W = torch.empty_like(U)
        torch.div(U, mesh.to_torch()["cell_volume"], out=W)
        st.update(W=W, pos_out=torch.empty_like(pos), U_out=torch.empty_like(U),
                  mesh=_mesh_buffers(pos.shape[1], dev))
    torch.cuda.synchronize()
    return st


def _prepare_batch(case, gen, dev, st):
    sizes = _batch_sizes(case)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    pos = torch.rand((3, n), dtype=F8, generator=gen, device=dev)
    vel = 0.1 * torch.randn((3, n), dtype=F8, generator=gen, device=dev)
    U = torch.empty((5, n), dtype=F8, device=dev)
    helper = binding.Context()
    for b, m in enumerate(sizes):
        sl = slice(int(off[b]), int(off[b + 1]))
        p = pos[:, sl].contiguous()
        rho = torch.exp(0.5 * _sample(_random_field(gen, dev), p) - 0.125)
        mesh = helper.mm_tessellate(p, (1.0, 1.0, 1.0))
        U[:, sl] = helper.mm_prims_to_charges(mesh, rho, vel[:, sl].contiguous(), torch.ones_like(rho))
    helper.close()
    torch.cuda.synchronize()
    st.update(pos0=pos.clone(), U0=U.clone())
    st.update(ctx=binding.Context(stream=stream, **_config(case, 5.0 / 3.0)), stream=stream, pos=pos, U=U, off=off,
              boxes=np.ones((len(sizes), 3)), dt=torch.empty(len(sizes), dtype=F8, device=dev))
    return st


def run(st):
    ctx, kind = st["ctx"], st["kind"]
    if kind in ("step", "batch"):
        # each pass is the same step: from the snapshot the program keeps, not
        # hundreds of steps into a run (an unregularised blast mesh tangles there)
        st["pos"].copy_(st["pos0"])
        st["U"].copy_(st["U0"])
    if kind == "step":
        ctx.mm_step(st["pos"], st["U"], st["box"], dt_out=st["dt"])
    elif kind == "batch":
        # the step runs on the context's own stream: order it with the caller's on both sides
        cur = torch.cuda.current_stream()
        st["stream"].wait_stream(cur)
        ctx.mm_step_batched(st["pos"], st["U"], st["off"], st["boxes"], dt_out=st["dt"])
        cur.wait_stream(st["stream"])
    elif kind == "host":
        ctx.mm_step_host(st["pos"], st["U"], st["box"], dt_out=st["dt"])
    elif kind == "tessellate":
        return _read_mesh(ctx.mm_tessellate(st["pos"], st["box"]), st["mesh"])
    else:
        pos, U = st["pos_out"], st["U_out"]
        pos.copy_(st["pos"])
        U.copy_(st["U"])
        mesh = ctx.mm_tessellate(pos, st["box"])
        out = _read_mesh(mesh, st["mesh"])
        w = ctx.mm_mesh_velocity(mesh, pos, U)
        dt = ctx.mm_timestep(mesh, U, w)
        grad = ctx.mm_gradients(mesh, st["W"])
        ctx.mm_flux_step(mesh, pos, w, dt, U)
        ctx.mm_drift(pos, w, dt, st["box"])
        out.update(w=w, dt=dt, grad=grad, U=U, pos=pos, totals=ctx.mm_totals(U))
        return out
    return {"pos": st["pos"], "U": st["U"], "dt": st["dt"]}


# --------------------------------------------------------------------------
# the same results in 64 bits by plain numpy, for the small lattices
# --------------------------------------------------------------------------
EXACT_CELLS = 5000
EXACT_PLANES = 34  # neighbours a jittered lattice cell is cut with


def _voronoi(pos, box):
    """Directed faces (cell, neighbour, image shift, area, centroid relative to
    the cell's generator, separation q), volumes and centroids of a periodic
    Voronoi mesh whose cells are bounded by their EXACT_PLANES nearest
    neighbours, or None where that does not hold.  A vertex is the
    intersection of three bisector planes that lies behind every other one."""
    n, K = pos.shape[0], EXACT_PLANES
    img = np.stack(np.meshgrid(*[np.arange(-1, 2)] * 3, indexing="ij"), -1).reshape(-1, 3)
    tri = np.array([(a, b, c) for a in range(K) for b in range(a + 1, K) for c in range(b + 1, K)])
    a, b, c = tri.T
    cells, nbs, shs, qs, verts, corner = [], [], [], [], [], []
    for lo in range(0, n, 64):
        ids = np.arange(lo, min(n, lo + 64))
        d = pos[None, :, :] - pos[ids][:, None, :]
        s0 = -np.rint(d / box)
        d0 = d + s0 * box
        near = np.argpartition((d0 ** 2).sum(-1), min(4 * K, n - 1), axis=1)[:, :4 * K + 1]
        q = np.take_along_axis(d, near[..., None], 1)[:, :, None, :] + (img * box)[None, None]
        r2 = (q ** 2).sum(-1).reshape(len(ids), -1)
        r2[r2 == 0.0] = np.inf
        pick = np.argsort(r2, axis=1)[:, :K + 1]
        reach = np.sqrt(np.take_along_axis(r2, pick[:, K:], 1))[:, 0]
        pick = pick[:, :K]
        q = np.take_along_axis(q.reshape(len(ids), -1, 3), pick[..., None], 1)
        nb = np.take_along_axis(near, pick // 27, 1)
        o = 0.5 * (q ** 2).sum(-1)
        qa, qb, qc = q[:, a], q[:, b], q[:, c]
        bc = np.cross(qb, qc)
        det = (qa * bc).sum(-1)
        ok = np.abs(det) > 1e-9 * (np.sqrt((2 * o) ** 3).max())
        v = (o[:, a, None] * bc + o[:, b, None] * np.cross(qc, qa) + o[:, c, None] * np.cross(qa, qb)) / np.where(
            ok, det, 1.0)[..., None]
        ok &= (v ** 2).sum(-1) < (0.25 * reach ** 2)[:, None]
        for k in range(len(ids)):
            t = np.nonzero(ok[k])[0]
            behind = v[k, t] @ q[k].T - o[k]
            behind[np.arange(len(t))[:, None], tri[t]] = -1.0
            t = t[(behind <= 0.0).all(1)]
            used = np.unique(tri[t])
            if len(t) != 2 * (len(used) - 2):
                return None
            cells.append(np.full(K, ids[k]))
            nbs.append(nb[k])
            shs.append(img[pick[k] % 27])
            qs.append(q[k])
            verts.append(v[k, t])
            corner.append(tri[t] + K * ids[k])
    cells, nbs, shs, qs = (np.concatenate(x) for x in (cells, nbs, shs, qs))
    verts, corner = np.concatenate(verts), np.concatenate(corner)
    # order each face's vertices by angle about their mean, then sum the fan
    f = corner.ravel()
    vv = np.repeat(verts, 3, axis=0)
    cnt = np.bincount(f, minlength=len(cells))
    mean = np.stack([np.bincount(f, vv[:, d], len(cells)) for d in range(3)], 1) / np.maximum(cnt, 1)[:, None]
    nrm = qs / np.linalg.norm(qs, axis=1)[:, None]
    e1 = np.cross(nrm, np.eye(3)[np.argmin(np.abs(nrm), axis=1)])
    e1 /= np.linalg.norm(e1, axis=1)[:, None]
    e2 = np.cross(nrm, e1)
    r = vv - mean[f]
    u, w = (r * e1[f]).sum(1), (r * e2[f]).sum(1)
    order = np.lexsort((np.arctan2(w, u), f))
    f, u, w = f[order], u[order], w[order]
    first = np.concatenate([[True], f[1:] != f[:-1]])
    start = np.nonzero(first)[0]
    nxt = np.arange(len(f)) + 1
    nxt[np.concatenate([start[1:], [len(f)]]) - 1] = start
    cr = u * w[nxt] - w * u[nxt]
    area = 0.5 * np.bincount(f, cr, len(cells))
    with np.errstate(divide="ignore", invalid="ignore"):
        cu = np.bincount(f, cr * (u + u[nxt]), len(cells)) / (6.0 * area)
        cw = np.bincount(f, cr * (w + w[nxt]), len(cells)) / (6.0 * area)
    keep = cnt > 2
    fc = mean + cu[:, None] * e1 + cw[:, None] * e2
    cells, nbs, shs, qs, area, fc = (x[keep] for x in (cells, nbs, shs, qs, area, fc))
    vp = area * np.linalg.norm(qs, axis=1) / 6.0
    vol = np.bincount(cells, vp, n)
    cen = pos + 0.75 * np.stack([np.bincount(cells, vp * fc[:, d], n) for d in range(3)], 1) / vol[:, None]
    # the image shift of the pair: q = r_j + s L - r_i
    shs = np.rint((qs - pos[nbs] + pos[cells]) / box).astype(np.int64)
    big = area > 1e-10 * (np.prod(box) / n) ** (2.0 / 3.0)
    return dict(i=cells[big], j=nbs[big], s=shs[big], q=qs[big], area=area[big], fc=fc[big], vol=vol, cen=cen)


def _limited_gradient(T, box, W):
    """Centroid Green-Gauss gradient of W (n, k) with the S10 limiter, (n, k, 3)."""
    n, i, j = len(T["vol"]), T["i"], T["j"]
    an = T["area"][:, None] * T["q"] / np.linalg.norm(T["q"], axis=1)[:, None]
    d = T["cen"][j] + T["s"] * box - T["cen"][i]
    M = np.zeros((n, 3, 3))
    b = np.zeros((n, W.shape[1], 3))
    dW = W[j] - W[i]
    np.add.at(M, i, 0.5 * an[:, :, None] * d[:, None, :])
    np.add.at(b, i, 0.5 * dW[:, :, None] * an[:, None, :])
    g = np.einsum("nab,nkb->nka", np.linalg.inv(M), b)
    hi, lo = W.copy(), W.copy()
    np.maximum.at(hi, i, W[j])
    np.minimum.at(lo, i, W[j])
    delta = np.einsum("fka,fa->fk", g[i], d)
    alpha = np.ones_like(W)
    with np.errstate(divide="ignore", invalid="ignore"):
        psi = np.where(delta > 0, (hi - W)[i] / delta, np.where(delta < 0, (lo - W)[i] / delta, 1.0))
    np.minimum.at(alpha, i, psi)
    return g * np.minimum(1.0, alpha)[:, :, None]


def _hllc(L, R, nrm, gamma):
    """HLLC flux along nrm of primitive rows (rho, v, P), Davis speeds."""
    def side(S):
        rho, v, P = S[:, 0], S[:, 1:4], S[:, 4]
        u = (v * nrm).sum(1)
        E = P / (gamma - 1.0) + 0.5 * rho * (v ** 2).sum(1)
        U = np.concatenate([rho[:, None], rho[:, None] * v, E[:, None]], 1)
        F = U * u[:, None]
        F[:, 1:4] += P[:, None] * nrm
        F[:, 4] += P * u
        return rho, v, P, u, np.sqrt(gamma * P / rho), E, U, F

    rl, vl, pl, ul, cl, El, Ul, Fl = side(L)
    rr, vr, pr, ur, cr, Er, Ur, Fr = side(R)
    sl, sr = np.minimum(ul - cl, ur - cr), np.maximum(ul + cl, ur + cr)
    ml, mr = rl * (sl - ul), rr * (sr - ur)
    ss = (pr - pl + ul * ml - ur * mr) / (ml - mr)

    def star(rho, v, P, u, s, E, U, F):
        f = rho * (s - u) / (s - ss)
        Us = np.concatenate([f[:, None], f[:, None] * (v + (ss - u)[:, None] * nrm),
                             (f * (E / rho + (ss - u) * ss) + (ss - u) * P / (s - ss))[:, None]], 1)
        return F + s[:, None] * (Us - U)

    out = np.where((ss >= 0)[:, None], star(rl, vl, pl, ul, sl, El, Ul, Fl), star(rr, vr, pr, ur, sr, Er, Ur, Fr))
    out = np.where((sl >= 0)[:, None], Fl, out)
    return np.where((sr <= 0)[:, None], Fr, out)


def _exact_step(T, pos, box, U, gamma, W=None):
    """w, dt, limited gradients of W, and the charges and positions after one
    half-step MUSCL-HLLC step with the mesh moving at the fluid velocity."""
    vol, cen, i, j = T["vol"], T["cen"], T["i"], T["j"]
    W0 = U / vol[:, None]
    w = U[:, 1:4] / U[:, :1]

    def pressure(W):
        return (gamma - 1.0) * (W[:, 4] - 0.5 * (W[:, 1:4] ** 2).sum(1) / W[:, 0])

    R = np.cbrt(3.0 * vol / (4.0 * math.pi))
    dt = (0.3 * R / np.sqrt(gamma * pressure(W0) / W0[:, 0])).min()
    grad = _limited_gradient(T, box, W0 if W is None else W)
    g = _limited_gradient(T, box, W0)
    u = W0[:, 1:4] / W0[:, :1]
    du = (g[:, 1:4] - u[:, :, None] * g[:, :1]) / W0[:, 0][:, None, None]
    dP = (gamma - 1.0) * (g[:, 4] - (u[:, :, None] * g[:, 1:4]).sum(1) + 0.5 * (u ** 2).sum(1)[:, None] * g[:, 0])
    div = du[:, 0, 0] + du[:, 1, 1] + du[:, 2, 2]
    rate = np.empty_like(W0)
    rate[:, 0] = -(g[:, 1, 0] + g[:, 2, 1] + g[:, 3, 2])
    rate[:, 1:4] = -((g[:, 1:4] * u[:, None, :]).sum(2) + W0[:, 1:4] * div[:, None]) - dP
    rate[:, 4] = -((u * (g[:, 4] + dP)).sum(1) + (W0[:, 4] + pressure(W0)) * div)
    Wh = W0 + 0.5 * dt * rate
    gh = _limited_gradient(T, box, Wh)
    code = (T["s"] + 1) @ np.array([1, 3, 9])
    uni = (i < j) | ((i == j) & (code > 13))
    i, j, s, q, A, fc = (T[k][uni] for k in ("i", "j", "s", "q", "area", "fc"))
    xf = pos[i] + fc
    L = Wh[i] + np.einsum("fka,fa->fk", gh[i], xf - cen[i])
    Rt = Wh[j] + np.einsum("fka,fa->fk", gh[j], xf - cen[j] - s * box)
    corr = ((w[i] - w[j]) * (fc - 0.5 * q)).sum(1) / (q ** 2).sum(1)
    wf = corr[:, None] * q + 0.5 * (w[i] + w[j])

    def boosted(W):
        return np.concatenate([W[:, :1], W[:, 1:4] / W[:, :1] - wf, pressure(W)[:, None]], 1)

    F = _hllc(boosted(L), boosted(Rt), q / np.linalg.norm(q, axis=1)[:, None], gamma)
    F[:, 4] += (F[:, 1:4] * wf).sum(1) + 0.5 * (wf ** 2).sum(1) * F[:, 0]
    F[:, 1:4] += F[:, :1] * wf
    F *= A[:, None]
    Un = U.copy()
    np.add.at(Un, i, -dt * F)
    np.add.at(Un, j, dt * F)
    return w, dt, grad, Un, np.mod(pos + w * dt, box)


def exact(case, seed):
    plain = all(_opt(case, k) == v for k, v in DEFAULTS.items() if k != "phase")
    if case["kind"] not in ("step", "host", "stages") or case["recipe"] != "wave" or not plain:
        return None
    if not 500 <= _cells(case) <= EXACT_CELLS or min(case["nx"], case["ny"], case["nz"]) < 8:
        return None
    dev = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    p, box = _lattice(case, gen, dev)
    rho, vel, pres, gamma = (x.cpu().numpy() if torch.is_tensor(x) else x for x in _fields(case, p, box))
    pos, box = np.ascontiguousarray(p.cpu().numpy().T), np.array(box)
    T = _voronoi(pos, box)
    if T is None:
        return None
    m = rho * T["vol"]
    E = (pres / (gamma - 1.0) + 0.5 * rho * (vel ** 2).sum(0)) * T["vol"]
    U = np.stack([m, m * vel[0], m * vel[1], m * vel[2], E], 1)
    w, dt, grad, Un, pn = _exact_step(T, pos, box, U, gamma)

    def rows(a):
        return torch.from_numpy(np.ascontiguousarray(a.T))

    dt = torch.tensor([dt], dtype=F8)
    if case["kind"] != "stages":
        return {"pos": rows(pn), "U": rows(Un), "dt": dt}
    out = dict.fromkeys(["face_i", "face_j", "face_shift", "face_area", "face_normal", "face_centroid", "inc_off",
                         "inc_face"])
    out.update(cell_volume=torch.from_numpy(T["vol"]), cell_centroid=rows(T["cen"]), w=rows(w), dt=dt,
               grad=rows(grad.reshape(len(pos), 15)), U=rows(Un), pos=rows(pn), totals=torch.from_numpy(Un.sum(0)))
    return out
