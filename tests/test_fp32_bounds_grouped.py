"""The FP32 bounds of the grouped clipper's own screens, by host emulation of
its FP32 arithmetic (the vertices and their bounds are test_fp32_bounds.py's):

* it tests planes with |q| rmax + o in place of the sum of magnitudes, rmax
  being 1 % above the root of the security limit;
* it drops a candidate when no vertex comes nearer its plane than 17 u of that;
* it passes over bins whose nearest point lies beyond the gather threshold by
  2 % and a slack.

The hardware's root is taken one unit in the last place low, its worst."""
import numpy as np

from tests.test_fp32_bounds import U32, _f32, _fma, _mul, _vertex32

UNIT = U32(5.9604645e-8)


def root(x):
    return np.nextafter(np.sqrt(x.astype(U32)), U32(0.0))


def screened(qn, rmax, fo, E, s32):
    """Candidates the clipper drops: no vertex nearer the plane than 17 u (|q| rmax + o)."""
    far = _fma(np.repeat(qn[:, None], E.shape[1], 1), E, s32).max(1)
    return far < -_mul(U32(17.0) * UNIT * U32(1.0001), _fma(qn, rmax, fo))


def test_plane_test_and_screen():
    """Cells of vertices of random bisectors and candidate planes at all
    distances, many within the bounds of a vertex: every settled sign is the
    exact test's, and no dropped candidate has a vertex beyond it."""
    rng = np.random.default_rng(1713)
    m, nv = 4000, 12
    settled = dropped = worst = 0
    for scale in (2.0 ** -20, 1.0, 2.0 ** 20):
        def planes(k):
            d = rng.normal(size=(k, 3))
            d /= np.linalg.norm(d, axis=1, keepdims=True)
            return d * rng.uniform(0.3, 3.0, (k, 1)) * scale
        qa, qb, qc = planes(m * nv), planes(m * nv), planes(m * nv)
        o = [0.5 * (q * q).sum(1) for q in (qa, qb, qc)]
        v32, err = _vertex32(qa, o[0], qb, o[1], qc, o[2])
        A = np.stack([qa, qb, qc], 1)
        det = np.abs(np.linalg.det(A)) / np.prod(np.linalg.norm(A, axis=2), axis=1)
        v = np.linalg.solve(np.where(det[:, None, None] > 1e-9, A, np.eye(3) * scale), np.stack(o, 1)[..., None])[..., 0]
        # ill-conditioned ones: the clipper keeps the FP32 rounding of the exact vertex
        exact = ~np.isfinite(err)
        v[det <= 1e-9] = scale
        v32[exact] = _f32(v[exact])
        err = np.where(exact, _fma(U32(1.2e-7) * np.ones(len(v), U32), _f32(np.abs(v32).sum(1)), U32(1e-38) * np.ones(len(v), U32)), err)
        # near vertices only: cells are bounded
        near = np.linalg.norm(v, axis=1) < 20.0 * scale
        v[~near], v32[~near], err[~near] = 0.0, 0.0, U32(1e-30)
        x, y, z = v32.T
        e = err.astype(U32)
        l1 = np.abs(x) + np.abs(y) + np.abs(z)
        r2 = _mul(_fma(e, _fma(U32(2.0) * np.ones_like(l1), l1, e), _fma(x, x, _fma(y, y, _mul(z, z)))), U32(1.00001))
        lim4 = U32(4.0) * r2.reshape(m, nv).max(1)
        rmax = _mul(root(_mul(U32(0.25), lim4)), U32(1.01))
        assert np.all(rmax[:, None] >= np.linalg.norm(v, axis=1).reshape(m, nv))
        assert np.all(rmax[:, None] >= np.linalg.norm(v32.astype(float), axis=1).reshape(m, nv))
        # candidate planes, a third of them through a vertex up to a few parts in 1e7
        q = planes(m)
        V = v.reshape(m, nv, 3)
        touch = rng.random(m) < 0.34
        d = q / np.linalg.norm(q, axis=1, keepdims=True)
        t = (V[:, 0] * d).sum(1)
        touch &= t > 0.01 * scale
        q[touch] = (2.0 * t * (1.0 + 3e-7 * rng.normal(size=m)))[touch, None] * d[touch]
        oq = 0.5 * (q * q).sum(1)
        fq, fo = _f32(q), _f32(oq)
        qn = _mul(root(_mul(U32(2.0), fo)), U32(1.00003))
        W = v32.reshape(m, nv, 3)
        c = [np.repeat(fq[:, k, None], nv, 1) for k in range(3)]
        s32 = _fma(c[0], W[..., 0], _fma(c[1], W[..., 1], _fma(c[2], W[..., 2], np.repeat(-fo[:, None], nv, 1))))
        s = (q[:, None] * V).sum(2) - oq[:, None]
        size = _fma(qn, rmax, fo)
        E = err.astype(U32).reshape(m, nv)
        B = _fma(np.repeat(qn[:, None], nv, 1), E, np.repeat(_mul(U32(16.0) * UNIT * U32(1.0001), size)[:, None], nv, 1))
        margin = (np.spacing(oq) * 2.0 ** 13)[:, None]
        beyond, inside = s32 > B, s32 < -B
        # (the exact test's own sign, rounding of the reference aside)
        noise = 1e-13 * (np.linalg.norm(q, axis=1) * np.linalg.norm(V, axis=2).max(1) + oq)[:, None]
        assert np.all((s > margin - noise)[beyond]) and np.all((s <= margin + noise)[inside])
        assert np.all(np.abs(s32.astype(float) - s) <= B + noise)
        worst = max(worst, float(np.max(np.abs(s32.astype(float) - s) / (B + noise))))
        settled += int(beyond.sum() + inside.sum())
        drop = screened(qn, rmax, fo, E, s32)
        assert np.all((s <= margin + noise)[drop])
        dropped += int(drop.sum())
        # candidates further out, which rarely cut, against the same vertices
        q *= rng.uniform(1.0, 20.0, (m, 1))
        oq = 0.5 * (q * q).sum(1)
        fq, fo = _f32(q), _f32(oq)
        qn = _mul(root(_mul(U32(2.0), fo)), U32(1.00003))
        c = [np.repeat(fq[:, k, None], nv, 1) for k in range(3)]
        s32 = _fma(c[0], W[..., 0], _fma(c[1], W[..., 1], _fma(c[2], W[..., 2], np.repeat(-fo[:, None], nv, 1))))
        s = (q[:, None] * V).sum(2) - oq[:, None]
        noise = 1e-13 * (np.linalg.norm(q, axis=1) * np.linalg.norm(V, axis=2).max(1) + oq)[:, None]
        drop = screened(qn, rmax, fo, E, s32)
        assert np.all((s <= (np.spacing(oq) * 2.0 ** 13)[:, None] + noise)[drop])
        dropped += int(drop.sum())
    print(f"[grouped clipper bounds] worst |ds|/B {worst:.2f}, {settled} settled, {dropped} dropped")
    assert settled > 0.9 * 3 * m * nv * 0.9 and dropped > 0.1 * m and worst < 1.0


def test_no_bin_with_a_gathered_candidate_is_passed_over():
    """Generators of the bins around a cell's, in boxes of several shapes and
    scales: whatever the FP32 filter keeps at a threshold lies in a bin whose
    nearest point, as the clipper forms it, is within reach of it."""
    rng = np.random.default_rng(1714)
    n = 200000
    closest = np.inf
    for L in (np.array([1.0, 1.0, 1.0]), np.array([1.0, 0.5, 2.0]), 2.0 ** 30 * np.array([1.0, 1.0, 0.25]),
              2.0 ** -38 * np.array([3.0, 1.0, 1.0])):
        g = np.array([40, 23, 64])
        bs = L / g
        bsf, ibsf = _f32(bs), _f32(g / L)
        slack = U32(2e-6) * _f32(L.max())
        p = rng.uniform(0.0, 1.0, (n, 3)) * L
        q = rng.normal(size=(n, 3))
        q *= (bs.max() * rng.uniform(0.05, 5.0, (n, 1))) / np.linalg.norm(q, axis=1, keepdims=True)
        # half of them put against a bin wall, where rounding decides the bin
        x = p + q
        wall = rng.random((n, 3)) < 0.5
        x = np.where(wall, np.round(x / bs) * bs * (1.0 + rng.normal(size=(n, 3)) * 2.0 ** -52), x)
        ok = np.all((x >= 0.0) & (x < L), axis=1)
        p, x = p[ok], x[ok]
        cb = np.clip(np.floor(_f32(p) * ibsf).astype(int), 0, g - 1)  # the cell's own bin, in FP32
        ob = np.clip(np.floor(x * (g / L)).astype(int), 0, g - 1)     # the generator's, in FP64
        pf = _f32(p)
        lo = _f32(_f32(pf - _f32(cb.astype(U32) * bsf)) - slack)
        hi = _f32(_f32(_f32((cb + 1).astype(U32) * bsf) - pf) - slack)
        o = ob - cb
        one = np.broadcast_to(bsf, o.shape)
        d = np.where(o == 0, U32(0.0), np.maximum(np.where(o > 0, _fma((o - 1).astype(U32), one, hi),
                                                           _fma((-o - 1).astype(U32), one, lo)), U32(0.0)))
        near2 = _fma(d[:, 0], d[:, 0], _fma(d[:, 1], d[:, 1], _mul(d[:, 2], d[:, 2])))
        q32 = _f32(_f32(x) - pf)
        d2f = _fma(q32[:, 0], q32[:, 0], _fma(q32[:, 1], q32[:, 1], _mul(q32[:, 2], q32[:, 2])))
        limk = d2f  # the tightest threshold that keeps it
        reach = _mul(U32(1.02), _fma(slack * np.ones_like(limk), root(limk), limk))
        assert np.all(near2 <= reach)
        closest = min(closest, float(np.min((reach.astype(float) - near2) / reach)))
    print(f"[bins within reach] least margin {closest:.4f} of the reach")
    assert closest > 0.0
