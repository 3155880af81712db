"""The MIXED push's object hits to the last bit: which particle is collected, and in which
cut cell, against the same FP32 operations (fused where the kernel fuses them) in numpy.
Millions of particles next to the surface in a frozen zero field, so that some end within
rounding of it, or cross it within rounding of a cell's face."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

F = np.float32


def _fma(a, b, c):
    """a b + c rounded once: the product is exact in FP64, where the sum is rounded to 53 bits first
    (which moves the FP32 result once in about 2^29)."""
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(F)


def _sum2(a, b, c, d, first):
    """a b + c d with the first product, else the second, rounded before the fused sum."""
    return _fma(c, d, F(a) * F(b)) if first else _fma(a, b, F(c) * F(d))


def _level(obj, x, y, z, first):
    kind, q = obj
    if kind == "sphere":
        dx, dy, dz = x - F(q[0]), y - F(q[1]), z - F(q[2])
        return _fma(dz, dz, _sum2(dx, dx, dy, dy, first)) - F(q[3] * q[3])
    if kind == "plane":
        return _fma(F(q[2]), z, _sum2(F(q[0]), x, F(q[1]), y, first)) - F(q[3])
    zg, xc, yc = q[:3]
    dx, dy = x - F(xc), y - F(yc)
    r2 = _sum2(dx, dx, dy, dy, first)
    if kind == "cap_crater":
        a, D = q[3:]
        Rs = (a * a + D * D) / (2.0 * D)
        with np.errstate(invalid="ignore"):
            return z - np.where(r2 < F(a * a), F((zg - D) + Rs) - np.sqrt(F(Rs * Rs) - r2), F(zg))
    ri, rt, ro, H, D = q[3:]
    r = np.sqrt(r2)
    t, u = (r - F(ri)) / F(rt - ri), (r - F(rt)) / F(ro - rt)
    up = _fma(F(D + H), (t * t) * (F(3) - F(2) * t), F(zg - D))
    down = _fma(-F(H), (u * u) * (F(3) - F(2) * u), F(zg + H))
    return z - np.where(r <= F(ri), F(zg - D), np.where(r <= F(rt), up, np.where(r < F(ro), down, F(zg))))


def _surface(obj, x, y):
    kind, q = obj
    if kind == "plane":
        return (q[3] - q[0] * x - q[1] * y) / q[2]
    zg, xc, yc = q[:3]
    r2 = (x - xc) ** 2 + (y - yc) ** 2
    if kind == "cap_crater":
        a, D = q[3:]
        Rs = (a * a + D * D) / (2.0 * D)
        return np.where(r2 < a * a, (zg - D) + Rs - np.sqrt(np.maximum(Rs * Rs - r2, 0.0)), zg)
    ri, rt, ro, H, D = q[3:]
    r = np.sqrt(r2)
    s = lambda t: t * t * (3 - 2 * t)
    return np.where(r <= rt, zg - D + (D + H) * s(np.clip((r - ri) / (rt - ri), 0, 1)),
                    zg + H - H * s(np.clip((r - rt) / (ro - rt), 0, 1)))


@pytest.mark.parametrize("edge,refine", [(4, 1), (8, 1), (4, 2)])
@pytest.mark.parametrize("obj,rounds", [(("sphere", (23.7, 24.1, 24.4, 13.3)), 6), (("plane", (0.31, -0.42, 1.0, 17.3)), 3),
                                        (("cap_crater", (14.3, 23.9, 24.2, 15.1, 6.3)), 2),
                                        (("rim_crater", (16.3, 24.2, 23.7, 6.1, 11.9, 17.6, 3.6, 6.2)), 2)])
def test_hits_to_the_last_bit(obj, rounds, edge, refine):
    from paper_2011_10214_gb300 import capi
    n, dt = 48, 0.15
    kinds = dict(sphere=capi.OBJ_SPHERE, plane=capi.OBJ_PLANE, cap_crater=capi.OBJ_CAP_CRATER,
                 rim_crater=capi.OBJ_RIM_CRATER)
    N = 1200000 if edge == 4 else 400000
    for k in range(rounds if (edge, refine) == (4, 1) else 1):
        g = np.random.default_rng(17 * k + len(obj[0]))
        off = g.uniform(1e-3, 0.2, N)
        if obj[0] == "sphere":
            d = g.normal(size=(3, N))
            d /= np.linalg.norm(d, axis=0)
            X = np.array(obj[1][:3])[:, None] + (obj[1][3] + off) * d
        else:
            X = g.uniform(1.0, 47.0, (3, N))
            X[2] = _surface(obj, X[0], X[1]) + off
        V = g.normal(size=(3, N)).astype(F).astype(np.float64)
        sim = capi.Simulation((n, n, n), 1.0, dt, precision=capi.MIXED, ife_refine=refine)
        sim.set_bin_edge(edge)
        sim.set_field_bc([("D", 0.0)] * 6)
        sim.set_object(kinds[obj[0]], list(obj[1]), 4.0, 1.0)
        sim.add_species(-1.0, 1.0, 0.01)
        sim.load_particles(0, *X, *V)
        sim.set_external_E(np.zeros(((n * refine + 1) ** 3, 3)))
        st = sim.step(1)
        assert st["dropped"][0] == 0
        # the move: an offset in a cell, drifted and split again
        cell = np.floor(X).astype(np.int64)
        f0 = np.minimum((X - cell).astype(F), F(0.99999994))
        f = _fma(V.astype(F), F(dt), f0)
        s = np.floor(f)
        f, new = f - s, cell + s.astype(np.int64)
        over = f >= 1
        f[over], new = F(0), new + over
        old, end = cell.astype(F) + f0, new.astype(F) + f
        inside = ((new >= 0) & (new < n)).all(0)
        Ln = _level(obj, *end, True)
        hit = inside & (Ln < 0)
        Lo = _level(obj, *old, False)[hit]
        t = Lo / (Lo - Ln[hit])
        at = [_fma(t, (e - o)[hit], o[hit]) for o, e in zip(old, end)]
        c = [np.clip(np.floor(F(refine) * a).astype(np.int64), 0, n * refine - 1) for a in at]
        target = sim.cell_target()[c[0] + n * refine * (c[1] + n * refine * c[2])]
        want = np.bincount(target[target >= 0], minlength=sim.sizes()["n_cut_cells"])
        assert hit.sum() > 0.1 * N
        assert st["collected"][0] == hit.sum()
        assert np.array_equal(sim.surface_counts(0), want), np.abs(sim.surface_counts(0) - want).sum()
        sim.close()
