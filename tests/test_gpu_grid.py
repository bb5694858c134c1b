"""Labels from the cell grid (the default path) against the general tile
kernels and the FP64 oracle: the surfaces and points where a cell's anchor,
its triangle list or a crossing test could go wrong."""
import math

import numpy as np
import pytest

import zef_synth as zs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
FOUR_PI = 4.0 * math.pi


def _surf(v, t, cid=1):
    return zs.Surface(cid, "s", np.ascontiguousarray(v, np.float32), np.ascontiguousarray(t, np.int32))


def _sphere(r, f, c=(0, 0, 0), flip=False):
    u, t = zs.geodesic_sphere(f)
    return u * r + np.asarray(c, float), (t[:, [0, 2, 1]] if flip else t)


def _join(*parts):
    v, t, n = [], [], 0
    for pv, pt in parts:
        v.append(pv)
        t.append(np.asarray(pt) + n)
        n += len(pv)
    return np.concatenate(v), np.concatenate(t)


def _surfaces(name):
    if name == "box":            # 12 triangles, each over many cells
        return [_surf(*zs.box_surface((-1, -1, -1), (1, 2, 0.5)))]
    if name == "box_grid":       # faces in lattice planes
        return [_surf(*zs.box_surface((-4, -4, -4), (4, 4, 4), m=8))]
    if name == "tetra":
        v = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], float)
        return [_surf(v, [[0, 2, 1], [0, 1, 3], [0, 3, 2], [1, 2, 3]])]
    if name == "torus":
        return [_surf(*zs.torus(10.0, 3.0, 60, 24, seed=3, amp=0.5))]
    if name == "shell":          # a hole: winding number 0 between the inner sphere and the centre
        return [_surf(*_join(_sphere(2.0, 6), _sphere(1.0, 5, flip=True)))]
    if name == "double":         # overlapping sheets: winding number 2 in the lens
        return [_surf(*_join(_sphere(1.0, 6), _sphere(1.0, 6, c=(0.7, 0.1, 0.0))))]
    if name == "far_small":      # a small surface far from the origin
        return [_surf(*_sphere(0.5, 7, c=(300.0, -200.0, 100.0)))]
    if name == "far_fine":       # cells of a few float32 steps
        return [_surf(*_sphere(0.5, 12, c=(30000.0, -20000.0, 100.0)))]
    if name == "tiny":
        return [_surf(*_sphere(3e-5, 7, c=(1e-4, 0, 0)))]
    if name == "flat":           # one cell thick
        return [_surf(*zs.box_surface((-50, -50, -0.05), (50, 50, 0.05), m=12))]
    if name == "mixed_sizes":    # fine triangles on a corner of a coarse box, and intersecting spheres
        a = _surf(*zs.box_surface((-5, -5, -5), (5, 5, 5), m=2), cid=1)
        b = _surf(*_sphere(0.4, 12, c=(5, 5, 5)), cid=2)
        c = _surf(*_sphere(3.0, 9, c=(4, 0, 0)), cid=3)
        return [b, a, c]
    raise KeyError(name)


NAMES = ["box", "box_grid", "tetra", "torus", "shell", "double", "far_small", "far_fine", "tiny", "flat", "mixed_sizes"]


def _points(surfs, n, seed):
    rng = np.random.default_rng(seed)
    v = np.concatenate([s.verts for s in surfs]).astype(np.float64)
    lo, hi = v.min(0), v.max(0)
    ext = (hi - lo).max()
    pts = [rng.uniform(lo - 0.1 * ext, hi + 0.1 * ext, size=(n, 3))]
    for s in surfs:              # a hair off the triangles, and off their edges and vertices
        tri = s.verts[s.tris].astype(np.float64)
        t = rng.integers(0, len(tri), n)
        w = rng.dirichlet((1, 1, 1), n)
        w[: n // 4, 0] = 0.0
        w[: n // 8, 1] = 0.0
        w /= w.sum(1, keepdims=True)
        off = rng.standard_normal((n, 3)) * ext * 10.0 ** rng.uniform(-7, -1, (n, 1))
        pts.append((tri[t] * w[:, :, None]).sum(1) + off)
    m = 12                       # lattice planes through faces and vertices
    g = np.stack(np.meshgrid(*[np.linspace(lo[k], hi[k], m + 1) for k in range(3)], indexing="ij"), -1).reshape(-1, 3)
    pts.append(g)
    return np.concatenate(pts).astype(np.float32)


def _off_surface(oracle, pts, surfs, prio, oom):
    """Points whose label is well posed: the FP64 sum is 4 pi k there, and has
    the same k a hair away on every side (a lattice point in a face, on an
    edge or on a vertex has not, whatever its own sum rounds to)."""
    ok = np.all(np.abs(oom - FOUR_PI * np.round(oom / FOUR_PI)) < 1e-9, axis=0)
    v = np.concatenate([s.verts for s in surfs]).astype(np.float64)
    eps = 2e-7 * max((v.max(0) - v.min(0)).max(), np.abs(v).max())
    for d in np.stack(np.meshgrid(*[[-1.0, 1.0]] * 3, indexing="ij"), -1).reshape(-1, 3):
        _, om2 = oracle.label_points(pts.astype(np.float64) + eps * d, surfs, prio)
        ok &= np.all(np.round(om2 / FOUR_PI) == np.round(oom / FOUR_PI), axis=0)
    return ok


def _label(zef, surfs, prio, pts, **kw):
    ctx = zef.Context(0)
    for s in surfs:
        ctx.add_compartment(s.id, s.verts, s.tris)
    ctx.set_priority(prio)
    lab, om, st = ctx.label_points(torch.from_numpy(pts).cuda(), opts=zef.make_opts(**kw), want_omega=True)
    early, _, st2 = ctx.label_points(torch.from_numpy(pts).cuda(), opts=zef.make_opts(**kw))
    torch.cuda.synchronize()
    ctx.close()
    return lab.cpu().numpy(), om.cpu().numpy().astype(np.float64), early.cpu().numpy(), st, st2


@pytest.fixture(scope="module")
def zef():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10000_gb300 import zef as z
    return z


@pytest.mark.parametrize("name", NAMES)
def test_grid_labels_equal_general_kernels_and_oracle(zef, name):
    import oracle
    surfs = _surfaces(name)
    prio = [s.id for s in surfs]
    pts = _points(surfs, 3000, seed=17)
    lab, om, early, st, _ = _label(zef, surfs, prio, pts)
    glab, gom, gearly, gst, _ = _label(zef, surfs, prio, pts, block_threads=256, points_per_thread=2)
    assert st["kernel_launches"] <= 2 < gst["kernel_launches"]      # the grid path, the tile kernels
    olab, oom = oracle.label_points(pts, surfs, prio)
    off = _off_surface(oracle, pts, surfs, prio, oom)
    assert off.sum() > (0.1 if name == "far_fine" else 0.6) * len(pts)
    for kind, got in (("grid", lab), ("grid, early exit", early), ("general", glab), ("general, early exit", gearly)):
        bad = off & (got != olab)
        assert not bad.any(), (kind, int(bad.sum()), pts[bad][:3], got[bad][:3], olab[bad][:3])
    # a certified value is 4 pi k in float32, an FP64 sum its rounding
    assert np.abs(om - oom)[:, off].max() <= 1e-6
    assert np.abs(gom - oom)[:, off].max() <= 1e-6


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 511, 512, 513, 4097])
def test_grid_point_counts(zef, n):
    import oracle
    surfs = _surfaces("mixed_sizes")
    prio = [1, 3, 2]
    pts = _points(surfs, 2000, seed=n)
    pts = pts[np.random.default_rng(n).permutation(len(pts))[:n]]
    if n > 2:
        pts[n // 2] = [np.nan, 0, 0]
        pts[n // 3] = [0, np.inf, 0]
    lab, om, early, st, _ = _label(zef, surfs, prio, pts)
    olab, oom = oracle.label_points(pts, surfs, prio)
    fin = np.isfinite(pts).all(1)
    ok = ~fin
    ok[fin] = _off_surface(oracle, pts[fin], surfs, prio, oom[:, fin])
    assert np.array_equal(lab[ok], olab[ok]) and np.array_equal(early[ok], olab[ok])
    assert np.isnan(om[:, ~fin]).all() and np.isfinite(om[:, fin]).all()
    assert st["nonfinite_points"] == int((~fin).sum()) and st["points"] == n


def test_grid_registration_order_and_priority(zef):
    """The surfaces' common scale changes as larger ones are registered, the
    priority after it: the labels are those of the final set."""
    import oracle
    small, big = _surf(*_sphere(1.0, 8), cid=7), _surf(*_sphere(900.0, 8), cid=2)
    pts = np.concatenate([_points([small], 1500, 3), _points([big], 1500, 4)])
    for order in ([small, big], [big, small]):
        for prio in ([7, 2], [2, 7]):
            lab, _, early, _, _ = _label(zef, order, prio, pts)
            olab, oom = oracle.label_points(pts, order, prio)
            ok = _off_surface(oracle, pts, order, prio, oom)
            assert np.array_equal(lab[ok], olab[ok]) and np.array_equal(early[ok], olab[ok])


def test_surface_without_a_grid_takes_the_general_kernels(zef):
    """Most of the triangles in one corner of a wide surface: its cells would
    list them all, so the surface gets no grid and labels stay exact."""
    import oracle
    surfs = [_surf(*_join(_sphere(100.0, 2), _sphere(0.01, 24, c=(3, 2, 1)), _sphere(0.02, 24, c=(-3, 2, 1))))]
    pts = _points(surfs, 2000, seed=5)
    lab, om, early, st, _ = _label(zef, surfs, [1], pts)
    assert st["kernel_launches"] > 2
    olab, oom = oracle.label_points(pts, surfs, [1])
    ok = _off_surface(oracle, pts, surfs, [1], oom)
    assert np.array_equal(lab[ok], olab[ok]) and np.array_equal(early[ok], olab[ok])
