"""The cell grid's calls that other tests' sizes leave out: point counts around
the limit from which the open points are listed, sets of more than 32
surfaces, and the statistics of its calls."""
import numpy as np
import pytest

import zef_synth as zs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LISTED = 1 << 18  # points from which on a call lists the open ones


@pytest.fixture(scope="module")
def zef():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10000_gb300 import zef as z
    return z


def _context(zef, surfs, prio=None):
    ctx = zef.Context(0)
    for s in surfs:
        ctx.add_compartment(s.id, s.verts, s.tris)
    if prio:
        ctx.set_priority(prio)
    return ctx


@pytest.mark.parametrize("n", [5000, LISTED])
def test_evaluated_pairs_are_those_of_the_cells_triangles(zef, n):
    """A tetrahedron's cells list four triangles at most: no point can have
    been compared with more, however its cell's list is padded."""
    v = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], np.float32)
    ctx = _context(zef, [zs.Surface(1, "t", v, np.array([[0, 2, 1], [0, 1, 3], [0, 3, 2], [1, 2, 3]], np.int32))])
    rng = np.random.default_rng(n)
    p = rng.dirichlet((1, 1, 1), n) @ v[1:].astype(np.float64)       # on the slanted face, and a hair off it
    p += 1e-3 * rng.standard_normal((n, 3))
    _, _, st = ctx.label_points(torch.from_numpy(p.astype(np.float32)).cuda())
    ctx.close()
    first = st["pairs_evaluated"] - st["pairs_rescued"]
    assert 0.9 * n < first <= 4 * n
    assert st["pairs_nominal"] == 4 * n


def _equal_general(zef, ctx, pts):
    """Labels, early and full, and solid angles of the default path against the
    general kernels'."""
    p = torch.from_numpy(pts).cuda()
    lab, om, st = ctx.label_points(p, want_omega=True)
    early, _, _ = ctx.label_points(p, stats=False)
    opts = zef.make_opts(block_threads=256, points_per_thread=2)
    glab, gom, gst = ctx.label_points(p, want_omega=True, opts=opts)
    ctx.synchronize()
    assert torch.equal(lab, glab) and torch.equal(early, glab)
    assert torch.equal(om.isnan(), gom.isnan())
    # a certified value is 4 pi k in float32, an FP64 sum its rounding
    assert float((om - gom).nan_to_num().abs().max()) <= 1e-6
    assert st["nonfinite_points"] == gst["nonfinite_points"] and st["points"] == len(pts)
    return lab.cpu().numpy(), st


# a warp of the streaming kernel takes 128 points at a time, lists 256 together
@pytest.mark.parametrize("n", [LISTED - 1, LISTED, LISTED + 1, LISTED + 127, LISTED + 128, LISTED + 129, LISTED + 32 * 128 + 1])
def test_calls_around_the_listed_size(zef, n):
    w = zs.config1(npts_limit=0)
    ctx = _context(zef, w.surfaces, w.priority)
    rng = np.random.default_rng(n)
    v = np.concatenate([s.verts for s in w.surfaces])
    pts = rng.uniform(v.min(0) * 1.1, v.max(0) * 1.1, (n, 3)).astype(np.float32)
    # a stretch where every point is open, at the end too, and points not finite
    near = v[rng.integers(0, len(v), 3000)] + rng.normal(0, 0.3, (3000, 3)).astype(np.float32)
    pts[1000:3500] = near[:2500]
    pts[-500:] = near[2500:]
    bad = np.concatenate([rng.integers(0, n, 300), [0, n - 1]])
    pts[bad, rng.integers(0, 3, len(bad))] = rng.choice([np.nan, np.inf, -np.inf], len(bad))
    lab, st = _equal_general(zef, ctx, pts)
    ctx.close()
    assert np.array_equal(lab == -1, ~np.isfinite(pts).all(1))
    assert st["kernel_launches"] == (2 if n < LISTED else 4)


def _spheres(count):
    v, t = zs.geodesic_sphere(6)
    rng = np.random.default_rng(count)
    return [zs.Surface(k + 1, "s", (v * rng.uniform(0.4, 1.5) + rng.uniform(-3, 3, 3)).astype(np.float32), t)
            for k in range(count)]


# up to 32 surfaces a cell of the label field is two 32-bit words, then two of 64
@pytest.mark.parametrize("count", [32, 33, 64])
@pytest.mark.parametrize("n", [1000, 65_000, LISTED + 77])
def test_many_surfaces(zef, count, n):
    surfs = _spheres(count)
    prio = [s.id for s in surfs[::-1]]
    ctx = _context(zef, surfs, prio)
    rng = np.random.default_rng(n)
    v = np.concatenate([s.verts for s in surfs])
    pts = rng.uniform(v.min(0), v.max(0), (n, 3)).astype(np.float32)
    lab, _ = _equal_general(zef, ctx, pts)
    assert len(np.unique(lab)) > count // 2 or n < 10_000
    # the four-nodes rule takes every row's bit of every node
    tets = torch.from_numpy(rng.integers(0, min(n, 500), (4000, 4)).astype(np.int32)).cuda()
    nodes = torch.from_numpy(pts).cuda()
    el, _, _ = ctx.label_elements(nodes, tets, stats=False)
    gel, _, _ = ctx.label_elements(nodes, tets, opts=zef.make_opts(block_threads=256, points_per_thread=2), stats=False)
    ctx.synchronize()
    assert torch.equal(el, gel)
    ctx.close()


@pytest.mark.parametrize("n", [1000, LISTED])
def test_statistics_say_which_path_served_the_call(zef, n):
    w = zs.config0()
    ctx = _context(zef, w.surfaces)
    pts = torch.rand((n, 3), device="cuda")
    assert ctx.label_points(pts)[2]["cell_grids"] == 1
    assert ctx.label_points(pts, opts=zef.make_opts(block_threads=256, points_per_thread=2))[2]["cell_grids"] == 0
    ctx.close()


@pytest.mark.parametrize("n", [100, 5000, 100_000, LISTED])
def test_work_items_do_not_depend_on_the_split(zef, n):
    """Of 64 points of the surfaces' box each, however few a warp was given."""
    w = zs.config0()
    ctx = _context(zef, w.surfaces)
    v = w.surfaces[0].verts
    pts = np.random.default_rng(n).uniform(v.min(0) * 1.2, v.max(0) * 1.2, (n, 3)).astype(np.float32)
    inside = int(((pts >= v.min(0)) & (pts <= v.max(0))).all(1).sum())
    st = ctx.label_points(torch.from_numpy(pts).cuda())[2]
    ctx.close()
    assert st["work_items"] == st["tiles"] == (inside + 63) // 64
