"""Points on a surface, whose pairs neither the FP32 nor the FP64 crossings
decide (electrodes are vertices of the scalp mesh): the FP64 solid angle of
each, whatever the number of such points and wherever they stand in the call,
equal to the general kernels' bit for bit, and no slower."""
import time

import numpy as np
import pytest

import zef_synth as zs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def zef():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10000_gb300 import zef as z
    return z


def _context(zef, surfs, prio):
    ctx = zef.Context(0)
    for s in surfs:
        ctx.add_compartment(s.id, s.verts, s.tris)
    ctx.set_priority(prio)
    return ctx


def _spheres():
    """Two spheres with a common octant of vertices, one bump apart elsewhere."""
    v, t = zs.geodesic_sphere(10)
    b = v * np.where(v.min(1, keepdims=True) >= 0, 1.0, 1.0 + 0.1 * np.abs(v[:, :1]))
    return [zs.Surface(1, "a", v.astype(np.float32), t), zs.Surface(2, "b", b.astype(np.float32), t)]


def _call(ctx, pts, **kw):
    lab, om, st = ctx.label_points(torch.from_numpy(np.ascontiguousarray(pts)).cuda(), want_omega=True, **kw)
    early, _, _ = ctx.label_points(torch.from_numpy(np.ascontiguousarray(pts)).cuda(), **kw)
    ctx.synchronize()
    return lab.cpu().numpy(), om.cpu().numpy(), early.cpu().numpy(), st


# a warp's share is 8 points at least; one kernel below 2^18 points, from there
# on a list of 32,768 such points, and what it does not hold once more
@pytest.mark.parametrize("n,share", [(n, 0.875) for n in (1, 7, 8, 9, 64, 65, 1000, 2432, 2433, 40_000, 160_001, 262_143)] +
                         [(262_144, 0.0), (262_144, 1e-5), (262_145, 0.02), (300_001, 0.1), (262_144, 0.13), (262_144, 0.875)])
def test_points_on_surfaces_equal_the_general_kernels(zef, oracle_mod, n, share):
    surfs = _spheres()
    ctx = _context(zef, surfs, [2, 1])
    on = np.unique(np.concatenate([s.verts for s in surfs]), axis=0)
    rng = np.random.default_rng(n)
    pts = on[rng.integers(0, len(on), n)]
    off = rng.random(n) >= share
    pts[off] *= rng.choice([0.5, 0.9, 1.3], off.sum())[:, None].astype(np.float32)
    lab, om, early, st = _call(ctx, pts)
    assert np.array_equal(lab, early)
    # the general kernels sum a pair whole where more than 1,024 are uncertain
    every = np.concatenate([on, on])
    assert 2 * len(on) > 1024
    opts = zef.make_opts(block_threads=256, points_per_thread=2)
    glab, gom, _, gst = _call(ctx, every, opts=opts)
    assert gst["uncertain_pairs"] > 1024
    at = {p.tobytes(): k for k, p in enumerate(every)}
    k = np.array([at[p.tobytes()] for p in pts[~off]], dtype=np.int64)
    assert np.array_equal(lab[~off], glab[k])
    assert np.array_equal(om[:, ~off].view(np.uint32), gom[:, k].view(np.uint32))
    if n <= 1000:
        # (on a vertex the oracle has no value of its own: its triangles there
        # are taken as they round)
        olab, oom = oracle_mod.label_points(pts, surfs, [2, 1])
        assert np.array_equal(lab[off], olab[off])
        assert np.abs(om - oom)[:, off].max(initial=0.0) <= 1e-6   # float32 of a value up to 4 pi: 4.8e-7
    ctx.close()


def _time(ctx, pts, opts):
    lab = torch.empty(pts.shape[0], dtype=torch.int32, device="cuda")
    best = float("inf")
    for rep in range(8):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx.label_points(pts, labels=lab, opts=opts, stats=False)
        ctx.synchronize()
        if rep >= 2:
            best = min(best, time.perf_counter() - t0)
    return best


@pytest.mark.parametrize("n,on", [(64, 64), (4096, 4096), (300_000, 64), (300_000, 4096)])
def test_points_on_a_surface_are_no_slower_than_the_general_kernels(zef, n, on):
    """`on` consecutive points are vertices of the scalp, the others in its box."""
    w = zs.config1(npts_limit=0)
    ctx = _context(zef, w.surfaces, w.priority)
    scalp = max(w.surfaces, key=lambda s: float(np.ptp(s.verts, axis=0).max()))
    rng = np.random.default_rng(n)
    pts = rng.uniform(scalp.verts.min(0), scalp.verts.max(0), (n, 3)).astype(np.float32)
    pts[n // 2 - on // 2: n // 2 + on - on // 2] = scalp.verts[rng.permutation(len(scalp.verts))[:on]]
    pts = torch.from_numpy(pts).cuda()
    grid = _time(ctx, pts, zef.make_opts())
    general = _time(ctx, pts, zef.make_opts(block_threads=256, points_per_thread=2))
    ctx.close()
    assert grid <= general, (n, on, grid, general)


@pytest.mark.parametrize("n", [40_000, 270_000])
def test_a_captured_call_decides_other_points_on_replay(zef, n):
    """The call's kernels in a graph of the caller's (they leave their lists
    empty): replays on other points, the last on none on a surface, and plain
    calls in between."""
    surfs = _spheres()
    on = np.unique(np.concatenate([s.verts for s in surfs]), axis=0)
    rng = np.random.default_rng(n)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = _context(zef, surfs, [2, 1])
        pts = torch.zeros((n, 3), device="cuda")
        lab = torch.empty(n, dtype=torch.int32, device="cuda")
        ctx.label_points(pts, labels=lab, stats=False)
        graph = torch.cuda.CUDAGraph()
        stream.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            ctx.label_points(pts, labels=lab, stats=False)
        for share in (0.05, 0.001, 0.5, 0.0):
            p = on[rng.integers(0, len(on), n)] * np.where(rng.random(n) < share, 1.0, 0.9).astype(np.float32)[:, None]
            want = torch.from_numpy(np.ascontiguousarray(p)).cuda()
            plain, _, _ = ctx.label_points(want, stats=False)
            pts.copy_(want)
            lab.fill_(-7)
            graph.replay()
            stream.synchronize()
            assert torch.equal(lab, plain), share
        ctx.close()
