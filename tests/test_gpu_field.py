"""The label field over surfaces whose own cells are far finer than its own:
the time to rebuild it (with a priority order), and labels from it."""
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


def test_a_fine_surface_in_a_wide_one(zef):
    """A sphere of 450,000 triangles in one fifty times as wide: a cell of the
    field holds some 50,000 of its own.  A new order rebuilds the field; one
    thread for all cells of a field cell took 17 ms, the warp together 4: the
    limit lies between."""
    v, t = zs.geodesic_sphere(150)
    u, s = zs.geodesic_sphere(8)
    at = np.array([10.0, 5.0, 3.0])
    ctx = zef.Context(0)
    ctx.add_compartment(1, (2.0 * v + at).astype(np.float32), t)
    ctx.add_compartment(2, (100.0 * u).astype(np.float32), s)
    times = []
    for k in range(7):
        t0 = time.perf_counter()
        ctx.set_priority([2, 1] if k % 2 == 0 else [1, 2])
        ctx.synchronize()
        times.append(time.perf_counter() - t0)
    ctx.set_priority([1, 2])
    rng = np.random.default_rng(0)
    pts = np.concatenate([rng.uniform(-3, 3, (100_000, 3)) + at, rng.uniform(-110, 110, (100_000, 3))]).astype(np.float32)
    p = torch.from_numpy(pts).cuda()
    lab, om, _ = ctx.label_points(p, want_omega=True)
    glab, gom, _ = ctx.label_points(p, want_omega=True, opts=zef.make_opts(block_threads=256, points_per_thread=2))
    ctx.synchronize()
    ctx.close()
    assert torch.equal(lab, glab) and float((om - gom).abs().max()) <= 1e-6
    assert len(torch.unique(lab)) == 3
    assert min(times) < 9e-3, times
