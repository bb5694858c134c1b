"""The debug build (ZEF_DEBUG_BOUNDS) on every form of the default path: small
and listed calls, with and without solid angles, points on surfaces (in the
list, beyond it, in place), up to 40 surfaces.  No check may fail, and the
labels equal the release build's."""
import os
import subprocess
import sys

import numpy as np
import pytest

import zef_synth as zs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def spheres(count):
    v, t = zs.geodesic_sphere(5)
    rng = np.random.default_rng(count)
    return [zs.Surface(k + 1, "s", (v * rng.uniform(0.3, 1.0) + rng.uniform(-3, 3, 3)).astype(np.float32), t)
            for k in range(count)]


def points(surfs, n, share):
    rng = np.random.default_rng(n)
    on = np.concatenate([s.verts for s in surfs])
    p = rng.uniform(-4, 4, (n, 3)).astype(np.float32)
    k = rng.random(n) < share
    p[k] = on[rng.integers(0, len(on), int(k.sum()))]
    return p


CASES = [(count, n, share) for count in (3, 40) for n, share in ((1, 1.0), (3000, 0.1), (262_144, 0.001), (262_144, 0.3))]

CHILD = r'''
import sys
import numpy as np
import torch
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import test_gpu_debug_grid as t
from paper_2203_10000_gb300 import zef
assert zef.LIB_PATH.endswith("_build_debug/libzef.so"), zef.LIB_PATH
np.savez(sys.argv[2], **{str(k): v for k, v in enumerate(t.run(zef))})
print("debug build ok")
'''


def run(zef):
    out = []
    for count, n, share in CASES:
        surfs = spheres(count)
        ctx = zef.Context(0)
        for s in surfs:
            ctx.add_compartment(s.id, s.verts, s.tris)
        pts = torch.from_numpy(points(surfs, n, share)).cuda()
        lab, om, _ = ctx.label_points(pts, want_omega=True)
        early, _, _ = ctx.label_points(pts, stats=False)
        ctx.synchronize()                       # raises on ZEF_ERR_BOUNDS
        assert torch.equal(lab, early), (count, n, share)
        out += [lab.cpu().numpy(), om.cpu().numpy()]
        ctx.close()
    return out


def test_debug_build_on_every_form_of_the_default_path(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10000_gb300 import build
    lib = build.build(debug=True)
    build.build()
    from paper_2203_10000_gb300 import zef
    f = str(tmp_path / "out.npz")
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, f], env=dict(os.environ, ZEF_LIBRARY=lib),
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "debug build ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
    got = np.load(f)
    for k, want in enumerate(run(zef)):
        assert np.array_equal(got[str(k)].view(np.uint32), want.view(np.uint32)), CASES[k // 2]
