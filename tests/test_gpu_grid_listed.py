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
