"""Neighbour rows of the post-processing, and the boundary faces of its
surface variant, on meshes whose tets are in random
order (an edge in many runs of tets), in runs of every remainder, with a node
of several hundred neighbours (rows longer than the staged ones) and with
repeated nodes: one smoothing step against the FP64 oracle, which builds its
neighbourhoods from sets; boundary smoothing of labelings that make every
node, or hardly any, a boundary node."""
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


def _meshes():
    nodes, tets = zs.lattice_5tet(11, 1.0, (0.0, 0.0, 0.0))
    rng = np.random.default_rng(5)
    yield "lattice", nodes, tets
    yield "shuffled", nodes, tets[rng.permutation(len(tets))]
    for k in (1, 255, 256, 257, 513):
        yield f"{k} tets", nodes, tets[rng.permutation(len(tets))[:k]]
    # a fan: node 0 joined to hundreds of others (any tets will do for the rows)
    pts = rng.standard_normal((700, 3)).astype(np.float32)
    fan = np.stack([np.zeros(900, np.int32), *[rng.integers(1, 700, 900).astype(np.int32) for _ in range(3)]], 1)
    yield "fan", pts, fan                      # some with a repeated node
    order = rng.permutation(len(nodes)).astype(np.int32)
    yield "renumbered", nodes[np.argsort(order)], order[tets]


@pytest.mark.parametrize("name,nodes,tets", list(_meshes()), ids=lambda v: v if isinstance(v, str) else "")
def test_rows_by_one_smoothing_step(zef, name, nodes, tets):
    rng = np.random.default_rng(9)
    x = (nodes + 0.1 * rng.standard_normal(nodes.shape)).astype(np.float32)
    ctx = zef.Context(0)
    got = torch.from_numpy(x.copy()).cuda()
    assert ctx.taubin_smooth(got, torch.from_numpy(np.ascontiguousarray(tets)).cuda(), 0.4, 0.4, 0.0, 1) == 1
    ctx.close()
    nbr = [set() for _ in range(len(x))]
    for t in tets:
        for a in t:
            nbr[a].update(int(b) for b in t if b != a)
    p = x.astype(np.float64)
    for w in (np.float64(np.float32(0.4)), -np.float64(np.float32(0.4))):
        p = np.stack([p[i] + w / (len(s) + 1) * (p[sorted(s)] - p[i]).sum(0) if s else p[i] for i, s in enumerate(nbr)])
    # a row of d float32 differences summed in order: d 2^-24 of their size each way
    d = max(len(s) for s in nbr)
    assert np.abs(got.cpu().numpy() - p).max() <= 2 * (d + 8) * 2.0 ** -24 * 2 * np.abs(x).max()


@pytest.mark.parametrize("kind", ["random", "extremes", "one tet", "halves", "one label"])
def test_boundary_faces_and_rows(zef, kind):
    from oracle import postprocess as pp
    nodes, tets = zs.lattice_5tet(7, 1.0, (0.0, 0.0, 0.0))
    rng = np.random.default_rng(3)
    tets = tets[rng.permutation(len(tets))]
    lab = {"random": rng.integers(-1, 4, len(tets)),
           "extremes": rng.choice([-2 ** 31, 2 ** 31 - 1], len(tets)),
           "one tet": (np.arange(len(tets)) == 77) * 5,
           "halves": (nodes[tets].mean(1)[:, 0] > 3.3) * 9 - 4,
           "one label": np.full(len(tets), 6)}[kind].astype(np.int32)
    x = (nodes + 0.1 * rng.standard_normal(nodes.shape)).astype(np.float32)
    ctx = zef.Context(0)
    got = torch.from_numpy(x.copy()).cuda()
    it, faces = ctx.taubin_smooth_surface(got, torch.from_numpy(np.ascontiguousarray(tets)).cuda(),
                                          torch.from_numpy(lab).cuda(), 0.4, 0.4, 0.0, 3)
    ctx.close()
    want, oit, ofaces = pp.taubin_smooth_surface(x, tets, lab, 0.4, 0.4, 0.0, 3)
    assert (it, faces) == (oit, ofaces)
    # 2 k half-steps of about 2^-20 of the largest coordinate each
    assert np.abs(got.cpu().numpy() - want).max() <= 2 * 3 * 2.0 ** -20 * np.abs(x).max()


@pytest.mark.parametrize("cells,freq", [(3, 24), (9, 24), (24, 6), (17, 2)])
def test_inflation_by_cells_and_by_tree(zef, cells, freq):
    """Edges from a tenth of a grid cell to longer than thousands of cells
    (left to the cap tree) against the oracle's test of every triangle."""
    from oracle import postprocess as pp
    u, t = zs.geodesic_sphere(freq)
    surf = zs.Surface(1, "s", (u * [1.0, 0.8, 0.9]).astype(np.float32), t.astype(np.int32))
    nodes, tets = zs.lattice_5tet(cells, 2.4 / cells, (-1.21, -1.19, -1.2))
    ctx = zef.Context(0)
    ctx.add_compartment(1, surf.verts, surf.tris)
    got = torch.from_numpy(nodes.copy()).cuda()
    moved = ctx.inflate(got, torch.from_numpy(tets).cuda(), 1, 0.1)
    ctx.close()
    want, omoved = pp.inflate(nodes, tets, surf, 0.1)
    assert moved == omoved and moved > 0
    assert np.abs(got.cpu().numpy() - want).max() <= 1e-6 * np.abs(nodes).max()
