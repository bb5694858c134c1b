"""The stopping rule of the smoothing loops on meshes with a coordinate that is
not finite: the iterations that the rule, as the oracle applies it, runs."""
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


def _mesh():
    nodes, tets = zs.lattice_5tet(5, 1.0, (1.0, 1.0, 1.0))
    rng = np.random.default_rng(2)
    x = (nodes + 0.1 * rng.standard_normal(nodes.shape)).astype(np.float32)
    return np.concatenate([x, np.full((1, 3), 2.0, np.float32)]), np.ascontiguousarray(tets)  # the last: in no tet


# an infinite coordinate makes every ratio of norms not a number, which is not
# below xi: the loop runs to its limit, whether the node has neighbours or not
@pytest.mark.parametrize("xi", [0.0, 0.5])
@pytest.mark.parametrize("node", [-1, 7])
@pytest.mark.parametrize("held", [False, True])
def test_an_infinite_coordinate_does_not_end_the_loop(zef, xi, node, held):
    from oracle import postprocess as pp
    x, tets = _mesh()
    x[node, 1] = np.inf
    fixed = np.zeros(len(x), np.uint8)
    fixed[node] = held
    with np.errstate(invalid="ignore"):
        _, want = pp.taubin_smooth(x, tets, 0.4, 0.4, xi, 6, fixed=fixed)
    assert want == 6
    ctx = zef.Context(0)
    got = ctx.taubin_smooth(torch.from_numpy(x).cuda(), torch.from_numpy(tets).cuda(), 0.4, 0.4, xi, 6,
                            fixed=torch.from_numpy(fixed).cuda())
    ctx.close()
    assert got == want


# the norms of the boundary variant run over the boundary's nodes alone: a node
# off it has no say (xi = 0: everything is still at the first iteration)
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("xi,lam", [(0.5, 0.4), (0.0, 0.0)])
def test_a_node_off_the_boundary_has_no_say(zef, xi, lam, value):
    from oracle import postprocess as pp
    x, tets = _mesh()
    lab = (x[tets].mean(1)[:, 0] > 3.3).astype(np.int32)
    x[-1, 2] = value
    with np.errstate(invalid="ignore"):
        _, want, faces = pp.taubin_smooth_surface(x, tets, lab, lam, lam, xi, 6)
    assert want == 1 and faces > 0
    ctx = zef.Context(0)
    got = ctx.taubin_smooth_surface(torch.from_numpy(x).cuda(), torch.from_numpy(tets).cuda(),
                                    torch.from_numpy(lab).cuda(), lam, lam, xi, 6)
    ctx.close()
    assert got == (want, faces)
