"""Nodes joined to more neighbours than a warp stages in shared memory: their
rows against sets on the host, at the edges of the sort's runs, and the time
of one whose edges come again and again from tets in random order."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def zef():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_10000_gb300 import zef as z
    return z


def _fan(d, m, seed):
    """Node 0 joined to d others by m tets in random order, every other node used."""
    rng = np.random.default_rng(seed)
    rim = np.concatenate([rng.permutation(d), rng.integers(0, d, 3 * m - d)]) + 1
    tets = np.concatenate([np.zeros((m, 1), np.int64), rng.permutation(rim).reshape(m, 3)], 1).astype(np.int32)
    return rng.standard_normal((d + 1, 3)).astype(np.float32), tets


# entries of the row before its repeats go (three per tet): around the longest
# row placed by counting (768), one run of the sort (1,024), two and several
@pytest.mark.parametrize("d,m", [(700, 256), (768, 256), (769, 257), (1022, 341), (1024, 342), (1026, 342),
                                 (2047, 683), (2049, 683), (300, 1400), (5000, 9001)])
def test_long_rows_by_one_smoothing_step(zef, d, m):
    x, tets = _fan(d, m, seed=d + m)
    ctx = zef.Context(0)
    got = torch.from_numpy(x.copy()).cuda()
    assert ctx.taubin_smooth(got, torch.from_numpy(tets).cuda(), 0.4, 0.4, 0.0, 1) == 1
    ctx.close()
    nbr = [set() for _ in range(len(x))]
    for t in tets:
        for a in t:
            nbr[a].update(int(b) for b in t if b != a)
    assert len(nbr[0]) == d
    p = x.astype(np.float64)
    for w in (np.float64(np.float32(0.4)), -np.float64(np.float32(0.4))):
        p = np.stack([p[i] + w / (len(s) + 1) * (p[sorted(s)] - p[i]).sum(0) if s else p[i] for i, s in enumerate(nbr)])
    # a row of k float32 differences summed in order: k 2^-24 of their size each way
    k = max(len(s) for s in nbr)
    assert np.abs(got.cpu().numpy() - p).max() <= 2 * (k + 8) * 2.0 ** -24 * 2 * np.abs(x).max()


def test_a_node_of_many_neighbours_takes_no_square_time(zef):
    """1,024 neighbours in 5,120 tets.  One lane that inserts them without
    repeats takes d^2 / 4 dependent steps of about 100 ns, 26 ms; four times
    that is the limit (with the repeats it took 1.26 s)."""
    x, tets = _fan(1024, 5120, seed=1)
    ctx = zef.Context(0)
    got, t = torch.from_numpy(x).cuda(), torch.from_numpy(tets).cuda()
    times = []
    for _ in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx.taubin_smooth(got, t, 0.4, 0.4, 0.0, 1)
        times.append(time.perf_counter() - t0)
    ctx.close()
    assert min(times) < 4 * 0.026, times
