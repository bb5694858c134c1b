"""Workloads of the labeling library, as a program calls it.

Each case is one call (or, for the in-place entry points, one call on a fresh
copy of its arrays) through paper_2203_10000_gb300.zef: point labeling from
the smallest host batch to the 56 M-point head, element labels, refinement,
boundary re-labeling and the post-processing of a refined mesh.  The surfaces
are zef_synth's (three-layer head, the head with 8 deep structures, 20 deep
structures, the full 24-compartment head, unit spheres); a seed turns, scales
and shifts them as one body and moves the points, so every seed is another
subject in the scanner.
"""
from __future__ import annotations

import ctypes
import functools
import math

import numpy as np
import torch

import zef_synth as zs
from paper_2203_10000_gb300 import zef

DEV = "cuda"
FOUR_PI = 4.0 * math.pi


# ---------------------------------------------------------------- surfaces
@functools.lru_cache(maxsize=None)
def _base(name: str, freq: int = 8):
    """[(id, vertices float64, triangles)], priority, half extent of the lattice."""
    if name == "sphere":
        v, t = zs.geodesic_sphere(freq)
        return [(1, v, t)], [1], 1.5
    w = {"head": lambda: zs.config1(npts_limit=0), "head8": zs.config3,
         "deep": lambda: zs.config2(npts_limit=0),
         "full": lambda: zs.config4(with_points=False)}[name]()
    half = {"head": 100.0, "head8": 100.0, "deep": 80.0, "full": 112.0}[name]
    return [(s.id, s.verts.astype(np.float64), s.tris) for s in w.surfaces], list(w.priority), half


def _surfaces(case, seed: int):
    """The case's surfaces in the pose of this seed, outward oriented."""
    surfs, prio, half = _base(case["surfaces"], case.get("freq", 8))
    rng = np.random.default_rng([seed, 101])
    ax = rng.standard_normal(3)
    ax /= np.linalg.norm(ax)
    ang = rng.uniform(-0.1, 0.1)
    K = np.array([[0, -ax[2], ax[1]], [ax[2], 0, -ax[0]], [-ax[1], ax[0], 0]])
    R = np.eye(3) + math.sin(ang) * K + (1 - math.cos(ang)) * (K @ K)
    R *= rng.uniform(0.96, 1.0)
    shift = rng.uniform(-0.01, 0.01, size=3) * half
    return [(i, (v @ R.T + shift).astype(np.float32), t) for i, v, t in surfs], prio, half


def _context(case, seed: int):
    surfs, prio, half = _surfaces(case, seed)
    ctx = zef.Context(0)
    for cid, v, t in surfs:
        ctx.add_compartment(cid, v, t)
    ctx.set_priority(prio)
    return ctx, half


# ---------------------------------------------------------------- points and meshes
_OFF = [[c & 1, (c >> 1) & 1, (c >> 2) & 1] for c in range(8)]


def _cells(n: int, k0: int, k1: int):
    """Integer cell coordinates (x fastest) of the layers [k0, k1)."""
    z, y, x = torch.meshgrid(torch.arange(k0, k1, device=DEV), torch.arange(n, device=DEV),
                             torch.arange(n, device=DEV), indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)


def _lattice_origin(n: int, half: float, seed: int):
    h = 2.0 * half / n
    j = np.random.default_rng([seed, 202]).integers(-8, 9, size=3) / 64.0
    return h, torch.tensor(-half + h * j, dtype=torch.float64, device=DEV)


def _centroids(n: int, half: float, seed: int):
    """Tet centroids of the five-tet split of an n^3 lattice, lattice order."""
    h, org = _lattice_origin(n, half, seed)
    off = torch.tensor(_OFF, dtype=torch.float64, device=DEV)
    tabs = [off[torch.tensor(t, device=DEV)].mean(1) for t in (zs._EVEN_O, zs._ODD_O)]
    out = torch.empty((n ** 3 * 5, 3), dtype=torch.float32, device=DEV)
    for k in range(0, n, 16):
        c = _cells(n, k, min(n, k + 16))
        sub = torch.where((c.sum(1) & 1)[:, None, None] == 0, tabs[0][None], tabs[1][None])
        s = k * n * n * 5
        out[s:s + 5 * c.shape[0]] = (org + h * (c[:, None, :].double() + sub)).reshape(-1, 3).float()
    return out


def _lattice(n: int, half: float, seed: int):
    """Nodes and five-tet tetrahedra of an n^3 lattice."""
    h, org = _lattice_origin(n, half, seed)
    nodes = (org + h * _cells(n + 1, 0, n + 1).double()).float()
    c = _cells(n, 0, n)
    off = torch.tensor(_OFF, device=DEV)
    q = c[:, None, :] + off[None]
    corner = (q[..., 2] * (n + 1) + q[..., 1]) * (n + 1) + q[..., 0]
    even = torch.tensor(zs._EVEN_O, device=DEV)
    odd = torch.tensor(zs._ODD_O, device=DEV)
    tets = torch.where((c.sum(1) & 1)[:, None, None] == 0, corner[:, even], corner[:, odd])
    return nodes.contiguous(), tets.reshape(-1, 4).to(torch.int32).contiguous()


def _flagged(case):
    """Tets split over the levels of a refinement (the boundary grows by
    about four per level; 98,238 at the first level of a 4 mm lattice)."""
    f1 = 98_238 * (case["cells"] / 50.0) ** 2
    return f1 * sum(4.15 ** k for k in range(case["levels"]))


def _capacity(case):
    n0, m0 = (case["cells"] + 1) ** 3, 5 * case["cells"] ** 3
    f = _flagged(case) * (2.2 if case.get("conforming") else 1.3) + 1000
    return int(n0 + 2.0 * f), int(m0 + 8.0 * f)


def _refined(ctx, case, half, seed):
    """A mesh as refinement leaves it: nodes, tets."""
    nodes, tets = _lattice(case["cells"], half, seed)
    if not case["levels"]:
        return nodes, tets
    cn, cm = _capacity(case)
    bn = torch.zeros((cn, 3), device=DEV)
    bt = torch.zeros((cm, 4), dtype=torch.int32, device=DEV)
    bl = torch.zeros(cn, dtype=torch.int32, device=DEV)
    bn[:nodes.shape[0]] = nodes
    bt[:tets.shape[0]] = tets
    n1, m1, _ = ctx.refine_and_relabel(bn, bt, bl, nodes.shape[0], tets.shape[0], case["levels"])
    return bn[:n1].clone(), bt[:m1].clone()


def _gen(seed: int, stream: int):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 16 + stream)
    return g


def _uniform_points(n: int, half: float, seed: int):
    return (torch.rand((n, 3), generator=_gen(seed, 1), device=DEV) * 2.0 - 1.0) * half


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # a probe placement or a few electrode positions checked from host
        # code: one small numpy batch, latency counts
        {"name": "host_small", "kind": "host", "surfaces": "sphere", "freq": 8, "points": 4099},
        # a latency-critical loop that may not allocate: the allocation-free
        # entry point with solid angles, the unit sphere of the tests
        {"name": "noalloc_omega", "kind": "noalloc", "surfaces": "sphere", "freq": 8, "points": 36_864,
         "omega": True},
        # dipole positions drawn at random in the head, in no order, with the
        # solid angle of every compartment
        {"name": "scatter_omega", "kind": "scatter", "surfaces": "head", "points": 1_000_003, "omega": True},
        # initial labeling of a 2 mm mesh of the three-layer head
        {"name": "head_2mm", "kind": "lattice", "surfaces": "head", "cells": 100},
        # 20 uneven deep structures on a 1 mm lattice
        {"name": "deep_1mm", "kind": "lattice", "surfaces": "deep", "cells": 160},
        # the full 24-compartment head on a 1 mm lattice (the headline size)
        {"name": "full_head_1mm", "kind": "lattice", "surfaces": "full", "cells": 224},
        # element labels by the four-nodes rule on a 2 mm lattice
        {"name": "elements_2mm", "kind": "elements", "surfaces": "head8", "cells": 100},
        # recursive refinement of a 4 mm lattice, three levels
        {"name": "refine_3", "kind": "refine", "surfaces": "head8", "cells": 50, "levels": 3,
         "conforming": False},
        # labels repaired after the nodes moved by up to 0.4 of a lattice step
        {"name": "relabel_2mm", "kind": "relabel", "surfaces": "head8", "cells": 100, "move": 0.4},
        # volume smoothing of the refined mesh, ten iterations
        {"name": "smooth_refined", "kind": "smooth", "surfaces": "head8", "cells": 50, "levels": 3, "iters": 10,
         "fixed": False},
        # tissue-boundary smoothing of the refined mesh, the usual stop rule
        {"name": "surface_refined", "kind": "surface", "surfaces": "head8", "cells": 50, "levels": 3, "xi": 0.1,
         "iters": 100},
        # inflation of the refined mesh towards the brain surface
        {"name": "inflate_refined", "kind": "inflate", "surfaces": "head8", "cells": 50, "levels": 3,
         "zeta": 0.05},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["host", "noalloc", "scatter", "lattice", "lattice", "elements", "refine", "relabel", "smooth",
                       "surface", "inflate"])
    if kind == "host":
        return {"kind": kind, "surfaces": "sphere", "freq": rng.randint(3, 24), "points": _log(rng, 1000, 40_000)}
    if kind == "noalloc":
        return {"kind": kind, "surfaces": rng.choice(["sphere", "head"]), "freq": rng.randint(3, 24),
                "points": _log(rng, 1000, 65_536), "omega": rng.random() < 0.5}
    if kind == "scatter":
        return {"kind": kind, "surfaces": rng.choice(["head", "head8", "deep"]), "points": _log(rng, 20_000, 4_000_000),
                "omega": rng.random() < 0.5}
    if kind == "lattice":
        s = rng.choice(["head", "deep", "full"])
        return {"kind": kind, "surfaces": s, "cells": _log(rng, 20, 180)}
    if kind == "elements":
        return {"kind": kind, "surfaces": rng.choice(["head", "head8"]), "cells": _log(rng, 20, 130)}
    if kind == "refine":
        return {"kind": kind, "surfaces": "head8", "cells": rng.randint(20, 50), "levels": rng.randint(1, 3),
                "conforming": rng.random() < 0.5}
    if kind == "relabel":
        return {"kind": kind, "surfaces": "head8", "cells": _log(rng, 20, 120), "move": round(rng.uniform(0.05, 0.4), 3)}
    mesh = {"surfaces": "head8", "cells": rng.randint(20, 50), "levels": rng.randint(0, 3)}
    if kind == "smooth":
        return {"kind": kind, **mesh, "iters": rng.randint(1, 12), "fixed": rng.random() < 0.5}
    if kind == "surface":
        return {"kind": kind, **mesh, "xi": rng.choice([0.1, 0.0]), "iters": rng.randint(1, 8)}
    return {"kind": kind, **mesh, "zeta": round(rng.uniform(0.01, 0.2), 3)}


# ---------------------------------------------------------------- inputs
def _jitter(nodes, amount: float, seed: int):
    r = torch.rand(nodes.shape, generator=_gen(seed, 3), device=DEV) * 2.0 - 1.0
    return (nodes + amount * r).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    ctx, half = _context(case, seed)
    st = {"case": case, "ctx": ctx}
    if kind == "host":
        n = case["points"]
        st["pts"] = np.random.default_rng([seed, 7]).uniform(-half, half, size=(n, 3)).astype(np.float32)
        st["labels"] = np.empty(n, dtype=np.int32)
    elif kind in ("noalloc", "scatter", "lattice"):
        pts = _centroids(case["cells"], half, seed) if kind == "lattice" else _uniform_points(case["points"], half, seed)
        st["pts"] = pts
        st["labels"] = torch.empty(pts.shape[0], dtype=torch.int32, device=DEV)
        st["omega"] = torch.empty((ctx.info()[0], pts.shape[0]), device=DEV) if case.get("omega") else None
    elif kind == "elements":
        st["nodes"], st["tets"] = _lattice(case["cells"], half, seed)
        st["elem"] = torch.empty(st["tets"].shape[0], dtype=torch.int32, device=DEV)
        st["labels"] = torch.empty(st["nodes"].shape[0], dtype=torch.int32, device=DEV)
    elif kind == "refine":
        st["nodes"], st["tets"] = _lattice(case["cells"], half, seed)
        cn, cm = _capacity(case)
        st["wn"] = torch.zeros((cn, 3), device=DEV)
        st["wt"] = torch.zeros((cm, 4), dtype=torch.int32, device=DEV)
        st["wl"] = torch.zeros(cn, dtype=torch.int32, device=DEV)
    elif kind == "relabel":
        nodes, st["tets"] = _lattice(case["cells"], half, seed)
        st["labels0"] = ctx.label_points(nodes, stats=False)[0]
        st["nodes"] = _jitter(nodes, case["move"] * 2.0 * half / case["cells"], seed)
        st["labels"] = torch.empty_like(st["labels0"])
    else:
        nodes, st["tets"] = _refined(ctx, case, half, seed)
        h = 2.0 * half / case["cells"] / 2 ** case["levels"]
        if kind == "surface":
            st["elem"] = ctx.label_elements(nodes, st["tets"], stats=False)[0]
        if kind == "smooth":
            st["fixed"] = ((torch.rand(nodes.shape[0], generator=_gen(seed, 4), device=DEV) < 0.1).to(torch.uint8)
                           if case["fixed"] else None)
        st["nodes0"] = nodes if kind == "inflate" else _jitter(nodes, 0.1 * h, seed)
        # the mesh lives in arrays of the refinement's capacity
        st["array"] = torch.zeros((_capacity(case)[0], 3), device=DEV)
        st["nodes"] = st["array"][:nodes.shape[0]]
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "host":
        return ctx.label_points(st["pts"], labels=st["labels"], stats=False)[0]
    if kind == "noalloc":
        om = st["omega"]
        status = zef.lib().zef_label_points_noalloc(ctx.handle, st["pts"].data_ptr(), st["pts"].shape[0],
                                                    st["labels"].data_ptr(), None if om is None else om.data_ptr(),
                                                    ctypes.byref(zef.make_opts()), None)
        if status != zef.ZEF_OK:
            raise zef.ZefError(status, "zef_label_points_noalloc")
        return {"labels": st["labels"], "omega": om} if om is not None else {"labels": st["labels"]}
    if kind in ("scatter", "lattice"):
        lab, om, _ = ctx.label_points(st["pts"], labels=st["labels"], omega=st["omega"], stats=False)
        return {"labels": lab, "omega": om} if om is not None else {"labels": lab}
    if kind == "elements":
        el, nl, _ = ctx.label_elements(st["nodes"], st["tets"], elem_labels=st["elem"], node_labels=st["labels"],
                                       stats=False)
        return {"elements": el, "nodes": nl}
    if kind == "refine":
        n0, m0 = st["nodes"].shape[0], st["tets"].shape[0]
        st["wn"][:n0].copy_(st["nodes"])
        st["wt"][:m0].copy_(st["tets"])
        n1, m1, _ = ctx.refine_and_relabel(st["wn"], st["wt"], st["wl"], n0, m0, case["levels"],
                                           conforming=case["conforming"])
        return {"nodes": st["wn"], "tets": st["wt"], "labels": st["wl"], "counts": [n1, m1]}
    if kind == "relabel":
        st["labels"].copy_(st["labels0"])
        per, conv = ctx.relabel_boundary(st["nodes"], st["tets"], st["labels"], 64)
        passes = np.zeros((64, 2), dtype=np.int64)
        passes[:len(per)] = per
        return {"labels": st["labels"], "passes": passes, "converged": int(conv)}
    st["nodes"].copy_(st["nodes0"])
    if kind == "smooth":
        it = ctx.taubin_smooth(st["nodes"], st["tets"], 0.4, 0.4, 0.0, case["iters"], fixed=st["fixed"])
        return {"nodes": st["array"], "iterations": it}
    if kind == "surface":
        it, faces = ctx.taubin_smooth_surface(st["nodes"], st["tets"], st["elem"], 0.4, 0.4, case["xi"], case["iters"])
        return {"nodes": st["array"], "iterations": it, "faces": faces}
    moved = ctx.inflate(st["nodes"], st["tets"], 3, case["zeta"])
    return {"nodes": st["array"], "moved": moved}


# ---------------------------------------------------------------- work of one pass
def work(case):
    surfs, _, _ = _base(case["surfaces"], case.get("freq", 8))
    C = len(surfs)
    sb = sum(12 * v.shape[0] + 12 * t.shape[0] for _, v, t in surfs)
    kind = case["kind"]
    if kind in ("host", "noalloc", "scatter", "lattice"):
        n = 5 * case["cells"] ** 3 if kind == "lattice" else case["points"]
        # points in, labels (and solid angles) out, the surfaces once; every
        # point is compared with every compartment's box
        return {"bytes": 16 * n + sb + (4 * C * n if case.get("omega") else 0), "flops": 6 * C * n}
    n, m = (case["cells"] + 1) ** 3, 5 * case["cells"] ** 3
    if kind == "elements":
        return {"bytes": 16 * n + 20 * m + sb, "flops": 6 * C * n + 4 * m}
    if kind == "relabel":
        return {"bytes": 20 * n + 16 * m + sb, "flops": 6 * C * n // 4}
    f = _flagged(case)
    n1, m1 = int(n + 1.72 * f), int(m + 7 * f)
    if kind == "refine":
        return {"bytes": 16 * n1 + 16 * m1 + 12 * n + 16 * m + sb, "flops": 6 * C * n1}
    it = 1 if case.get("xi") else case.get("iters", 0)
    base = {"bytes": 24 * n1 + 16 * m1, "flops": int(2 * it * 6 * 2.4 * m1)}
    if kind == "surface":
        base = {"bytes": base["bytes"] + 4 * m1, "flops": int(it * 30 * f)}
    elif kind == "inflate":
        base = {"bytes": base["bytes"] + sb, "flops": 6 * C * n1}
    return base


# ---------------------------------------------------------------- 64-bit values
def _omega64(pts, surfs):
    """Solid angles of closed surfaces at pts: sum over the triangles of
    2 atan2(R1 . (R2 x R3), r1 r2 r3 + ...), all in 64 bits."""
    rows = []
    for _, v, t in surfs:
        vv = torch.from_numpy(v).to(DEV).double()
        tri = vv[torch.from_numpy(np.ascontiguousarray(t)).to(DEV).long()]
        out = torch.zeros(pts.shape[0], dtype=torch.float64, device=DEV)
        step = max(1, 40_000_000 // tri.shape[0])
        for s in range(0, pts.shape[0], step):
            r = tri[None] - pts[s:s + step, None, None, :].double()
            a, b, c = r[:, :, 0], r[:, :, 1], r[:, :, 2]
            la, lb, lc = a.norm(dim=-1), b.norm(dim=-1), c.norm(dim=-1)
            num = (a * torch.linalg.cross(b, c)).sum(-1)
            den = la * lb * lc + (a * b).sum(-1) * lc + (a * c).sum(-1) * lb + (b * c).sum(-1) * la
            out[s:s + step] = 2.0 * torch.atan2(num, den).sum(1)
        rows.append(out)
    return torch.stack(rows)


def _pairs_unique(a, b):
    lo, hi = torch.minimum(a, b).long(), torch.maximum(a, b).long()
    k = torch.unique((lo << 32) | hi)
    return k >> 32, k & 0xFFFFFFFF


_EDGE = [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]


def _mesh_edges(tets):
    a = torch.cat([tets[:, i] for i, _ in _EDGE])
    b = torch.cat([tets[:, j] for _, j in _EDGE])
    return _pairs_unique(a, b)


def _taubin64(x, a, b, n, iters, fixed=None):
    deg = torch.zeros(n, dtype=torch.float64, device=DEV)
    one = torch.ones(a.shape[0], dtype=torch.float64, device=DEV)
    deg.index_add_(0, a, one)
    deg.index_add_(0, b, one)
    lam = torch.tensor(np.float32(0.4), device=DEV).double()
    move = torch.ones((n, 1), dtype=torch.float64, device=DEV)
    if fixed is not None:
        move[fixed != 0] = 0.0
    w = lam * move / (deg + 1.0)[:, None]

    def lap(p):
        d = p[b] - p[a]
        s = torch.zeros_like(p)
        s.index_add_(0, a, d)
        s.index_add_(0, b, -d)
        return s

    for _ in range(iters):
        x = x + w * lap(x)
        x = x - w * lap(x)
    return x


def _boundary_edges(tets, lab, n):
    """Edges of the faces between tets of different labels, and their count."""
    idx = [(0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3)]
    f = torch.cat([tets[:, list(q)] for q in idx]).long().sort(1).values
    l = lab.repeat(4)
    _, ab = torch.unique((f[:, 0] << 32) | f[:, 1], return_inverse=True)
    _, face = torch.unique(ab * n + f[:, 2], return_inverse=True)
    nf = int(face.max()) + 1
    lo = torch.full((nf,), 1 << 30, dtype=l.dtype, device=DEV).scatter_reduce_(0, face, l, "amin")
    hi = torch.full((nf,), -(1 << 30), dtype=l.dtype, device=DEV).scatter_reduce_(0, face, l, "amax")
    rep = torch.zeros(nf, dtype=torch.long, device=DEV)
    rep[face] = torch.arange(f.shape[0], device=DEV)
    t = f[rep[lo != hi]]
    if not t.shape[0]:
        return t[:, 0], t[:, 0], 0
    a, b = _pairs_unique(torch.cat([t[:, 0], t[:, 0], t[:, 1]]), torch.cat([t[:, 1], t[:, 2], t[:, 2]]))
    return a, b, t.shape[0]


def _inflate64(x, tets, v, t, zeta):
    """Inside nodes moved towards the surface along their crossing edges."""
    inside = _omega64(x, [(0, v, t)])[0] > 2.0 * math.pi
    a, b = _mesh_edges(tets)
    cross = inside[a] != inside[b]
    i = torch.where(inside[a], a, b)[cross]
    j = torch.where(inside[a], b, a)[cross]
    xd = x.double()
    tri = torch.from_numpy(v).to(DEV).double()[torch.from_numpy(np.ascontiguousarray(t)).to(DEV).long()]
    e1, e2 = tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    best = torch.full((i.shape[0],), math.inf, dtype=torch.float64, device=DEV)
    eps = 2.0 ** -20
    step = max(1, 20_000_000 // tri.shape[0])
    for s in range(0, i.shape[0], step):
        p, d = xd[i[s:s + step]][:, None], (xd[j[s:s + step]] - xd[i[s:s + step]])[:, None]
        h = torch.linalg.cross(d.expand(-1, tri.shape[0], -1), e2[None].expand(d.shape[0], -1, -1))
        det = (e1[None] * h).sum(-1)
        tv = p - tri[None, :, 0]
        u = (tv * h).sum(-1) / det
        q = torch.linalg.cross(tv, e1[None].expand(d.shape[0], -1, -1))
        w = (d * q).sum(-1) / det
        tt = (e2[None] * q).sum(-1) / det
        ok = (u >= -eps) & (u <= 1 + eps) & (w >= -eps) & (u + w <= 1 + eps) & (tt >= 0) & (tt <= 1 + eps)
        best[s:s + step] = torch.where(ok, tt, math.inf).amin(1)
    hit = best < math.inf
    i, j, best = i[hit], j[hit], best[hit].clamp(max=1.0)
    mv = torch.zeros_like(xd)
    cnt = torch.zeros(x.shape[0], dtype=torch.float64, device=DEV)
    mv.index_add_(0, i, float(np.float32(zeta)) * best[:, None] * (xd[j] - xd[i]))
    cnt.index_add_(0, i, torch.ones_like(best))
    return xd + mv / cnt.clamp(min=1.0)[:, None]


def _padded(x, case):
    out = torch.zeros((_capacity(case)[0], 3), dtype=x.dtype, device=DEV)
    out[:x.shape[0]] = x
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("noalloc", "scatter") and case.get("omega"):
        surfs, _, half = _surfaces(case, seed)
        if case["points"] * sum(t.shape[0] for _, _, t in surfs) > 3e9:
            return None
        return {"labels": None, "omega": _omega64(_uniform_points(case["points"], half, seed), surfs)}
    if kind in ("smooth", "surface"):
        st = prepare(case, seed)
        x = st["nodes0"].double()
        n = x.shape[0]
        if kind == "smooth":
            a, b = _mesh_edges(st["tets"])
            return {"nodes": _padded(_taubin64(x, a, b, n, case["iters"], st["fixed"]), case), "iterations": None}
        a, b, faces = _boundary_edges(st["tets"], st["elem"], n)
        # the stop rule at xi = 0.1 ends after the first iteration: a step
        # never moves the nodes by a tenth of their distance to the origin
        it = 1 if case["xi"] else case["iters"]
        return {"nodes": _padded(_taubin64(x, a, b, n, it), case), "iterations": None, "faces": None}
    if kind == "inflate":
        surfs, _, half = _surfaces(case, seed)
        v, t = next((v, t) for cid, v, t in surfs if cid == 3)
        f = _flagged(case)
        if ((case["cells"] + 1) ** 3 + 1.72 * f) * t.shape[0] > 2.5e10:
            return None
        st = prepare(case, seed)
        return {"nodes": _padded(_inflate64(st["nodes0"], st["tets"], v, t, case["zeta"]), case), "moved": None}
    return None
