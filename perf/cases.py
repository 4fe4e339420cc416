"""The calls that a program using this library makes, as measured cases.

A case names a mesh, a batch of queries on it and the call that takes them: the exponential map
alone, a differentiated step (forward and the vector-Jacobian product of one of the estimators), the
K-step map of a vector field and its gradient, the traced geodesics, walks around holes, and a step
that moves the vertices.  Meshes and query distributions are the ones of the repository's workloads
(icospheres, a noisy torus, sliver heightfields, uneven multi-mesh batches, a sphere with faces
removed): area-weighted start faces, points uniform on the face, uniform directions, lengths uniform
up to a stated bound.

`exact` walks the same queries in 64 bits: a plain torch walk in 3-D over all queries in lock step,
with the paper's finite differences and, for vertex positions, automatic differentiation of the walk.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2603_15780_gb300 as sg


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # The smallest call: a thousand points on a coarse sphere, one carried vector (an interactive
        # tool, one patch of a convolution).  Latency and launches decide.
        _c("exp-1k", "exp", "sphere", level=3, queries=1000, lo=0.0, hi=math.pi, carried=1),
        # A training step on tens of thousands of points over several meshes at once, GFD gradients in
        # the point and the vector.
        _c("step-20k-multimesh-gfd", "step", "batch", meshes=8, faces=20000, queries=20011, lo=0.0, hi=0.3,
           estimator="gfd", eps=1e-3),
        # The full-precision reference walk on a batch that a program checks its results with.
        _c("exp-fp64-16k", "exp", "torus", na=256, nb=128, queries=16385, lo=0.0, hi=1.0, precision=64),
        # The headline forward: a million points on an 81,920-face noisy sphere.
        _c("exp-1m-sphere", "exp", "sphere", level=6, queries=1048576, lo=0.1, hi=1.0),
        # The headline training step on the same mesh: GFD gradients in point, vector and vertices.
        _c("step-1m-sphere-gfd-V", "step", "sphere", level=6, queries=1048576, lo=0.1, hi=1.0, estimator="gfd",
           grad_V=True),
        # The largest forward batch: four million points on a noisy torus, two carried vectors.
        _c("exp-4m-torus-2w", "exp", "torus", na=512, nb=256, queries=4194304, lo=0.0, hi=2.0, carried=2),
        # Geodesic convolution over a batch of 64 uneven meshes with the cheap EP gradient; walks up to
        # half a mesh long, so a part of them needs the wider arithmetic.
        _c("step-64meshes-ep", "step", "batch", meshes=64, faces=60000, queries=1000003, lo=0.0, hi=0.5,
           estimator="ep"),
        # Long walks (hundreds to thousands of crossings) on a sliver heightfield larger than the L2.
        _c("exp-heightfield-long", "exp", "heightfield", n=1025, queries=524288, lo=0.0, hi=3.0),
        # Geodesics drawn as polylines.
        _c("trace-10k", "trace", "sphere", level=5, queries=10007, lo=0.1, hi=1.0, cap=64),
        # A scanned surface with many holes: walks go round them.
        _c("exp-holes-262k", "exp", "holes", level=6, queries=262147, lo=0.1, hi=1.0, boundary=1),
        # Flow matching: five steps along a field sampled at the vertices, and the gradient in the field.
        _c("field-5steps-262k-gfd", "field", "sphere", level=6, queries=262144, lo=0.1, hi=1.0, K=5, estimator="gfd",
           eps=1e-3),
        # Optimising a shape: move the vertices, walk, and take the gradient back to them.
        _c("update-100k-gfd-V", "update", "torus", na=256, nb=128, queries=100003, lo=0.0, hi=0.5, estimator="gfd",
           eps=1e-3, grad_V=True),
    ]


def _c(name, call, mesh, **kw):
    return {"name": name, "call": call, "mesh": mesh, **kw}


def draw(rng):
    """Another case of the same ranges: any of the calls, on any of the meshes it is used with."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["exp", "exp", "exp", "step", "step", "step", "trace", "field", "update"])
    hi_q = {"exp": 2000000, "step": 1000000, "trace": 200000, "field": 200000, "update": 500000}[call]
    c = {"call": call, "queries": size(200, hi_q)}
    kinds = ["sphere", "torus"] + (["batch", "heightfield"] if call in ("exp", "step") else [])
    c["mesh"] = rng.choice(kinds + (["holes"] if call == "exp" else []))
    if c["mesh"] in ("sphere", "holes"):
        c["level"] = rng.randint(3, 6)
    elif c["mesh"] == "torus":
        c["na"], c["nb"] = size(24, 512), size(12, 256)
    elif c["mesh"] == "batch":
        c["meshes"], c["faces"] = size(2, 64), size(2000, 60000)
    else:
        c["n"] = size(64, 800)
        c["queries"] = min(c["queries"], 300000)
    c["lo"] = 0.0
    c["hi"] = {"sphere": 1.0, "holes": 1.0, "torus": 1.0, "batch": 0.5, "heightfield": 3.0}[c["mesh"]]
    c["hi"] *= rng.uniform(0.3, 1.0)
    if call == "exp":
        c["carried"] = rng.choice([0, 0, 1, 2, 3])
        if c["mesh"] == "holes":
            c["boundary"] = 1
        elif c["queries"] <= 20000 and rng.random() < 0.3:
            c["precision"] = rng.choice([32, 40, 48, 64])
    if call == "step":
        c["estimator"] = rng.choice(["gfd", "ep"])
        if c["mesh"] == "heightfield":
            c["hi"] = rng.uniform(0.05, 0.4)
        c["grad_V"] = rng.random() < 0.4
    if call == "trace":
        c["cap"] = rng.choice([30, 64, 100])
    if call == "field":
        c["K"], c["estimator"] = rng.randint(2, 8), rng.choice(["gfd", "ep"])
    if call == "update":
        c["estimator"], c["grad_V"] = "gfd", True
    if c.get("estimator") == "gfd":   # a step that suits coarse meshes; the library's default on large batches
        c["eps"] = 1e-4 if c["queries"] > 300000 else 1e-3
    return c


# --------------------------------------------------------------------------- meshes
@functools.lru_cache(maxsize=None)
def _icosphere(level):
    t = (1.0 + math.sqrt(5.0)) / 2.0
    V = np.array([(-1, t, 0), (1, t, 0), (-1, -t, 0), (1, -t, 0), (0, -1, t), (0, 1, t), (0, -1, -t), (0, 1, -t),
                  (t, 0, -1), (t, 0, 1), (-t, 0, -1), (-t, 0, 1)], float)
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    F = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                  (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11),
                  (6, 2, 10), (8, 6, 7), (9, 8, 1)])
    for _ in range(level):
        e = np.sort(F[:, [0, 1, 1, 2, 2, 0]].reshape(-1, 2), axis=1)
        u, inv = np.unique(e[:, 0] * len(V) + e[:, 1], return_inverse=True)
        m = V[u // len(V)] + V[u % len(V)]
        ab, bc, ca = (len(V) + inv.reshape(-1, 3)).T
        a, b, c = F.T
        F = np.concatenate([np.stack(x, 1) for x in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
        V = np.concatenate([V, m / np.linalg.norm(m, axis=1, keepdims=True)])
    return V, F


def _sphere(level, rng):
    V, F = _icosphere(level)
    # radial noise of 0.003 on the finest sphere's edges, in proportion on coarser ones
    return V * (1.0 + rng.normal(0.0, 0.003 * 2.0 ** (6 - level) * 0.5, (len(V), 1))), F


def _holes(level, rng):
    """The sphere without a random set of faces no two of which share a vertex (about 8% of them), so
    that every vertex keeps one fan."""
    V, F = _sphere(level, rng)
    prio = rng.random(len(F))
    low = np.full(len(V), 2.0)
    for k in range(3):
        np.minimum.at(low, F[:, k], prio)
    return V, F[(prio[:, None] > low[F]).any(1)]


def _grid_faces(na, nb, wrap):
    i, j = (x.ravel() for x in np.meshgrid(np.arange(na), np.arange(nb), indexing="ij"))
    w = nb if wrap else nb + 1
    i1, j1 = ((i + 1) % na, (j + 1) % nb) if wrap else (i + 1, j + 1)
    v00, v10, v11, v01 = i * w + j, i1 * w + j, i1 * w + j1, i * w + j1
    return np.concatenate([np.stack([v00, v10, v11], 1), np.stack([v00, v11, v01], 1)])


def _torus(na, nb, rng):
    a, b = np.meshgrid(2 * np.pi * np.arange(na) / na, 2 * np.pi * np.arange(nb) / nb, indexing="ij")
    V = np.stack([(1 + 0.4 * np.cos(b)) * np.cos(a), (1 + 0.4 * np.cos(b)) * np.sin(a), 0.4 * np.sin(b)], -1)
    V = V.reshape(-1, 3)
    noise = 0.16 * min(2 * np.pi * 0.6 / na, 2 * np.pi * 0.4 / nb)   # 0.0012 on the 512 x 256 grid
    return V + rng.normal(0.0, noise, V.shape), _grid_faces(na, nb, True)


def _heightfield(n, rng, slivers=True):
    a, b, ph = rng.uniform(-4, 4, 8), rng.uniform(-4, 4, 8), rng.uniform(0, 2 * np.pi, 8)
    x, y = (g.ravel() for g in np.meshgrid(np.linspace(0, 1, n), np.linspace(0, 1, n), indexing="ij"))
    V = np.stack([x, y, np.zeros_like(x)], 1)
    if slivers:   # a tenth of the vertices, none of them neighbours, pushed close to a neighbour
        ii, jj = np.meshgrid(np.arange(2, n - 2, 2), np.arange(2, n - 2, 2), indexing="ij")
        cand = (ii * n + jj).ravel()
        pick = rng.choice(cand, size=min(len(cand), int(0.1 * n * n)), replace=False)
        step = rng.choice([-1.0, 1.0], len(pick)) * rng.uniform(0.45, 0.4995, len(pick)) / (n - 1)
        V[pick, rng.integers(0, 2, len(pick))] += step
    V[:, 2] = sum(0.05 * np.sin(2 * np.pi * (a[k] * V[:, 0] + b[k] * V[:, 1]) + ph[k]) for k in range(8))
    return V, _grid_faces(n - 1, n - 1, False)


def _meshes(case, rng):
    """[(V float32, F int32)] of a case."""
    kind = case["mesh"]
    if kind == "sphere":
        out = [_sphere(case["level"], rng)]
    elif kind == "holes":
        out = [_holes(case["level"], rng)]
    elif kind == "torus":
        out = [_torus(case["na"], case["nb"], rng)]
    elif kind == "heightfield":
        out = [_heightfield(case["n"], rng)]
    else:   # uneven sizes: log-uniform between a twentieth of `faces` and `faces`
        out = []
        for m in range(case["meshes"]):
            f = math.exp(rng.uniform(math.log(case["faces"] / 20), math.log(case["faces"])))
            if m % 3 == 0:
                out.append(_sphere(min(6, max(1, round(math.log(f / 20, 4)))), rng))
            elif m % 3 == 1:
                nb = max(4, round(math.sqrt(f / 4)))
                out.append(_torus(2 * nb, nb, rng))
            else:
                out.append(_heightfield(max(8, round(math.sqrt(f / 2)) + 1), rng, slivers=False))
    return [(np.ascontiguousarray(V, np.float32), np.ascontiguousarray(F, np.int32)) for V, F in out]


def _queries(case, meshes, rng):
    """Start faces (local to their mesh), points, vectors, carried vectors, mesh ids, upstream gradients."""
    nq, parts = case["queries"], []
    area = [0.5 * np.linalg.norm(np.cross(V[F[:, 1]] - V[F[:, 0]], V[F[:, 2]] - V[F[:, 0]]), axis=1) for V, F in meshes]
    share = np.array([len(F) for _, F in meshes], float)
    ids = np.sort(rng.choice(len(meshes), nq, p=share / share.sum())) if len(meshes) > 1 else np.zeros(nq, int)
    for m, (V, F) in enumerate(meshes):
        k = int((ids == m).sum())
        cdf = np.cumsum(area[m], dtype=np.float64)
        face = np.minimum(np.searchsorted(cdf, rng.random(k) * cdf[-1], side="right"), len(F) - 1)
        r1, r2, phi = np.sqrt(rng.random(k)), rng.random(k), rng.uniform(0, 2 * np.pi, k)
        bary = np.stack([1 - r1, r1 * (1 - r2), r1 * r2], 1)
        X = V.astype(np.float64)[F[face]]
        e1 = X[:, 1] - X[:, 0]
        e1 /= np.linalg.norm(e1, axis=1, keepdims=True)
        n = np.cross(X[:, 1] - X[:, 0], X[:, 2] - X[:, 0])
        n /= np.linalg.norm(n, axis=1, keepdims=True)
        e2 = np.cross(n, e1)
        # lengths are absolute on one mesh, fractions of the diagonal in batches and on heightfields
        diag = np.linalg.norm(V.max(0) - V.min(0)) if case["mesh"] in ("batch", "heightfield") else 1.0
        L = rng.uniform(case["lo"], case["hi"], k) * diag
        v = L[:, None] * (np.cos(phi)[:, None] * e1 + np.sin(phi)[:, None] * e2)
        psi = rng.uniform(0, 2 * np.pi, (k, case.get("carried", 0)))
        w = np.cos(psi)[..., None] * e1[:, None] + np.sin(psi)[..., None] * e2[:, None]
        parts.append((face, bary, v, w))
    face, bary, v, w = (np.concatenate(x) for x in zip(*parts))
    q = {"face": face.astype(np.int32), "bary": bary.astype(np.float32), "v": v.astype(np.float32),
         "w": w.astype(np.float32), "ids": ids.astype(np.int32), "g": rng.normal(size=(nq, 3)).astype(np.float32)}
    if len(meshes) > 1:   # the queries of a batch come mixed
        p = rng.permutation(nq)
        q = {k: x[p] for k, x in q.items()}
    return q


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    meshes = _meshes(case, rng)
    q = _queries(case, meshes, rng)
    nV = sum(len(V) for V, _ in meshes)
    if case["call"] == "field":   # a smooth field: an affine one, with lengths like the other cases'
        A = rng.normal(size=(3, 3)) * 0.5 * case["hi"]
        q["U"] = (meshes[0][0] @ A + rng.normal(size=3) * 0.3 * case["hi"]).astype(np.float32)
    if case["call"] == "update":  # a small move of every vertex
        V = meshes[0][0]
        q["V"] = (V * (1 + 0.02 * np.sin(3 * V[:, :1])) + 0.01 * rng.normal(size=3)).astype(np.float32)
    assert nV > 0
    return meshes, q


# --------------------------------------------------------------------------- the calls
def prepare(case, seed):
    meshes, q = _inputs(case, seed)
    mesh = sg.Mesh(*meshes[0]) if len(meshes) == 1 else sg.Mesh(meshes)
    s = {k: torch.as_tensor(x, device="cuda") for k, x in q.items()}
    s.update(case=case, mesh=mesh, mesh_id=s["ids"] if len(meshes) > 1 else None)
    if case["call"] in ("step", "update"):
        s["v"].requires_grad_()
        s["bary"].requires_grad_()
        if case.get("grad_V"):
            V = s["V"] if case["call"] == "update" else torch.as_tensor(mesh.V, device="cuda")
            s["V"] = V.requires_grad_()
    if case["call"] == "field":
        s["bary"].requires_grad_()
        s["U"].requires_grad_()
    return s


def run(s):
    c, mesh = s["case"], s["mesh"]
    if c["call"] == "exp":
        o = sg.exp_map(mesh, s["face"], s["bary"], s["v"], s["w"] if c.get("carried") else None, mesh_id=s["mesh_id"],
                       precision=c.get("precision"), boundary_mode=c.get("boundary"))
        return {k: o[k] for k in ("face", "bary", "pos", "dir", "w", "status", "ncross") if k in o}
    if c["call"] == "trace":
        o = sg.exp_map_trace(mesh, s["face"], s["bary"], s["v"], path_cap=c["cap"])
        # entries past a path's length are not written: the padding that a drawing program sets
        pad = torch.arange(c["cap"], device="cuda")[None] >= o["path_len"][:, None]
        o["path_face"].masked_fill_(pad, -1)
        o["path_pt"].masked_fill_(pad[..., None], 0.0)
        return {k: o[k] for k in ("face", "bary", "pos", "dir", "status", "ncross", "path_face", "path_pt", "path_len")}
    if c["call"] == "field":
        pos, face, bary, d, st = sg.ExpMapFieldSteps.apply(mesh, s["face"], s["bary"], s["U"], c["K"], None,
                                                           c["estimator"], None, c.get("eps", 1e-4))
        gb, gU = torch.autograd.grad(pos, [s["bary"], s["U"]], s["g"])
        return {"pos": pos.detach(), "face": face, "bary": bary.detach(), "dir": d.detach(), "status": st,
                "grad_bary": gb, "grad_U": gU}
    V = s.get("V")
    if c["call"] == "update":
        mesh.update_vertices(V.detach())
    pos, face, bary, d, st = sg.ExpMap.apply(mesh, s["face"], s["bary"], s["v"], c["estimator"], V, s["mesh_id"],
                                         c.get("eps", 1e-4))
    wrt = [s["v"], s["bary"]] + ([V] if V is not None else [])
    g = torch.autograd.grad(pos, wrt, s["g"])
    out = {"pos": pos.detach(), "face": face, "bary": bary.detach(), "dir": d.detach(), "status": st, "grad_v": g[0],
           "grad_bary": g[1]}
    if V is not None:
        out["grad_V"] = g[2]
    return out


def work(case):
    """The mesh and the queries read once, the outputs written once; about 60 operations for each edge
    crossed, and the crossings that the walks of the path cannot do without (a gradient in the vertices
    takes a second walk's adjoint, about as much again)."""
    kind, nq = case["mesh"], case["queries"]
    if kind in ("sphere", "holes"):
        nf, edge, ext = 20 * 4 ** case["level"], 1.1 / 2 ** case["level"], 1.0
    elif kind == "torus":
        nf, edge, ext = 2 * case["na"] * case["nb"], 2 * math.pi * (1 / case["na"] + 0.4 / case["nb"]) / 2, 1.0
    elif kind == "heightfield":
        # walks end at the border: nine tenths of a side on average once they are long
        nf, edge, ext = 2 * case["n"] ** 2, 1.8 / case["n"], 1.6
    else:
        # (the mean of a log-uniform size is about a third of its upper end)
        nf, edge, ext = case["meshes"] * case["faces"] // 3, 3.0 / math.sqrt(case["faces"] / 3), 2.0
    mean = 0.5 * (case["lo"] + case["hi"]) * ext
    if kind == "heightfield":
        mean = min(mean, 0.9)
    cross = 2.3 * mean / edge
    nv = nf // 2
    mesh = 12 * nf + 12 * nv
    q_in, q_out = 4 + 12 + 12, 4 + 12 + 12 + 12 + 4
    flops = 60.0 * cross * nq
    if case["call"] == "exp":
        k = case.get("carried", 0)
        per = q_in + q_out + 4 + 24 * k
    elif case["call"] == "trace":
        per = q_in + q_out + 8 + 16 * case["cap"]
    elif case["call"] == "field":
        per = 16 + q_out + 24
        mesh += 24 * nv
    else:
        per = q_in + q_out + 12 + 24
        if case.get("grad_V"):
            mesh += 12 * nv
            flops *= 2
        if case["call"] == "update":
            mesh += 12 * nv
    return {"bytes": mesh + per * nq, "flops": flops}


# --------------------------------------------------------------------------- 64-bit results
def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


class _Mesh64:
    """Positions and adjacency of all meshes of a case, faces numbered through."""

    def __init__(self, meshes):
        off = np.cumsum([0] + [len(V) for V, _ in meshes])
        self.foff = torch.as_tensor(np.cumsum([0] + [len(F) for _, F in meshes]), device="cuda")
        self.X = torch.as_tensor(np.concatenate([V for V, _ in meshes]).astype(np.float64), device="cuda")
        self.F = torch.as_tensor(np.concatenate([F + o for (_, F), o in zip(meshes, off)]).astype(np.int64), device="cuda")
        h = torch.stack([self.F, self.F.roll(-1, 1)], -1).reshape(-1, 2)     # half-edges 3f + k
        key = h.min(1).values * len(self.X) + h.max(1).values
        key, order = key.sort(stable=True)
        same = torch.nonzero(key[1:] == key[:-1])[:, 0]
        self.twin = torch.full((len(h),), -1, device="cuda")
        a, b = order[same], order[same + 1]
        self.twin[a], self.twin[b] = b, a
        ids = torch.searchsorted(self.foff, torch.arange(len(self.F), device="cuda"), right=True) - 1
        l = (self.X[h[:, 0]] - self.X[h[:, 1]]).norm(dim=1)
        # mean edge length per mesh, each edge once
        use = (self.twin < 0) | (torch.arange(len(h), device="cuda") < self.twin)
        ids3 = ids.repeat_interleave(3)[use]
        n = torch.zeros(len(meshes), dtype=torch.float64, device="cuda")
        self.lref = n.index_add(0, ids3, l[use]) / n.index_add(0, ids3, torch.ones_like(l[use]))
        self.mesh_of = ids

    def corners(self, f, X=None):
        return (self.X if X is None else X)[self.F[f]]


def _frame(P):
    """Unit normal of faces with corners P [..., 3, 3]."""
    return _unit(_cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]))


def _walk(M, f, p, d, L, carry=(), path=None):
    """Straightest walks in lock step from points p of faces f along unit tangents d over lengths L.
    Returns (face, point, direction, carried vectors)."""
    f, p, d, L = f.clone(), p.clone(), d.clone(), L.clone().reshape(-1)
    n0 = _frame(M.corners(f))
    ang = [(_dot(c, d), _dot(c, _cross(n0, d))) for c in carry]
    live = torch.nonzero(L > 0)[:, 0]
    fa, pa, da, La = f[live], p[live], d[live], L[live]
    entry = torch.full_like(fa, -1)
    step = 0
    if path is not None:
        path[live, 0] = pa
    while len(live):
        P = M.corners(fa)
        n = _frame(P)
        sig = (n[:, None] * _cross(da[:, None].expand_as(P), P - pa[:, None])).sum(-1)
        nxt = sig.roll(-1, 1)
        free = ((sig < 0) & (nxt >= 0)).to(torch.int64).argmax(1)
        apex = sig.gather(1, ((entry + 2) % 3)[:, None])[:, 0]
        j = torch.where(entry < 0, free, torch.where(apex > 0, (entry + 1) % 3, (entry + 2) % 3))[:, None]
        A = P.gather(1, j[..., None].expand(-1, 1, 3))[:, 0]
        B = P.gather(1, ((j + 1) % 3)[..., None].expand(-1, 1, 3))[:, 0]
        s0, s1 = sig.gather(1, j), sig.gather(1, (j + 1) % 3)
        q = A + (s0 / (s0 - s1)).clamp(0, 1) * (B - A)
        t = _dot(q - pa, da).clamp_min(0)[:, 0]
        tw = M.twin[3 * fa + j[:, 0]]
        end = t >= La
        stop = end | (tw < 0)
        if bool(stop.any()):
            i = live[stop]
            f[i], d[i] = fa[stop], da[stop]
            p[i] = torch.where(end[:, None], pa + La[:, None] * da, q)[stop]
        go = torch.nonzero(~stop)[:, 0]
        live, La, tw, q, A, B = live[go], (La - t)[go], tw[go], q[go], A[go], B[go]
        e, nd = _unit(B - A), da[go]
        along, out = _dot(nd, e), _dot(nd, _cross(e, n[go]))
        fa, entry, pa = tw // 3, tw % 3, q
        Pn = M.corners(fa)
        k = entry[:, None, None].expand(-1, 1, 3)
        eg = Pn.gather(1, (k + 1) % 3)[:, 0] - Pn.gather(1, k)[:, 0]
        da = _unit(along * e + out * _cross(_frame(Pn), _unit(eg)))
        step += 1
        if path is not None and step < path.shape[1]:
            path[live, step] = pa
    n1 = _frame(M.corners(f))
    return f, p, d, [a * d + b * _cross(n1, d) for a, b in ang]


def _bary(M, f, p):
    P = M.corners(f)
    u, w, r = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0], p - P[:, 0]
    uu, uw, ww, ru, rw = (_dot(a, b)[:, 0] for a, b in ((u, u), (u, w), (w, w), (r, u), (r, w)))
    det = uu * ww - uw * uw
    b1, b2 = (ww * ru - uw * rw) / det, (uu * rw - uw * ru) / det
    return torch.stack([1 - b1 - b2, b1, b2], 1)


def _start(M, f, b, v):
    P = M.corners(f)
    b = b.clamp_min(0)
    b = b / b.sum(1, keepdim=True)
    n = _frame(P)
    v = v - _dot(v, n) * n
    L = v.norm(dim=1)
    return (b[..., None] * P).sum(1), v / L.clamp_min(1e-300)[:, None], L


def _vjp(M, case, f, b, v, end, g):
    """(grad_v, grad_bary) of <g, Exp> by the case's estimator (finite differences of its step, the
    library's default if it gives none); `end` is (face, point, direction)."""
    est, step = case["estimator"], float(np.float32(case.get("eps", 1e-4)))
    P = M.corners(f)
    n, (p, d, L), (f1, p1, d1) = _frame(P), _start(M, f, b, v), end
    n1 = _frame(M.corners(f1))
    g = g - _dot(g, n1) * n1
    perp, perp1, ok = _cross(n, d), _cross(n1, d1), (L > 0)[:, None]
    if est == "ep":
        return torch.where(ok, _dot(g, d1) * d + _dot(g, perp1) * perp, 0.0), torch.zeros_like(g)
    eps = torch.full_like(L, step)
    diff = lambda x: _dot(x - p1, g) / step
    c_par = diff(_walk(M, f1, p1, d1, eps)[1])
    vp = L[:, None] * d + step * perp
    c_perp = diff(_walk(M, f, p, _unit(vp), vp.norm(dim=1))[1])
    eu, ev = _unit(P[:, 1] - P[:, 0]), _unit(P[:, 2] - P[:, 0])
    c = []
    for e in (eu, ev):
        fu, pu, _, (du,) = _walk(M, f, p, e, eps, [d])
        c.append(diff(_walk(M, fu, pu, du, L)[1]))
    a = _dot(eu, ev)
    det = 1 - a * a
    gp = (c[0] - a * c[1]) / det * eu + (c[1] - a * c[0]) / det * ev
    return (torch.where(ok, c_par * d + c_perp * perp, 0.0), torch.where(ok, (gp[:, None] * P).sum(-1), 0.0))


def _grad_V(M, f0, b, v, g, chunk=131072):
    """d<g, Exp>/dX with the face sequence held fixed, by automatic differentiation of the walk.  A walk
    that meets the border or passes a vertex within the library's snap radius has no such derivative."""
    X = M.X.clone().requires_grad_()
    total = torch.zeros_like(X)
    for i in range(0, len(f0), chunk):
        f, gi = f0[i:i + chunk], g[i:i + chunk]
        P = M.corners(f, X)
        n = _frame(P)
        p, vv = (b[i:i + chunk, :, None] * P).sum(1), v[i:i + chunk]
        vv = vv - _dot(vv, n) * n
        L = vv.norm(dim=1, keepdim=True)
        d, snap = vv / L, (1e-6 * M.lref[M.mesh_of[f]])[:, None]
        entry = torch.full_like(f, -1)
        live = torch.arange(len(f), device="cuda")
        loss = 0.0
        while len(live):
            P = M.corners(f, X)
            n = _frame(P)
            sig = (n[:, None] * _cross(d[:, None].expand_as(P), P - p[:, None])).sum(-1)
            free = ((sig < 0) & (sig.roll(-1, 1) >= 0)).to(torch.int64).argmax(1)
            apex = sig.gather(1, ((entry + 2) % 3)[:, None])[:, 0]
            j = torch.where(entry < 0, free, torch.where(apex > 0, (entry + 1) % 3, (entry + 2) % 3))[:, None]
            A = P.gather(1, j[..., None].expand(-1, 1, 3))[:, 0]
            B = P.gather(1, ((j + 1) % 3)[..., None].expand(-1, 1, 3))[:, 0]
            s0, s1 = sig.gather(1, j), sig.gather(1, (j + 1) % 3)
            q = A + s0 / (s0 - s1) * (B - A)
            t = _dot(q - p, d)
            end = (t >= L)[:, 0]
            loss = loss + (gi[live] * (p + L * d))[end].sum()
            tw = M.twin[3 * f + j[:, 0]]
            hit = (torch.minimum(s0.abs(), s1.abs()) <= snap)[:, 0]
            go = torch.nonzero(~end & (tw >= 0) & ~hit)[:, 0]
            live, L, tw, p, snap = live[go], (L - t)[go], tw[go], q[go], snap[go]
            e = _unit((B - A)[go])
            along, out = _dot(d[go], e), _dot(d[go], _cross(e, n[go]))
            f, entry = tw // 3, tw % 3
            Pn = M.corners(f, X)
            k = entry[:, None, None].expand(-1, 1, 3)
            eg = Pn.gather(1, (k + 1) % 3)[:, 0] - Pn.gather(1, k)[:, 0]
            d = along * e + out * _cross(_frame(Pn), _unit(eg))
        if torch.is_tensor(loss) and loss.requires_grad:
            total += torch.autograd.grad(loss, X)[0]
    return total


def exact(case, seed):
    """The 64-bit results; whole numbers (faces, statuses, counts) and walks around holes have none."""
    if case["mesh"] == "holes":
        return None
    meshes, q = _inputs(case, seed)
    if case["call"] == "update":
        meshes = [(q["V"], meshes[0][1])]
    M = _Mesh64(meshes)
    t = {k: torch.as_tensor(x, device="cuda").to(torch.float64) for k, x in q.items()}
    f = torch.as_tensor(q["face"], device="cuda").long() + M.foff[torch.as_tensor(q["ids"], device="cuda").long()]
    if case["call"] == "field":
        return _exact_field(case, M, f, t)
    p, d, L = _start(M, f, t["bary"], t["v"])
    k = case.get("carried", 0)
    path = torch.zeros(len(f), case["cap"], 3, dtype=torch.float64, device="cuda") if case["call"] == "trace" else None
    n = _frame(M.corners(f))
    carry = [t["w"][:, i] - _dot(t["w"][:, i], n) * n for i in range(k)]
    f1, p1, d1, w1 = _walk(M, f, p, d, L, carry, path)
    if case["call"] in ("exp", "trace"):
        out = {"face": None, "bary": _bary(M, f1, p1), "pos": p1, "dir": d1}
        if k:
            out["w"] = torch.stack(w1, 1)
        out.update(status=None, ncross=None)
        if case["call"] == "trace":
            out.update(path_face=None, path_pt=path, path_len=None)
    else:
        out = {"pos": p1, "face": None, "bary": _bary(M, f1, p1), "dir": d1, "status": None}
        out["grad_v"], out["grad_bary"] = _vjp(M, case, f, t["bary"], t["v"], (f1, p1, d1), t["g"])
        if case.get("grad_V"):
            out["grad_V"] = _grad_V(M, f, t["bary"] / t["bary"].sum(1, keepdim=True), t["v"], t["g"])
    return out


def _exact_field(case, M, f, t):
    K, U, b = case["K"], t["U"], t["bary"]
    h = float(np.float32(1.0 / K))
    steps = []
    for _ in range(K):
        v = h * (b[..., None] * U[M.F[f]]).sum(1)
        p, d, L = _start(M, f, b, v)
        f1, p1, d1, _ = _walk(M, f, p, d, L)
        steps.append((f, b, v, (f1, p1, d1)))
        f, b = f1, _bary(M, f1, p1)
    end = steps[-1][3]
    out = {"pos": end[1], "face": None, "bary": b, "dir": end[2], "status": None}
    gU, g = torch.zeros_like(U), t["g"]
    for f, b, v, e in reversed(steps):
        gv, gb = _vjp(M, case, f, b, v, e, g)
        Fk = M.F[f]
        gU.index_add_(0, Fk.reshape(-1), (h * b.clamp_min(0)[..., None] * gv[:, None]).reshape(-1, 3))
        gb = gb + h * (U[Fk] * gv[:, None]).sum(-1)
        # a gradient in the barycentrics of a point is the tangent gradient with (x_k - x_0).g = g_k - g_0
        P = M.corners(f)
        u, w = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
        uu, uw, ww = _dot(u, u), _dot(u, w), _dot(w, w)
        a, c = gb[:, 1:2] - gb[:, :1], gb[:, 2:] - gb[:, :1]
        det = uu * ww - uw * uw
        g = (ww * a - uw * c) / det * u + (uu * c - uw * a) / det * w
    out.update(grad_bary=gb, grad_U=gU)
    return out
