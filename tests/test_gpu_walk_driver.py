"""The persistent walks (hot loop and service phase) against the one-thread-per-query kernel.

Both run the same steps in the same arithmetic, so every output is equal bit for bit, whatever lanes
a query shares its warp with: batches around a warp, a block and a full grid, and with starts on
edges and vertices, invalid queries, zero lengths, boundary stops and low step caps among them.
"""
import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu


def _mesh_and_queries(n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    X, F, waves = meshgen.heightfield(40, rng)
    X = meshgen.jitter_slivers(X, 40, rng, 0.10, waves)
    q = meshgen.sample_queries(X, F, n, rng, 0.0, 0.8, 1)
    k = np.arange(n)
    q.bary[k % 11 == 3] = [0.25, 0.75, 0.0]          # on an edge
    q.bary[k % 13 == 4] = [1.0, 0.0, 0.0]            # on a vertex (half of them point out of the face)
    q.v[k % 17 == 5] = 0.0
    q.face[k % 19 == 6] = len(F)                     # no such face
    q.v[k % 23 == 7] *= np.nan
    return X, F, q


@pytest.mark.parametrize("max_steps", [0, 5])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 5000])
def test_persistent_equals_plain(n, max_steps):
    import torch

    import paper_2603_15780_gb300 as sg
    X, F, q = _mesh_and_queries(n, 11 + n)
    mesh = sg.Mesh(X.astype(np.float32), F)
    args = (mesh, q.face, q.bary.astype(np.float32), q.v.astype(np.float32), q.w.astype(np.float32))
    kw = {"want_hash": True, "precision": 32, "max_steps": max_steps or None}
    a = sg.exp_map(*args, **kw)                                        # small batch: one thread per query
    b = sg.exp_map(*args, kernel=sg.KERNEL_PERSISTENT, **kw)
    c = sg.exp_map(*args, kernel=sg.KERNEL_PERSISTENT, queries_per_thread=8, block=32, blocks_per_sm=1, sort=2, **kw)
    torch.cuda.synchronize()
    for o in (b, c):
        for k in ("face", "bary", "pos", "dir", "w", "status", "ncross", "hash"):
            assert torch.equal(a[k].view(torch.uint8), o[k].view(torch.uint8)), k


def test_grid_takes_many_tasks_per_lane():
    """Each lane takes many queries in turn (the first ticket is not a lane's only one)."""
    import torch

    import paper_2603_15780_gb300 as sg
    X, F, q = _mesh_and_queries(40000, 5)
    mesh = sg.Mesh(X.astype(np.float32), F)
    args = (mesh, q.face, q.bary.astype(np.float32), q.v.astype(np.float32), q.w.astype(np.float32))
    a = sg.exp_map(*args, want_hash=True, precision=32)
    b = sg.exp_map(*args, want_hash=True, precision=32, kernel=sg.KERNEL_PERSISTENT, block=32, blocks_per_sm=1)
    torch.cuda.synchronize()
    for k in ("face", "bary", "pos", "dir", "w", "status", "ncross", "hash"):
        assert torch.equal(a[k].view(torch.uint8), b[k].view(torch.uint8)), k


@pytest.mark.parametrize("precision", [40, 48, 64])
@pytest.mark.parametrize("n", [33, 1023, 1024, 1500])
def test_wide_walks_do_not_depend_on_the_order(n, precision):
    """The FP64 walk takes batches of 1024 queries and more in length order and in one-warp blocks."""
    import torch

    import paper_2603_15780_gb300 as sg
    X, F, q = _mesh_and_queries(n, 3 + n)
    mesh = sg.Mesh(X.astype(np.float32), F)
    args = (mesh, q.face, q.bary.astype(np.float32), q.v.astype(np.float32), q.w.astype(np.float32))
    a = sg.exp_map(*args, want_hash=True, precision=precision, sort=0, blocks_per_sm=1)
    for kw in ({}, {"sort": 2}, {"sort": 1}):
        b = sg.exp_map(*args, want_hash=True, precision=precision, **kw)
        torch.cuda.synchronize()
        for k in ("face", "bary", "pos", "dir", "w", "status", "ncross", "hash"):
            assert torch.equal(a[k].view(torch.uint8), b[k].view(torch.uint8)), (k, kw)


def test_update_of_a_batch_keeps_each_mesh():
    """Edge lengths are summed per block: blocks of one mesh, and blocks that meet two."""
    import torch

    import paper_2603_15780_gb300 as sg
    rng = np.random.Generator(np.random.PCG64(9))
    meshes = [meshgen.icosphere(2), meshgen.flat_grid(9), meshgen.icosphere(1), meshgen.torus(20, 11)]
    for scale in (1.0, 3.0):
        Vs = [(X * scale * (1 + i)).astype(np.float32) for i, (X, _) in enumerate(meshes)]
        made = sg.Mesh([(V, F) for V, (_, F) in zip(Vs, meshes)])
        moved = sg.Mesh([(X.astype(np.float32), F) for X, F in meshes])
        moved.update_vertices(torch.as_tensor(np.concatenate(Vs), device="cuda"))
        assert abs(made.info().l_ref_mean - moved.info().l_ref_mean) <= 1e-12 * made.info().l_ref_mean
        ids = rng.integers(0, len(meshes), 500).astype(np.int32)
        qs = [meshgen.sample_queries(V.astype(np.float64), F, 500, rng, 0.1, 2.0, 0) for V, (_, F) in zip(Vs, meshes)]
        pick = lambda f: np.stack([getattr(qs[m], f)[i] for i, m in enumerate(ids)])
        args = (pick("face").astype(np.int32), pick("bary").astype(np.float32), pick("v").astype(np.float32))
        a, b = (sg.exp_map(m, *args, mesh_id=ids) for m in (made, moved))
        torch.cuda.synchronize()
        assert torch.equal(a["face"], b["face"]) and torch.equal(a["ncross"], b["ncross"])
        assert torch.equal(a["status"], b["status"])
        assert torch.allclose(a["pos"], b["pos"], rtol=0, atol=1e-6 * 10)


@pytest.mark.parametrize("n", [1, 127, 129, 3000])
@pytest.mark.parametrize("max_steps", [0, 300])
def test_small_batches_of_the_automatic_precision(n, max_steps):
    """One launch for a small batch, with the mixed walks in their queries' own threads: each query's
    outputs are those of the mixed walk where its status says so, else of the FP32 walk -- queries that
    are too long for FP32 at the start, and (long thin triangles: more crossings per mean edge length)
    ones that reach the crossing budget."""
    import torch

    import paper_2603_15780_gb300 as sg
    X, F = meshgen.torus(200, 8)
    rng = np.random.Generator(np.random.PCG64(n))
    q = meshgen.sample_queries(X, F, n, rng, 0.0, 25.0, 2)
    q.v[np.arange(n) % 7 == 3] *= 0.05
    mesh = sg.Mesh(X.astype(np.float32), F)
    args = (mesh, q.face, q.bary.astype(np.float32), q.v.astype(np.float32), q.w.astype(np.float32))
    kw = {"want_hash": True, "max_steps": max_steps or None}
    a = sg.exp_map(*args, **kw)
    fp32 = sg.exp_map(*args, precision=32, **kw)
    wide = sg.exp_map(*args, precision=40, **kw)
    torch.cuda.synchronize()
    mixed = (a["status"] & sg.ST_MIXED) != 0
    for k in ("face", "bary", "pos", "dir", "w", "status", "ncross", "hash"):
        m = mixed.reshape(-1, *[1] * (a[k].dim() - 1))
        assert torch.equal(a[k].view(torch.uint8), torch.where(m, wide[k], fp32[k]).view(torch.uint8)), k
    long = torch.as_tensor(np.linalg.norm(q.v, axis=1), device="cuda") > 96 * mesh.info().l_ref_mean
    assert torch.equal(mixed, long | (fp32["ncross"] >= 256))
    if n == 3000:
        assert bool((mixed & long).any()) and bool((mixed & ~long).any()) and bool((~mixed).any())
