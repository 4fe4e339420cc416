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
    small = torch.empty(256, dtype=torch.uint8, device="cuda")     # no room for an order: taken all the same
    for kw in ({}, {"sort": 2}, {"sort": 1}, {"workspace": small}):
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


@pytest.mark.parametrize("n", [150, 182, 183])   # 44,402, 65,522 and 66,248 faces: around the far walks' line
def test_start_face_order_with_far_walks(n):
    """Walks of up to 3,000 mean edge lengths: each query's outputs are those of the walk that its status
    names, wherever the order puts it."""
    import torch

    import paper_2603_15780_gb300 as sg
    rng = np.random.Generator(np.random.PCG64(n))
    X, F = meshgen.torus(n - 1, n - 1) if n > 150 else meshgen.torus(149, 149)
    q = meshgen.sample_queries(X, F, 3001, rng, 0.0, 1.0, 0)
    mesh = sg.Mesh(X.astype(np.float32), F)
    q.v *= (mesh.info().l_ref_mean * 10.0 ** rng.uniform(-1.0, 3.5, 3001))[:, None]
    q.face[::97] = len(F)
    args = (mesh, q.face, q.bary.astype(np.float32), q.v.astype(np.float32))
    a = sg.exp_map(*args, sort=1, kernel=sg.KERNEL_PERSISTENT, want_hash=True)
    fp32 = sg.exp_map(*args, precision=32, want_hash=True)
    wide = sg.exp_map(*args, precision=40, want_hash=True)
    torch.cuda.synchronize()
    mixed = (a["status"] & sg.ST_MIXED) != 0
    assert bool(mixed.any()) and not bool(mixed.all())
    for k in ("face", "bary", "pos", "dir", "status", "ncross", "hash"):
        m = mixed.reshape(-1, *[1] * (a[k].dim() - 1))
        assert torch.equal(a[k].view(torch.uint8), torch.where(m, wide[k], fp32[k]).view(torch.uint8)), k


def test_field_gradient_with_and_without_the_accumulator():
    """A workspace without room for the accumulator is still accepted; both ways sum the same terms."""
    import ctypes as C

    import torch

    import paper_2603_15780_gb300 as sg
    X, F = meshgen.icosphere(3)
    rng = np.random.Generator(np.random.PCG64(4))
    q = meshgen.sample_queries(X, F, 3001, rng, 0.0, 1.0, 0)
    mesh, K, nq = sg.Mesh(X.astype(np.float32), F), 3, 3001
    cu = lambda x: torch.as_tensor(np.asarray(x, np.float32), device="cuda")
    U, g = cu(rng.normal(size=X.shape)), cu(q.g_pos)
    fwd = sg.exp_map_field_steps(mesh, q.face, q.bary.astype(np.float32), U, K)
    n = C.c_size_t()
    assert sg.lib().sg_exp_map_steps_backward_workspace_size(mesh.handle, sg.EST_GFD, K, nq, 0, C.byref(n)) == 0
    room = (16 * len(X) + 255) // 256 * 256
    out = []
    for size in (n.value, n.value - room, n.value - room - 1):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        o = sg.default_opts(workspace=ws.data_ptr(), workspace_bytes=size)
        gU, gb = torch.ones_like(U), torch.empty(nq, 3, device="cuda")
        p = lambda x: x.data_ptr()
        rc = sg.lib().sg_exp_map_steps_backward(
            mesh.handle, sg.EST_GFD, 1e-3, 1e-3, K, 1.0 / K, p(U), nq, None, p(fwd["step_face"]), p(fwd["step_bary"]),
            p(fwd["step_v"]), p(fwd["step_dir"]), p(fwd["step_status"]), p(g), None, p(gU), p(gb), None, C.byref(o),
            torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        out.append((rc, gU.double(), gb))
    assert [r[0] for r in out] == [0, 0, 5]   # the last: SG_ERR_OOM
    assert torch.equal(out[0][2], out[1][2])
    # about 3001 * 3 * 3 / 642 terms a vertex, summed in float32 in another order
    scale = float(out[1][1].abs().max())
    assert float((out[0][1] - out[1][1]).abs().max()) <= 64 * 2.0 ** -24 * scale
