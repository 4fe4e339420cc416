"""A vertex update re-derives every record of the mesh on its own stream, so that ordering later calls
after the update is all that a caller has to do: on any number of streams, and in captured graphs that
hold the update or the walks but not both.

The walks are those that read the FP64 and double-float records (the automatic precision's long walks,
the mixed, double-float and FP64 walks, the GFD backward of mixed walks); results are compared bit for bit
with the same calls made when the device is idle.
"""
import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu

KEYS = ("face", "bary", "pos", "dir", "status", "ncross", "hash")


def _setup(n, level=4, seed=3):
    import torch

    import paper_2603_15780_gb300 as sg
    rng = np.random.Generator(np.random.PCG64(seed))
    X, F = meshgen.icosphere(level)
    q = meshgen.sample_queries(X, F, n, rng, 0.0, 9.0, 0)      # up to some 130 mean edge lengths
    mesh = sg.Mesh(X.astype(np.float32), F)
    cu = lambda x: torch.as_tensor(np.ascontiguousarray(x, np.float32), device="cuda")
    move = cu(X * (1.0 + 0.2 * np.sin(5.0 * X[:, :1])))
    return torch, sg, mesh, (torch.as_tensor(q.face, device="cuda"), cu(q.bary), cu(q.v)), cu(X), move


def _same(a, b, what):
    import torch
    for k in KEYS:
        assert torch.equal(a[k].view(torch.uint8), b[k].view(torch.uint8)), (what, k)


@pytest.mark.parametrize("precision", [0, 40, 48, 64])
def test_a_captured_walk_follows_a_later_update(precision):
    torch, sg, mesh, args, _, move = _setup(2000)
    ws = torch.empty(sg.workspace_size(mesh, 2000, sg.default_opts(precision=precision)), dtype=torch.uint8, device="cuda")
    walk = lambda: sg.exp_map(mesh, *args, precision=precision, want_hash=True, workspace=ws)
    before = walk()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = walk()
    mesh.update_vertices(move)
    graph.replay()
    torch.cuda.synchronize()
    now = walk()
    torch.cuda.synchronize()
    _same(out, now, precision)
    assert not torch.equal(before["pos"], now["pos"])


@pytest.mark.parametrize("precision", [0, 40, 48, 64])
def test_a_capture_after_an_update_leaves_nothing_undone(precision):
    """A call that is only captured must not count as the one that brought the records up to date."""
    torch, sg, mesh, args, _, move = _setup(2000)
    fresh = sg.Mesh(move.cpu().numpy(), mesh.F)
    ws = torch.empty(sg.workspace_size(mesh, 2000, sg.default_opts(precision=precision)), dtype=torch.uint8, device="cuda")
    walk = lambda m: sg.exp_map(m, *args, precision=precision, want_hash=True, workspace=ws)
    walk(mesh)
    mesh.update_vertices(move)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        walk(mesh)
    now, ref = walk(mesh), walk(fresh)
    torch.cuda.synchronize()
    # a mesh made from the moved vertices: sums of angles and edge lengths in another order
    assert torch.equal(now["face"], ref["face"]) and torch.equal(now["hash"], ref["hash"])
    assert float((now["pos"] - ref["pos"]).abs().max()) <= 1e-5


def test_a_captured_update_counts_at_each_replay():
    torch, sg, mesh, args, start, move = _setup(2000)
    V = start.clone()
    mesh.update_vertices(V)                                  # (the first update allocates its scratch)
    walk = lambda: sg.exp_map(mesh, *args, precision=40, want_hash=True)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mesh.update_vertices(V)
    first = walk()
    V.copy_(move)
    graph.replay()
    moved = walk()
    mesh.update_vertices(move)
    ref = walk()
    torch.cuda.synchronize()
    _same(moved, ref, "replayed update")
    assert not torch.equal(first["pos"], moved["pos"])


def test_walks_on_two_streams_after_one_update():
    """Both streams wait for the update and for nothing else."""
    torch, sg, mesh, args, start, move = _setup(20000, level=6)
    face, bary, v = args
    streams = [torch.cuda.Stream() for _ in range(3)]
    g = torch.randn(len(face), 3, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))

    def calls(V, kind):
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[0]):
            mesh.update_vertices(V)
            done = torch.cuda.Event()
            done.record()
        out = []
        for s in streams[1:]:
            s.wait_event(done)
            with torch.cuda.stream(s):
                if kind == "gfd":
                    o = {"end": end}
                    r = sg.exp_map_backward(mesh, "gfd", face, bary, v, end["face"], end["bary"], end["dir"], end["status"],
                                            g, eps_v=1e-3, eps_p=1e-3)
                    o.update({k: r[k] for k in ("grad_v", "grad_p", "status")})
                else:
                    o = sg.exp_map(mesh, face, bary, v, precision=kind, want_hash=True)
                out.append(o)
        torch.cuda.synchronize()
        return out

    for kind in (0, 40, 48, "gfd"):
        for V in (move, start, move):
            if kind == "gfd":
                mesh.update_vertices(V)
                end = sg.exp_map(mesh, face, bary, v)
                assert bool(((end["status"] & sg.ST_MIXED) != 0).any())
                mesh.update_vertices(start if V is move else move)
            out = calls(V, kind)
            if kind == "gfd":
                ref = sg.exp_map_backward(mesh, "gfd", face, bary, v, end["face"], end["bary"], end["dir"], end["status"], g,
                                          eps_v=1e-3, eps_p=1e-3)
            else:
                ref = sg.exp_map(mesh, face, bary, v, precision=kind, want_hash=True)
            torch.cuda.synchronize()
            for o in out:
                for k in KEYS if kind != "gfd" else ("grad_v", "grad_p", "status"):
                    assert torch.equal(o[k].view(torch.uint8), ref[k].view(torch.uint8)), (kind, k)


def test_mesh_info_waits_for_an_update_on_another_stream():
    torch, sg, mesh, args, start, move = _setup(2000, level=6)
    made = {id(V): sg.Mesh(V.cpu().numpy(), mesh.F).info().l_ref_mean for V in (start, move)}
    flat = torch.zeros_like(start)
    s = torch.cuda.Stream()
    mesh.update_vertices(start)
    torch.cuda.synchronize()
    for V in (move, start, move):
        with torch.cuda.stream(s):
            for _ in range(20):                      # enough work ahead of the last update
                mesh.update_vertices(flat)
            mesh.update_vertices(V)
        info = mesh.info()
        assert info.n_degenerate == 0
        assert abs(info.l_ref_mean - made[id(V)]) <= 1e-12 * made[id(V)]
