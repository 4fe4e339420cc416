"""Calls with stream=: everything that a call makes besides its kernels (copies of host inputs, cleared
gradients, scratch) is in order with them on that stream, whatever the current stream is doing.

In the first test the current stream is far behind the given one, in the second far ahead of it, with
tensors of the scratch's sizes taken and overwritten right after each call.
"""
import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu

NQ, K = 70000, 2


def _calls():
    import torch

    import paper_2603_15780_gb300 as sg
    rng = np.random.Generator(np.random.PCG64(12))
    X, F = meshgen.icosphere(5, 0.003, rng)
    q = meshgen.sample_queries(X, F, NQ, rng, 0.1, 1.0, 1)
    f32 = lambda x: np.ascontiguousarray(x, np.float32)
    face, bary, v, w, g = q.face.astype(np.int32), f32(q.bary), f32(q.v), f32(q.w), f32(q.g_pos)
    U = f32(rng.normal(size=X.shape) * 0.2)
    mesh = sg.Mesh(f32(X), F)
    end = sg.exp_map(mesh, face, bary, v, w)
    steps = sg.exp_map_field_steps(mesh, face, bary, U, K)
    back = (mesh, "gfd", face, bary, v, end["face"], end["bary"], end["dir"], end["status"], g)
    torch.cuda.synchronize()
    return torch, {
        "exp_map": lambda **s: sg.exp_map(mesh, face, bary, v, w, want_hash=True, **s),
        "exp_map with an order": lambda **s: sg.exp_map(mesh, face, bary, v, sort=2, precision=32, **s),
        "trace": lambda **s: sg.exp_map_trace(mesh, face, bary, v, path_cap=8, **s),
        "backward": lambda **s: sg.exp_map_backward(*back, want_grad_V=True, eps_v=1e-3, eps_p=1e-3, **s),
        "transport_back": lambda **s: {"u": sg.transport_back(mesh, face, bary, v, end, g, **s)},
        "field": lambda **s: sg.exp_map_field_steps(mesh, face, bary, U, K, **s),
        "field backward": lambda **s: sg.exp_map_field_steps_backward(mesh, "gfd", steps, U, K, 0.5, g, want_grad_V=True, **s),
        "update": lambda **s: {"V": mesh.update_vertices(f32(X), **s), **sg.exp_map(mesh, face, bary, v, **s)},
    }


def _compare(torch, name, out, ref):
    for k, a in out.items():
        if k.startswith("_") or a is None:
            continue
        b = ref[k]
        if k == "path_face" or k == "path_pt":      # (entries past a path's length are not written)
            live = torch.arange(a.shape[1], device="cuda")[None] < ref["path_len"][:, None]
            a, b = a[live], b[live]
        if k in ("grad_V", "grad_U"):               # float32 sums of some hundred terms in any order
            assert float((a - b).abs().max()) <= 1024 * 2.0 ** -24 * float(b.abs().max()), (name, k)
        else:
            assert torch.equal(a, b), (name, k)


@pytest.mark.parametrize("behind", ["current", "given"])
def test_given_stream_keeps_its_own_order(behind):
    torch, calls = _calls()
    side = torch.cuda.Stream()
    for name, call in calls.items():
        ref = call()
        torch.cuda.synchronize()
        sizes = [t.numel() * t.element_size() for t in ref.values() if t is not None]
        if behind == "current":
            torch.cuda._sleep(40_000_000)           # about 20 ms
        else:
            with torch.cuda.stream(side):
                torch.cuda._sleep(40_000_000)
        out = call(stream=side)
        junk = []
        for n in sizes + [4 * NQ, 12 * NQ, 1 << 20, 1 << 22, 8 << 20, 16 << 20, 32 << 20, 64 << 20]:
            junk.append(torch.full((n,), 255, dtype=torch.uint8, device="cuda"))
        side.synchronize()
        torch.cuda.synchronize()
        _compare(torch, (name, behind), out, ref)
