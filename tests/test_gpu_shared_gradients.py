"""Gradients that are accumulated into the caller's array, from calls on several streams at once."""
import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu

STREAMS, CALLS = 4, 40


def _setup(level=6, nq=64):
    import torch

    import paper_2603_15780_gb300 as sg
    rng = np.random.Generator(np.random.PCG64(8))
    X, F = meshgen.icosphere(level)      # many vertices and few queries: the last additions overlap
    q = meshgen.sample_queries(X, F, nq, rng, 0.1, 0.5, 0)
    cu = lambda x: torch.as_tensor(np.ascontiguousarray(x, np.float32), device="cuda")
    return torch, sg, sg.Mesh(X.astype(np.float32), F), q, cu, rng


def _check(torch, one, shared, calls):
    """`calls` equal terms: each of the additions rounds to half an ulp of a partial sum, at most `calls`
    times the term; a lost term is 1 / calls of the sum.  The term itself, a sum of up to some 100 float32
    contributions in any order, may differ from call to call by its own rounding."""
    scale = float(one.abs().max())
    tol = (0.5 * calls * calls + 128 * calls) * 2.0 ** -24 * scale
    assert tol < 0.05 * scale
    assert float((shared.double() - calls * one.double()).abs().max()) <= tol


def test_field_gradient_shared_by_streams():
    torch, sg, mesh, q, cu, rng = _setup()
    U, g, K = cu(rng.normal(size=(mesh.n_vertices, 3))) * 0.2, cu(q.g_pos), 2
    fwd = sg.exp_map_field_steps(mesh, q.face, cu(q.bary), U, K)

    def call(grad_U):
        return sg.exp_map_field_steps_backward(mesh, "ep", fwd, U, K, 1.0 / K, g, grad_U=grad_U)

    one, shared = torch.zeros_like(U), torch.zeros_like(U)
    call(one)
    torch.cuda.synchronize()
    assert float(one.abs().max()) > 0
    streams, keep = [torch.cuda.Stream() for _ in range(STREAMS)], []
    for i in range(CALLS):
        for s in streams:
            with torch.cuda.stream(s):
                keep.append(call(shared))
    torch.cuda.synchronize()
    _check(torch, one, shared, STREAMS * CALLS)


@pytest.mark.parametrize("estimator", ["ep", "gfd"])
def test_vertex_gradient_shared_by_streams(estimator):
    torch, sg, mesh, q, cu, _ = _setup()
    face, bary, v, g = torch.as_tensor(q.face, device="cuda"), cu(q.bary), cu(q.v), cu(q.g_pos)
    end = sg.exp_map(mesh, face, bary, v)

    def call(grad_V):
        return sg.exp_map_backward(mesh, estimator, face, bary, v, end["face"], end["bary"], end["dir"], end["status"], g,
                                   grad_V=grad_V)

    one, shared = (torch.zeros(mesh.n_vertices, 3, device="cuda") for _ in range(2))
    call(one)
    torch.cuda.synchronize()
    assert float(one.abs().max()) > 0
    streams, keep = [torch.cuda.Stream() for _ in range(STREAMS)], []
    for i in range(CALLS):
        for s in streams:
            with torch.cuda.stream(s):
                keep.append(call(shared))
    torch.cuda.synchronize()
    _check(torch, one, shared, STREAMS * CALLS)
