"""What the entry points accept and how they launch: scratch limits, launch options."""
import ctypes as C

import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu

OUT = (("face", "int32", ()), ("bary", "float32", (3,)), ("pos", "float32", (3,)), ("dir", "float32", (3,)),
       ("status", "int32", ()), ("ncross", "int32", ()), ("hash", "int64", ()))


def _outputs(n):
    import torch
    return {k: torch.zeros((n, *s), dtype=getattr(torch, d), device="cuda") for k, d, s in OUT}


def _call(fn, mesh, face, bary, v, opts, out, stream=None):
    """sg_exp_map or sg_exp_map_noalloc into `out`; the status."""
    p = lambda k: out[k].data_ptr()
    return fn(mesh.handle, face.numel(), None, face.data_ptr(), bary.data_ptr(), v.data_ptr(), None, 0, None, p("face"),
              p("bary"), p("pos"), p("dir"), None, p("status"), p("ncross"), p("hash"), C.byref(opts), stream)


def _inputs(X, F, n, lo, hi, seed=5):
    import torch

    import paper_2603_15780_gb300 as sg
    rng = np.random.Generator(np.random.PCG64(seed))
    q = meshgen.sample_queries(X, F, n, rng, lo, hi, 0)
    cu = lambda x: torch.as_tensor(np.ascontiguousarray(x, np.float32), device="cuda")
    return sg, sg.Mesh(X.astype(np.float32), F), (torch.as_tensor(q.face, device="cuda"), cu(q.bary), cu(q.v))


def _kernels(launch):
    """(grid, block) of each kernel that `launch(stream)` enqueues, from a stream capture (nothing runs)."""
    import torch

    class Params(C.Structure):
        _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("shared", C.c_uint),
                    ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]
    cu = C.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    stream, graph, n, kind = C.c_void_p(s.cuda_stream), C.c_void_p(), C.c_size_t(), C.c_int()
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(stream, C.c_int(2)) == 0       # (relaxed)
    try:
        rc = launch(s.cuda_stream)
    finally:
        end = cu.cuStreamEndCapture(stream, C.byref(graph))
    assert rc == 0 and end == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, C.byref(n)) == 0
    out = []
    for x in nodes:
        assert cu.cuGraphNodeGetType(C.c_void_p(x), C.byref(kind)) == 0
        if kind.value == 0:
            k = Params()
            assert cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(x), C.byref(k)) == 0
            out.append((k.grid[0], k.block[0]))
    cu.cuGraphDestroy(graph)
    return out


@pytest.mark.parametrize("n,fits", [(7_200_000, True), (7_900_000, False)])
def test_noalloc_takes_fp64_batches_of_the_start_face_order(n, fits):
    """On 600,000 faces the 32 MiB hold the length order (5 bytes a query) of 6.7M queries and the
    start-face order (4 bytes a query and a face) of 7.8M: between the two the FP64 walk falls back to the
    second."""
    import torch
    X, F = meshgen.torus(600, 500)
    sg, mesh, few = _inputs(X, F, 4000, 0.0, 0.01)
    face, bary, v = (x.repeat(n // 4000, *[1] * (x.dim() - 1)).contiguous() for x in few)
    out = _outputs(n)
    rc = _call(sg.lib().sg_exp_map_noalloc, mesh, face, bary, v, sg.default_opts(precision=64), out)
    assert rc == (0 if fits else 5)                                   # 5: SG_ERR_OOM
    torch.cuda.synchronize()
    if not fits:
        assert not bool(out["hash"].any())                            # nothing was launched
        return
    ref = sg.exp_map(mesh, *few, precision=64, want_hash=True)
    torch.cuda.synchronize()
    for k, _, s in OUT:
        a = out[k].reshape(n // 4000, 4000, *s)
        assert torch.equal(a, ref[k].reshape(1, 4000, *s).expand_as(a)), k


@pytest.mark.parametrize("precision", [48, 64])
def test_wide_walk_keeps_the_residency_it_is_given(precision):
    """blocks_per_sm counts blocks of 128 threads at every batch size."""
    import torch
    X, F = meshgen.icosphere(2)
    sg, mesh, q = _inputs(X, F, 20000, 0.0, 0.1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out, ws = _outputs(20000), torch.empty(4096, dtype=torch.uint8, device="cuda")
    for per in (1, 2):
        opts = sg.default_opts(precision=precision, sort=0, blocks_per_sm=per, workspace=ws.data_ptr(), workspace_bytes=4096)
        got = _kernels(lambda s: _call(sg.lib().sg_exp_map, mesh, *q, opts, out, s))
        assert got == [(min(sms * per, -(-20000 // 128)), 128)]


@pytest.mark.parametrize("block,want", [(32, 32), (64, 64), (128, 128), (192, 192), (256, 128), (0, 128)])
def test_small_batch_launches_the_block_it_is_given(block, want):
    """(256 is the default options' value: the library's own choice.  Above 128 threads the walk that goes
    on in the mixed arithmetic is a second launch.)"""
    import torch
    X, F = meshgen.icosphere(2)
    sg, mesh, q = _inputs(X, F, 1000, 0.0, 1.0)
    ref = sg.exp_map(mesh, *q, want_hash=True)
    opts = sg.default_opts(block=block)
    out = _outputs(1000)
    got = _kernels(lambda s: _call(sg.lib().sg_exp_map, mesh, *q, opts, out, s))
    assert got[0] == (-(-1000 // want), want) and len(got) == (2 if want > 128 else 1)
    rc = _call(sg.lib().sg_exp_map, mesh, *q, opts, out)
    torch.cuda.synchronize()
    assert rc == 0 and all(torch.equal(out[k], ref[k]) for k, _, _ in OUT)


def test_small_batch_refuses_a_workspace_that_is_too_small():
    import torch
    X, F = meshgen.icosphere(2)
    sg, mesh, q = _inputs(X, F, 1000, 0.0, 1.0)
    need = sg.workspace_size(mesh, 1000, sg.default_opts())
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    for size, want in ((need, 0), (need - 1, 5), (64, 5)):
        out = _outputs(1000)
        rc = _call(sg.lib().sg_exp_map, mesh, *q, sg.default_opts(workspace=ws.data_ptr(), workspace_bytes=size), out)
        torch.cuda.synchronize()
        assert rc == want and bool(out["hash"].any()) == (want == 0)
