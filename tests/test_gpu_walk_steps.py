"""The hot loop's step (fast_step) against the general one (half_step), which it restates.

The walk kernels take every ordinary crossing by fast_step, so comparing them with each other says
nothing about the two.  Here the same walks run with fast_step and without it (tests/walk_steps.cu, built
by this test) and end in the same state bit for bit, in the FP32 walk and in the mixed walk, with vertex
hits, boundary stops, starts on edges and vertices, step caps and a wide near band among them.
"""
import ctypes as C
import subprocess

import numpy as np
import pytest

import meshgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    from paper_2603_15780_gb300 import build as b
    lib = tmp_path_factory.mktemp("steps") / "libsteps.so"
    nv = b.nvcc()
    subprocess.check_call([nv, "-shared", "-o", str(lib), __file__.replace("test_gpu_walk_steps.py", "walk_steps.cu"), "-O3",
                           "-std=c++17", "-Xcompiler", "-fPIC", *b.ARCH, "-cudart", "shared", "-Xlinker",
                           "-rpath," + b._cuda_lib_dir(nv)])
    f = C.CDLL(str(lib)).walk_steps
    p = C.c_void_p
    f.argtypes = [p, C.c_int, C.c_int, C.c_int64, p, p, p, C.c_int, C.c_float, p, p, p, p, p]
    f.restype = C.c_int
    return f


@pytest.mark.parametrize("tau_near", [1e-4, 1e-2])
@pytest.mark.parametrize("max_steps", [1 << 20, 7])
@pytest.mark.parametrize("mix", [0, 1])
def test_fast_step_restates_half_step(steps, mix, max_steps, tau_near):
    import torch

    import paper_2603_15780_gb300 as sg
    rng = np.random.Generator(np.random.PCG64(21))
    X, F, waves = meshgen.heightfield(60, rng)
    field = (meshgen.jitter_slivers(X, 60, rng, 0.10, waves), F)
    sphere, flat = meshgen.icosphere(5, 0.003, rng), meshgen.flat_grid(24)
    for (X, F), hi, aimed in ((sphere, 6.0, False), (field, 2.0, False), (flat, 1.0, True)):
        n = 20000
        q = meshgen.sample_queries(X, F, n, rng, 0.0, hi, 0)
        bary, v = q.bary.astype(np.float32), q.v.astype(np.float32)
        k = np.arange(n)
        bary[k % 11 == 3] = [0.25, 0.75, 0.0]
        bary[k % 13 == 4] = [1.0, 0.0, 0.0]
        v[k % 17 == 5] = 0.0
        if aimed:                            # at a vertex of the start face, and on
            P = X[F[q.face]].astype(np.float64)
            at = (P * bary[:, :, None]).sum(1)
            v = (4.0 * (P[k, k % 3] - at)).astype(np.float32)
        mesh = sg.Mesh(X.astype(np.float32), F)
        cu = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")
        face, bary, v = cu(q.face.astype(np.int32)), cu(bary), cu(v)
        out = []
        for fast in (1, 0):
            o = [torch.zeros(n, *s, dtype=d, device="cuda") for d, s in
                 ((torch.int32, ()), (torch.int32, ()), (torch.int32, ()), (torch.int64, ()), (torch.float32, (4,)))]
            torch.cuda.synchronize()
            assert steps(mesh.handle, mix, fast, n, face.data_ptr(), bary.data_ptr(), v.data_ptr(), max_steps, tau_near,
                         *(t.data_ptr() for t in o)) == 0
            torch.cuda.synchronize()
            out.append(o)
        if aimed:                            # (a hit vertex passes many walks on along its grid line)
            assert bool(((out[0][2] & sg.ST_VERTEX_HIT) != 0).any())
        else:
            assert int(out[0][1].max()) > (5 if max_steps == 7 else 20)
        for name, a, b in zip(("face", "ncross", "status", "hash", "state"), *out):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), name
