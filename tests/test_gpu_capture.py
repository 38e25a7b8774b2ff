"""Solves captured in a CUDA graph, and in a chain on one stream.

The kernels of a solve are launched so that each may start before the one ahead of it has
ended (it waits for that one's completion before it touches the fields). A captured solve, and
solves that follow one another on a stream with other kernels between them (writing the next
right-hand side into the same buffer), give bit for bit what single synchronised solves give.
"""

import numpy as np
import pytest

from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = [((64, 128, 256), "fp32_refine"), ((40, 48, 96), "fp32_refine"), ((64, 128, 128), "fp64"), ((33, 36, 54), "fp64"),
         ((48, 128, 128), "fp32"), ((4, 2048, 32), "fp32_refine")]


@pytest.mark.parametrize("shape,precision", CASES, ids=["x".join(map(str, s)) + "-" + p for s, p in CASES])
def test_chained_and_captured_solves_match_single_ones(lib, shape, precision):
    import torch
    nz, ny, nx = shape
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    plan = lib.Plan(nx, ny, nz, 6.0 / nx, 3.0 / ny, zf=zf, bcs=("P", "NN", "NN"), precision=precision,
                    rtol=1e-10, max_iter=4)
    dt = torch.float32 if precision == "fp32" else torch.float64
    fs = [torch.as_tensor(synth.uniform_noise(shape, seed=s), device="cuda").to(dt) for s in range(4)]
    want = []
    for f in fs:
        want.append(plan.solve(f))
        torch.cuda.synchronize()
    g, p, info = torch.empty_like(fs[0]), torch.empty_like(fs[0]), lib.info_tensor()
    got = []
    for f in fs + fs[::-1]:  # one stream, no synchronisation, the same buffers
        g.copy_(f)
        plan.solve(g, out=p, info=info)
        got.append(p.clone())
    torch.cuda.synchronize()
    for a, b in zip(got, want + want[::-1]):
        assert torch.equal(a, b)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.solve(g, out=p, info=info)
    for f, b in zip(fs, want):
        g.copy_(f)
        p.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(p, b)
    plan.close()
