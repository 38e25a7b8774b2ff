"""The workspace of FP32 plans does not grow with the columns they solve in double-float.

A Helmholtz shift beyond every coupling leaves no such column; the workspace must be the same
without it, so that a plan fits the fixed array of ps_solve_static (8 MiB) by its number of cells
alone. Grids just under that, and one with y lines solved on transposed planes; the solve through
the fixed array (FP32 fields: a workspace filled anew) must give the same bits.
"""

import ctypes

import pytest

from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu

GRIDS = [(48, 64, 130, ("P", "NN", "DD"), 6.0), (36, 36, 314, ("DD", "DN", "ND"), 1.0),
         (648, 6, 105, ("DD", "DD", "ND"), 6.0), (24, 96, 12, ("NN", "DN", "NN"), 1.0),
         (2, 2048, 96, ("NN", "P", "DD"), 6.0), (32, 384, 17, ("NN", "NN", "NN"), 6.0)]


@pytest.mark.parametrize("precision", ["fp32", "fp32_refine"])
@pytest.mark.parametrize("nx,ny,nz,bcs,lx", GRIDS)
def test_workspace_without_the_rectangle(lib, nx, ny, nz, bcs, lx, precision):
    import torch
    kw = dict(zf=synth.tanh_faces(nz, 1.0, 1.5), bcs=bcs, precision=precision)
    plan = lib.Plan(nx, ny, nz, lx / nx, 1.0 / ny, **kw)
    bare = lib.Plan(nx, ny, nz, lx / nx, 1.0 / ny, alpha=1e12, **kw)
    assert plan.workspace_bytes == bare.workspace_bytes <= 8 << 20
    bare.close()
    dt = torch.float32 if precision == "fp32" else torch.float64
    f = torch.randn((nz, ny, nx), generator=torch.Generator("cuda").manual_seed(3), device="cuda", dtype=dt)
    if all(b in ("P", "NN") for b in bcs):
        f -= f.mean()
    p, q = plan.solve(f), torch.empty_like(f)
    if precision == "fp32":  # (the fixed array serves FP64 fields)
        plan.workspace().fill_(0x7F)
        plan.solve(f, out=q)
    else:
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())
        lib._check(lib.ps_solve_static(plan.handle, ptr(f), ptr(q), lib._stream_ptr(None), None), plan.handle)
    torch.cuda.synchronize()
    plan.close()
    assert torch.equal(p, q)
