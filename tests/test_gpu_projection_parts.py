"""The projection operators on rows taken whole, in two parts and in parts of one vector a thread
(by the number of rows), against plain FP64 tensor arithmetic, to rounding as in the row test."""

import ctypes

import numpy as np
import pytest

from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny,nz", [(96, 512, 200), (1024, 36, 134), (972, 64, 70), (3072, 4, 2), (2, 54, 3)])
def test_operators_match_plain_arithmetic(lib, precision, nx, ny, nz):
    import torch
    dt, eps = (torch.float32, 1e-6) if precision == "fp32" else (torch.float64, 1e-14)
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 6.0 / nx, 3.0 / ny
    plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=("P", "NN", "NN"), precision=precision)
    st = lib._stream_ptr(None)
    g = torch.Generator(device="cuda").manual_seed(1)
    u = torch.randn((3, nz, ny, nx), generator=g, device="cuda", dtype=dt)
    p = torch.randn((nz, ny, nx), generator=g, device="cuda", dtype=dt)
    f, w, h, d = torch.empty_like(p), torch.empty_like(u), torch.empty_like(p), torch.empty_like(u)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    assert lib.ps_div(plan.handle, ptr(u), ptr(f), st) == 0
    assert lib.ps_grad_correct(plan.handle, ptr(u), ptr(p), ptr(w), st) == 0
    assert lib.ps_grad_adjoint(plan.handle, ptr(u), ptr(h), st) == 0
    assert lib.ps_div_adjoint_correct(plan.handle, ptr(u), ptr(p), ptr(d), st) == 0
    torch.cuda.synchronize()
    plan.close()

    # x periodic, walls on y and z: the wall face 0 of their components takes no part
    dz = torch.as_tensor(np.diff(zf), device="cuda")[:, None, None]
    dc = torch.cat([dz[:1], 0.5 * (dz[1:] + dz[:-1])])  # distance to the cell below (row 0: a wall)
    U, P = u.double(), p.double()
    wall = [torch.ones(1, 1, 1, dtype=torch.float64, device="cuda"),
            (torch.arange(ny, device="cuda") > 0).double()[None, :, None],
            (torch.arange(nz, device="cuda") > 0).double()[:, None, None]]
    axis, width, dist = (2, 1, 0), (dx, dy, dz), (dx, dy, dc)
    up = lambda a, ax: torch.roll(a, -1, ax)
    dn = lambda a, ax: torch.roll(a, 1, ax)
    face = [U[c] * wall[c] for c in range(3)]  # (the face above a last cell is the wrapped, zeroed one)
    div = sum((up(face[c], axis[c]) - face[c]) / width[c] for c in range(3))
    grad = torch.stack([wall[c] * (P - dn(P, axis[c])) / dist[c] for c in range(3)])
    gt = sum(face[c] / dist[c] - up(face[c] / dist[c], axis[c]) for c in range(3))
    dtr = torch.stack([wall[c] * (dn(P / width[c], axis[c]) - P / width[c]) for c in range(3)])
    for x, ref in ((f, div), (w, U - grad), (h, gt), (d, U - dtr)):
        assert (x.double() - ref).abs().max() <= 16 * eps * ref.abs().max()
