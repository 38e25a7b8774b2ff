"""The projection operators' vector and scalar rows agree bit for bit.

With 16-byte aligned fields and n_x a multiple of the vector they move 16 bytes a thread,
otherwise one value. The same field at an address one value off, and row lengths on both sides
of the thread rows (a warp, less than a warp, several passes), must give the same bits; one
shape of each precision is also compared with the oracle's matrices to rounding.
"""

import ctypes

import numpy as np
import pytest

from oracle import adjoint as A
from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx,ny,nz", [(8, 4, 3), (48, 6, 5), (128, 2, 2), (144, 4, 3), (288, 6, 4)])
@pytest.mark.parametrize("bcs", [("P", "P", "NN"), ("NN", "NN", "P"), ("NN", "P", "NN")])
def test_operator_rows(lib, precision, nx, ny, nz, bcs):
    import torch
    dt = torch.float32 if precision == "fp32" else torch.float64
    zf = synth.uniform_faces(nz, 1.0) if bcs[2] == "P" else synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 6.0 / nx, 3.0 / ny
    plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=bcs, precision=precision)
    st = lib._stream_ptr(None)
    n = nx * ny * nz
    g = torch.Generator(device="cuda").manual_seed(1)
    u = torch.randn(3 * n, generator=g, device="cuda", dtype=dt)
    p = torch.randn(n, generator=g, device="cuda", dtype=dt)

    def off(t):  # the same values at an address one value off
        b = torch.empty(t.numel() + 1, device="cuda", dtype=dt)
        b[1:] = t
        return b[1:]

    def run(u, p, new):
        f, w, h, d = new(torch.zeros(n, device="cuda", dtype=dt)), new(torch.zeros_like(u)), \
            new(torch.zeros(n, device="cuda", dtype=dt)), new(torch.zeros_like(u))
        assert lib.ps_div(plan.handle, _ptr(u), _ptr(f), st) == 0
        assert lib.ps_grad_correct(plan.handle, _ptr(u), _ptr(p), _ptr(w), st) == 0
        assert lib.ps_grad_adjoint(plan.handle, _ptr(u), _ptr(h), st) == 0
        assert lib.ps_div_adjoint_correct(plan.handle, _ptr(u), _ptr(p), _ptr(d), st) == 0
        torch.cuda.synchronize()
        return f, w, h, d

    a, b = run(u, p, lambda t: t), run(off(u), off(p), off)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    plan.close()
    D = A.divergence_matrix(nx, ny, dx, dy, zf, *bcs)
    G = A.gradient_matrix(nx, ny, dx, dy, zf, *bcs)
    U, P = u.double().cpu().numpy(), p.double().cpu().numpy()
    eps = 1e-6 if precision == "fp32" else 1e-14
    for x, ref in zip(a, (D @ U, U - G @ P, G.T @ U, U - D.T @ P)):
        assert np.abs(x.double().cpu().numpy() - ref).max() <= 16 * eps * np.abs(ref).max()
