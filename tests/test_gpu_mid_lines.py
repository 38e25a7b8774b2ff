"""The FP32 line kernels with the length at compile time, where the other tests do not reach.

* Every half length with each boundary pair on each axis (the pairs of lengths and two
  combinations of test_gpu_generic_lines, here the other three).
* The transpose solve, which multiplies rows by a factor of their plane on load and on store,
  with tiles of rows that span two planes.
* Guard regions around every buffer, on grids whose tiles are enough for these kernels (one per
  SM) with a partial last one on both axes.

Against the oracle; tolerances of the other parity tests (FP32 5e-5, refined 1e-9, rtol 1e-10).
"""

import ctypes

import numpy as np
import pytest

from oracle import adjoint as AD
from oracle import solve as S
from paper_1802_10323_gb300 import synth
from test_gpu_faults import Padded
from test_gpu_generic_lines import BCS, HALF, _solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mx,my", HALF + [(b, a) for a, b in HALF])
def test_all_pairs_match_oracle(lib, mx, my):
    nx, ny, nz = 2 * mx, 2 * my, 77
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 2.0 / nx, 1.0 / ny
    f = synth.uniform_noise((nz, ny, nx), seed=nx + ny, remove_mean=False)
    i = HALF.index((max(mx, my), min(mx, my)))
    for sx, sy in ((1, 0), (3, 2), (4, 3)):  # (0, 1) and (2, 4) there
        bcs = (BCS[(i + sx) % 5], BCS[(i + sy) % 5], "DD")
        q = S.solve(f, dx, dy, zf, *bcs)
        p = _solve(lib, f, dx, dy, zf, bcs, precision="fp32")
        assert np.abs(p - q).max() <= 5e-5 * np.abs(q).max(), (bcs, np.abs(p - q).max() / np.abs(q).max())


@pytest.mark.parametrize("nx,ny,nz,bcs", [(192, 18, 140, ("P", "NN", "NN")), (972, 18, 137, ("NN", "DD", "DN")),
                                          (36, 54, 141, ("DN", "P", "ND")), (486, 24, 103, ("DD", "ND", "DD"))])
def test_fp32_transpose_matches_oracle(lib, nx, ny, nz, bcs):
    import torch
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 2.0 / nx, 1.0 / ny
    g = synth.uniform_noise((nz, ny, nx), seed=nx, remove_mean=False)
    plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=bcs, precision="fp32")
    p = plan.solve_transpose(torch.as_tensor(g, dtype=torch.float32, device="cuda").contiguous()).double().cpu().numpy()
    plan.close()
    q = AD.solve_transpose(g, dx, dy, zf, *bcs)
    assert np.abs(p - q).max() <= 5e-5 * np.abs(q).max(), np.abs(p - q).max() / np.abs(q).max()


@pytest.mark.parametrize("shape,bcs", [((151, 36, 54), ("NN", "DD", "ND")), ((77, 72, 162), ("P", "DN", "NN")),
                                       ((139, 18, 972), ("DD", "P", "DN")), ((19, 864, 144), ("ND", "NN", "P"))])
@pytest.mark.parametrize("mode", ["fp32", "fp32_refine", "transpose"])
def test_guards_stay_intact(lib, shape, bcs, mode):
    import torch
    nz, ny, nx = shape
    zf = synth.uniform_faces(nz, 1.0) if bcs[2] == "P" else synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 1.0 / nx, 2.0 / ny
    f = np.random.default_rng(nx + nz).uniform(-1, 1, shape)
    plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=bcs, precision="fp32" if mode == "transpose" else mode, rtol=1e-10,
                    max_iter=8)
    dt, es = (torch.float64, 8) if mode == "fp32_refine" else (torch.float32, 4)
    pad = Padded([f.size * es, f.size * es, plan.workspace_bytes, 32])
    fd, pd = pad.view(0, dt, shape), pad.view(1, dt, shape)
    fd.copy_(torch.as_tensor(f, dtype=dt))
    fn = {"fp32": lib.ps_solve_f32, "fp32_refine": lib.ps_solve, "transpose": lib.ps_solve_transpose_f32}[mode]
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (fd, pd, pad.view(2, torch.uint8), pad.view(3, torch.float64))]
    lib._check(fn(plan.handle, *ptr[:3], ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), ptr[3]), plan.handle)
    torch.cuda.synchronize()
    assert pad.intact(), "a kernel wrote outside its buffers"
    q = AD.solve_transpose(f, dx, dy, zf, *bcs) if mode == "transpose" else S.solve(f, dx, dy, zf, *bcs)
    tol = 1e-9 if mode == "fp32_refine" else 5e-5
    assert np.abs(pd.double().cpu().numpy() - q).max() <= tol * np.abs(q).max()
    plan.close()
