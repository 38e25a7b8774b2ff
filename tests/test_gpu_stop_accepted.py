"""What the first correction of a refined solve has reached is not lost by a second one.

A first correction in (rtol/2, rtol] is followed by one more. On these grids (spacings along x
so fine beside the other axes that κ is beyond 10^14, right-hand sides alternating along x) the
second one raises the residual above rtol again. It is then taken back: the status is that of
the first, its residual is reported, and p is the first's up to the two roundings of p + e − e.
"""

import numpy as np
import pytest

from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu

GRIDS = [(512, 8, 8, 3e-6), (4096, 8, 8, 1e-5), (512, 128, 8, 3e-7)]  # nx, ny, nz, length along x


@pytest.mark.parametrize("nx,ny,nz,lx", GRIDS)
def test_accepted_first_correction_is_kept(lib, nx, ny, nz, lx):
    import torch
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    a = np.random.default_rng(3).uniform(1, 2, (nz, ny, 1))
    fh = torch.as_tensor(a * (2.0 * (np.arange(nx) % 2) - 1)).contiguous()
    f = fh.cuda()

    def solve(rtol, max_iter, host=False):
        plan = lib.Plan(nx, ny, nz, lx / nx, 1.0 / ny, zf=zf, bcs=("NN", "DN", "NN"), precision="fp32_refine",
                        rtol=rtol, max_iter=max_iter)
        if host:
            p = torch.full_like(fh, float("nan")).pin_memory()
            info = plan.solve_host(fh.pin_memory(), p, torch.empty_like(f), torch.empty_like(f))
        else:
            rec = lib.info_tensor()
            p = plan.solve(f, info=rec)
            torch.cuda.synchronize()
            info = lib.read_info(rec)
        plan.close()
        return p.cpu(), info

    p1, one = solve(1e-30, 1)
    p2, two = solve(1e-30, 2)
    assert two.rel_residual > 1.05 * one.rel_residual  # the grid does what the test is about
    rtol = 1.02 * one.rel_residual
    pf, first = solve(rtol, 1)  # (its pass 0 may have another form than at 1e-30)
    assert first.status == 0
    # roundings of p + e and − e: 2^-53 of the larger of |p| and |p + e| each
    tol = 2.0 ** -52 * (pf.abs().max() + (p2 - p1).abs().max()).item()
    for host in (False, True):
        p, info = solve(rtol, 4, host)
        assert (info.status, info.rel_residual) == (0, first.rel_residual)
        assert (p - pf).abs().max().item() <= tol


@pytest.mark.parametrize("nx,ny,nz,bcs", [(1024, 1024, 8, ("P", "P", "ND")), (2048, 512, 6, ("NN", "P", "DN")),
                                          (512, 512, 32, ("NN", "NN", "NN")), (64, 64, 64, ("NN", "NN", "NN")),
                                          (162, 64, 175, ("P", "NN", "NN")), (4096, 48, 12, ("DN", "DD", "NN"))])
def test_solution_error_at_the_stop(lib, nx, ny, nz, bcs):
    """The relative error of the solution (against the FP64 plan's) stays within ten times rtol
    wherever the loop ends: the amplification measured on grids of noise is 0.1 to 8."""
    import torch
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    f = torch.rand((nz, ny, nx), generator=torch.Generator("cuda").manual_seed(nx), device="cuda",
                   dtype=torch.float64).mul_(2.0).sub_(1.0)
    singular = all(b in ("P", "NN") for b in bcs)
    if singular:
        f -= f.mean()
    plan = lib.Plan(nx, ny, nz, 6.0 / nx, 3.0 / ny, zf=zf, bcs=bcs, precision="fp64")
    q = plan.solve(f)
    plan.close()
    for rtol in (1e-8, 1e-9, 3e-10, 1e-10, 3e-11, 1e-11):
        plan = lib.Plan(nx, ny, nz, 6.0 / nx, 3.0 / ny, zf=zf, bcs=bcs, precision="fp32_refine", rtol=rtol, max_iter=4)
        info = lib.info_tensor()
        d = plan.solve(f, info=info) - q
        rec = lib.read_info(info)
        plan.close()
        if singular:  # (the constant of p is free)
            d -= d.mean()
        assert rec.status == 0 and rec.rel_residual <= rtol
        assert d.abs().max() <= 10 * rtol * q.abs().max(), (rtol, rec.iterations, (d.abs().max() / q.abs().max()).item())
