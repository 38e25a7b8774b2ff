"""The first correction of a refined solve ends the loop at half of rtol, later ones at rtol.

The residual after one correction is measured (max_iter = 1), then rtol is put above and below
twice that value: in between a second correction runs if one is allowed, and the status is
that of rtol in every case.
"""

import pytest

from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,bcs", [(64, 48, 24, ("P", "NN", "DD")), (96, 32, 33, ("NN", "P", "NN"))])
def test_stop_margin(lib, nx, ny, nz, bcs):
    import torch
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    f = torch.as_tensor(synth.uniform_noise((nz, ny, nx), seed=9, remove_mean=False), device="cuda").contiguous()

    def solve(rtol, max_iter):
        plan = lib.Plan(nx, ny, nz, 2.0 / nx, 1.0 / ny, zf=zf, bcs=bcs, precision="fp32_refine", rtol=rtol,
                        max_iter=max_iter)
        info = lib.info_tensor()
        plan.solve(f, info=info)
        torch.cuda.synchronize()
        plan.close()
        return lib.read_info(info)

    r1 = solve(1e-15, 1).rel_residual
    above = solve(3.0 * r1, 4)
    assert (above.status, above.iterations) == (0, 1)
    between = solve(1.4 * r1, 4)
    assert (between.status, between.iterations) == (0, 2) and between.rel_residual <= 1.4 * r1
    last = solve(1.4 * r1, 1)
    assert (last.status, last.iterations) == (0, 1)
    below = solve(0.5 * r1, 1)
    assert below.status != 0
