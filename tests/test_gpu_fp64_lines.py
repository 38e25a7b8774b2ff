"""FP64 lines of 128, 256, 512 and 1024 values, whose stages take radices 16 and 8.

Every boundary pair on both axes; the numbers of lines leave the last warp of the x kernel with
one to three lines of its four, and the y kernel with tiles of one plane only. Against the
oracle, within 1e-12 of the largest value as the other FP64 parity tests.
"""

import numpy as np
import pytest

from oracle import solve as S
from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["P", "NN", "DD", "ND", "DN"])
@pytest.mark.parametrize("nx,ny,nz", [(128, 2, 3), (256, 18, 3), (512, 6, 3), (1024, 2, 3),
                                      (16, 128, 3), (48, 256, 2), (16, 512, 2), (16, 1024, 2), (128, 256, 2)])
def test_fp64_lines(lib, nx, ny, nz, bc):
    import torch
    bcs = (bc, "DD" if nx > ny and bc != "DD" else bc, "ND")
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 2.0 / nx, 1.0 / ny
    f = synth.uniform_noise((nz, ny, nx), seed=nx + ny, remove_mean=False)
    q = S.solve(f, dx, dy, zf, *bcs)
    plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=bcs, precision="fp64")
    p = plan.solve(torch.as_tensor(f, device="cuda").contiguous())
    torch.cuda.synchronize()
    plan.close()
    assert np.abs(p.cpu().numpy() - q).max() <= 1e-12 * np.abs(q).max()
