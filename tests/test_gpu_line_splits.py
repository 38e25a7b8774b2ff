"""The line transforms on both sides of the rules that split a pass over the chip.

FP64 x passes of power-of-two lines change their stages at 1216 lines (the passes beyond leave
the last warp with two of its four lines); lines of other lengths run in tiles of 256 to one, by
their length and number and the width of a plane. Against the oracle, with the tolerances of the
solver's other parity tests: FP64 1e-12, the refined solve 1e-9 (rtol 1e-10), FP32 5e-5 of ‖p‖∞.
"""

import numpy as np
import pytest

from oracle import solve as S
from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu

ALL = ("fp64", "fp32", "fp32_refine")
CASES = [(n, 64, 19, b, "P", ("fp64",)) for n, b in ((128, "DD"), (256, "P"), (512, "ND"))] + \
        [(n, 6, 203, b, "P", ("fp64",)) for n, b in ((128, "DN"), (256, "NN"), (256, "DD"), (512, "P"))] + \
        [(1296, 54, 7, "NN", "DD", ALL),    # 378 rows of 648 points
         (1296, 54, 23, "DN", "P", ALL),    # 1242
         (12, 1944, 3, "P", "ND", ALL),     # columns of 972 points, one each
         (108, 2592, 6, "NN", "DD", ALL),   # 648 columns of 1296
         (2, 1024, 160, "NN", "P", ALL),    # the shortest lines: tiles of 256 rows,
         (1024, 6, 40, "P", "DD", ALL),     # of 64 columns,
         (162, 16, 97, "ND", "DN", ALL),    # and a last one of 34
         (2, 972, 160, "P", "NN", ALL), (6, 1024, 30, "DD", "P", ALL),  # planes narrower than a tile
         (18, 128, 30, "DN", "ND", ALL),
         (4374, 2, 3, "DD", "NN", ALL), (4608, 6, 60, "P", "NN", ALL), (6, 7776, 2, "DN", "NN", ALL)]


@pytest.mark.parametrize("nx,ny,nz,bx,by,precs", CASES)
def test_lines_match_oracle(lib, nx, ny, nz, bx, by, precs):
    import torch
    bcs = (bx, by, "ND")
    zf = synth.tanh_faces(nz, float(nz), 1.5)
    dx, dy = 2.0 / nx, 1.0 / ny
    f = synth.uniform_noise((nz, ny, nx), seed=nx + ny, remove_mean=False)
    q = S.solve(f, dx, dy, zf, *bcs)
    tol = dict(fp64=1e-12, fp32=5e-5, fp32_refine=1e-9)
    for prec in precs:
        kw = dict(rtol=1e-10, max_iter=6) if prec == "fp32_refine" else {}
        plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=bcs, precision=prec, **kw)
        dt = torch.float32 if prec == "fp32" else torch.float64
        p = plan.solve(torch.as_tensor(f, device="cuda").to(dt).contiguous()).double().cpu().numpy()
        plan.close()
        assert np.abs(p - q).max() <= tol[prec] * np.abs(q).max(), (prec, np.abs(p - q).max() / np.abs(q).max())
