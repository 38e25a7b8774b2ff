"""The line transforms of lengths that are no power of two, at the edges of their tiles.

Lines whose half length is not a power of two, or that sit in planes whose n_x is no multiple
of a tile of lines, run in one kernel with run-time radices (16, 9, 8, 6, 4, 3, 2). The cases
put every radix and every boundary pair on both axes, with tiles cut by the end of the rows
and of the plane, the shortest lines (n = 2, no FFT stage) and the longest of the FP32 radix
range, against the oracle. Tolerances are those of the solver's other parity tests: FP64
1e-12 and the refined solve 1e-9 of ‖p‖∞ (rtol 1e-10), FP32 5e-5.
"""

import numpy as np
import pytest

from oracle import solve as S
from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu

# (nx, ny, nz, bcx, bcy)
CASES = [
    (2, 486, 3, "NN", "DD"),      # no FFT stage on x; 243 = 9·9·3 on y, tiles of 2 columns
    (54, 2, 5, "DN", "ND"),       # 27 = 9·3; no stage on y (DCT-IV pre-factor alone)
    (18, 162, 4, "DD", "P"),      # 81 = 9·9; a last tile of 2 columns
    (36, 24, 7, "ND", "NN"),      # 18 = 9·2, 12 = 6·2
    (192, 96, 9, "NN", "DN"),     # 96 = 16·6, 48 = 8·6
    (108, 576, 2, "P", "ND"),     # 54 = 9·6, 288 three stages
    (972, 12, 2, "DD", "NN"),     # 486 = 9·9·6
    (64, 32, 3, "NN", "P"),       # 32 and 16 points
]


def _solve(lib, f, dx, dy, zf, bcs, **kw):
    import torch
    nz, ny, nx = f.shape
    plan = lib.Plan(nx, ny, nz, dx, dy, zf=zf, bcs=bcs, **kw)
    dt = torch.float32 if kw.get("precision") == "fp32" else torch.float64
    p = plan.solve(torch.as_tensor(f, device="cuda").to(dt).contiguous())
    torch.cuda.synchronize()
    plan.close()
    return p.double().cpu().numpy()


@pytest.mark.parametrize("nx,ny,nz,bx,by", CASES)
def test_generic_lines_match_oracle(lib, nx, ny, nz, bx, by):
    bcs = (bx, by, "ND")
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 2.0 / nx, 1.0 / ny
    f = synth.uniform_noise((nz, ny, nx), seed=nx + ny, remove_mean=False)
    q = S.solve(f, dx, dy, zf, *bcs)
    scale = np.abs(q).max()
    for prec, tol, kw in (("fp64", 1e-12, {}), ("fp32", 5e-5, {}),
                          ("fp32_refine", 1e-9, dict(rtol=1e-10, max_iter=6))):
        p = _solve(lib, f, dx, dy, zf, bcs, precision=prec, **kw)
        assert np.abs(p - q).max() <= tol * scale, (prec, np.abs(p - q).max() / scale)


# half lengths with a compile-time kernel, paired so that each runs on x and on y; n_z gives
# every SM a tile (the rule of the dispatch), the last tiles of a plane are partial
HALF = [(486, 16), (432, 18), (384, 24), (324, 27), (288, 32), (243, 36), (216, 48), (192, 54), (162, 72),
        (144, 81), (108, 96)]
BCS = ["P", "NN", "DD", "ND", "DN"]


@pytest.mark.parametrize("mx,my", HALF + [(b, a) for a, b in HALF])
def test_compile_time_lines_match_oracle(lib, mx, my):
    nx, ny, nz = 2 * mx, 2 * my, 77
    zf = synth.tanh_faces(nz, 1.0, 1.5)
    dx, dy = 2.0 / nx, 1.0 / ny
    f = synth.uniform_noise((nz, ny, nx), seed=nx + ny, remove_mean=False)
    i = HALF.index((max(mx, my), min(mx, my)))
    for bx, by, prec, tol, kw in ((BCS[i % 5], BCS[(i + 1) % 5], "fp32", 5e-5, {}),
                                  (BCS[(i + 2) % 5], BCS[(i + 4) % 5], "fp32_refine", 1e-9,
                                   dict(rtol=1e-10, max_iter=6))):
        bcs = (bx, by, "DD")
        q = S.solve(f, dx, dy, zf, *bcs)
        p = _solve(lib, f, dx, dy, zf, bcs, precision=prec, **kw)
        assert np.abs(p - q).max() <= tol * np.abs(q).max(), (prec, bcs, np.abs(p - q).max() / np.abs(q).max())
