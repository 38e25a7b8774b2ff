"""The batched solve at the edges of its residual tiles (256 columns by 16 planes).

Column counts below, at and above a multiple of 256 and plane counts around a multiple of 16,
with every kind of end on each axis: the residual of each grid, measured again by the oracle's
stencil in FP64, is within the tolerance that the solve reports plus the double-float
residual's own rounding, 2^-46 of the sum of its terms' magnitudes.
"""

import numpy as np
import pytest

from oracle import operator as O
from paper_1802_10323_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 15), (16, 16, 16), (18, 16, 17), (12, 24, 33), (32, 16, 8), (54, 6, 48)]
BCS = [("P", "ND", "DD"), ("DD", "P", "P"), ("DN", "NN", "ND"), ("NN", "DD", "DN"), ("P", "P", "P"), ("NN", "NN", "NN")]


@pytest.mark.parametrize("shift", [0.0, 30.0])
@pytest.mark.parametrize("turn", range(len(BCS)))
def test_batch_residual_tiles(lib, turn, shift):
    import torch
    grids, fs = [], []
    for g, (nx, ny, nz) in enumerate(SHAPES):
        bcs = BCS[(g + turn) % len(BCS)]
        zf = synth.uniform_faces(nz, 1.0) if bcs[2] == "P" else synth.tanh_faces(nz, 1.0, 1.2)
        grids.append(dict(nx=nx, ny=ny, nz=nz, dx=1.0 / nx, dy=2.0 / ny, zf=zf, bcs=bcs, alpha=shift))
        f = np.random.default_rng(100 * turn + g).uniform(-1, 1, (nz, ny, nx))
        fs.append(torch.as_tensor(f, device="cuda").contiguous())
    ps = [torch.zeros_like(f) for f in fs]
    b = lib.Batch(grids, rtol=1e-10, max_iter=6)
    fptr, pptr = b.pointers(fs, ps)
    infos = lib.infos_tensor(len(grids))
    b.solve(fptr, pptr, infos)
    torch.cuda.synchronize()
    for g, (d, inf) in enumerate(zip(grids, lib.read_infos(infos, len(grids)))):
        f, p = fs[g].cpu().numpy(), ps[g].cpu().numpy()
        terms = 4 * (d["dx"] ** -2 + d["dy"] ** -2 + np.diff(d["zf"]).min() ** -2) + shift
        rounding = 2.0 ** -46 * terms * np.abs(p).max() / np.abs(f).max()
        assert inf.status == 0, (g, inf.status, inf.rel_residual)
        assert O.relative_residual(p, f, d["dx"], d["dy"], d["zf"], *d["bcs"], alpha=shift) <= 1e-10 + rounding, g
    b.close()
